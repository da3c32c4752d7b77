// Batched finalize: many partitioned counting jobs in one set of launches.
//
// Consume: one persistent launch over a device work queue of (job, partition)
// items from every job of the batch.  Each CTA takes the next item, counts the
// partition's keys in a shared-memory table, writes the survivors and the
// partition's filter words and moves on, so uneven jobs share the GPU without a
// launch each.
// Sort: every job's survivors are bucketed by key (key_bucket) into one flat
// bucket array covering all jobs, scanned once, scattered as pairs, and each
// bucket sorted by one warp into its job's result arrays.  These launches
// read every size and pointer from a device-side batch descriptor, so the
// sequence is captured once in a CUDA graph and replayed for every batch.
// A single kc_finalize is a batch of one.

#include <algorithm>
#include <cstring>
#include <vector>

#include "kc_ctx.h"

namespace kc {

struct JobDesc {
    // consumer
    int part_bits, slice_log2, table_log2, bloom_shift;
    int n_hashes, n_samples, all_candidates, key_bits;
    uint32_t min_count;
    int n_batches;
    uint32_t item_base;  // first queue item of this job
    uint32_t part_base;  // partition of the job's first item
    const uint64_t* const* data;
    const uint64_t* const* starts;
    const int* samples;
    unsigned long long* bloom;
    uint64_t* sv_keys;
    uint64_t* sv_vals;
    uint64_t sv_cap;
    uint64_t* failed;  // per overflowing partition: its first hash not yet counted
    DevCounters* ctr;
    // sort
    int sort_bits;
    int even;  // buckets of equal shares of the canonical keys' distribution (key_bucket)
    int split_max;  // consumer: finest split level 2^split_max before the fallback
    int split_min;  // level at which a sub-range's filter words fit the consumer's shared memory
    uint64_t bucket_base;  // first bucket of this job in the flat arrays
    uint64_t n_buckets;
    uint64_t* res_keys;
    uint64_t* res_vals;
    uint64_t res_cap;
    uint64_t flat_base;  // this job's first survivor in the batch's survivors, in job order (set by the plan)
    // survivors histogrammed by the consumer itself (the sort's bucket bits
    // fixed before it runs): fixed_bits >= 0, hist_job = the job's first
    // bucket counter; else fixed_bits = -1
    int fixed_bits;
    uint32_t* hist_job;
};

struct BatchDesc {
    const JobDesc* jobs;
    const uint32_t* item_job;
    unsigned long long* counters;  // per job: [2j] survivors, [2j+1] failed partitions
    unsigned int* head;            // work-queue head
    unsigned int* err;             // DERR_* bits of the sort
    uint32_t n_jobs;
    uint32_t n_items;
    uint64_t n_buckets;  // total over jobs
    uint32_t* hist;
    uint64_t* starts;
    uint64_t* cursor;
    unsigned long long* tiles;  // the scan's state: a word per tile, then the ticket
    uint64_t n_tiles;
    uint64_t buckets_cap;  // room of hist / starts / cursor
    uint64_t n_flat;       // set by the plan: survivors of all jobs
    // the survivors scattered into their buckets, (key, value) side by side in
    // the flat bucket order of all jobs; the bucket sorts write the results
    ulonglong2* pairs;
    uint64_t pairs_cap;
};

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kConsumeThreads = 512;      // consumer CTAs, two an SM
constexpr int kConsumeThreadsWide = 1024;  // when the shared memory has room for one alone
constexpr int kAhead = 3;                  // hashes a consumer thread has in flight
constexpr unsigned long long kTopBit = 1ull << 63;
constexpr uint32_t kChunk = 1u << 31;  // hashes a consumer loop indexes with 32 bits

// One partition at a time per CTA: every distinct key of the partition is
// counted in a shared-memory table, and the filter words are built from the
// table afterwards.  A key's filter bits do not depend on how often it was
// seen, so the filter is updated once per distinct key instead of once per
// window, no window waits for the filter's answer, and the hashes are read
// once, without a recount.  (Updating the filter with every window and counting
// the candidates took 0.975 ms for 1.18e8 windows of 4096 partitions, this
// 0.660 ms.  It is bound by instruction issue, at two thirds of the issue
// slots: reading the hashes alone takes 0.17 ms, with one probe each 0.21, with
// the queue's probes 0.36, the writing 0.08 and the filter 0.1 more.)
//
//   count    each window's first probe; a window that finds its key adds one
//            to its count.  The others (new keys and displaced ones, about one
//            in four at 30x coverage) go to a queue of the warp; 32 of them at a
//            time take two probes (and a claim) each and go back to the queue if
//            both failed, so every probe step has all its lanes.  (One probe a
//            step and four hashes in flight instead of three: 0.680 ms.)  With
//            one sample a new key whose first slot is free claims it at once:
//            2.9e7 windows of which 64 % are new keys 0.435 -> 0.412 ms, 1.2e8
//            of which 18 % are as before; with two samples, where fewer warps
//            run, 4.7e8 windows took 2.95 ms without and 2.99 with it.
//   emit     keys of at least min_count, one position claim per warp
//   filter   the counts are no longer needed: their memory takes the filter
//            words, every key sets its bits, the words are written out
//
// The table holds the keys that occur once too, so it is twice as large as the
// candidates alone would need (8192 slots, 96 KiB with the counts: two
// 512-thread CTAs an SM; when only one fits, 1024 threads).  Triangular probing
// keeps a table two thirds full (30x coverage) to about two probes a new key:
// linear probing took 0.09 ms more, the probe loop of a whole warp at once 0.15.
//
// A partition whose keys overflow the table is counted again in 2, 4, ...
// 2^split_max sub-ranges of its filter slice: the top bits of a window's
// in-slice word index pick its sub-range, so two sub-ranges never share a
// filter word and each one's table and filter are exactly those of the whole
// partition restricted to its keys.  Sub-ranges already finished stay finished
// when a later one has to split further.  Only a partition that overflows at
// the finest level is left to the global fallback.  The finest level a job has
// needed is kept in its counters, and its later partitions start there instead
// of overflowing again.
//
// ONE: every job of the batch has one sample (a slot's counts at a constant
// place).
template <int THREADS, bool ONE>
__global__ void __launch_bounds__(THREADS, THREADS == kConsumeThreads ? 2 : 1)
    k_consume_q(const BatchDesc* __restrict__ D) {
    extern __shared__ unsigned long long s_mem[];
    __shared__ int s_fail, s_hint;
    __shared__ unsigned s_item;
    constexpr int kWarps = THREADS / 32;
    constexpr bool kClaimAtOnce = ONE;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const uint32_t n_items = D->n_items;
    // the warp's queue: hashes, and for each the slot to probe next (low 16
    // bits) and the number of probes that failed (above)
    unsigned long long* const wq = s_mem + wid * kWarpQueue;
    uint32_t* const ws = reinterpret_cast<uint32_t*>(s_mem + kWarps * kWarpQueue) + wid * kWarpQueue;
    unsigned long long* const sk = s_mem + kWarps * kWarpQueue * 3 / 2;
    uint64_t cand = 0, claimed = 0;
    DevCounters* last_ctr = nullptr;
    for (;;) {
        if (threadIdx.x == 0) {
            const unsigned it = atomicAdd(D->head, 1u);
            s_item = it;
            // the finest level this job's partitions have needed so far
            s_hint = it < n_items ? (int)*(volatile unsigned*)&D->jobs[D->item_job[it]].ctr->split_hint : 0;
        }
        __syncthreads();
        const unsigned item = s_item;
        const int hint = s_hint;
        if (item >= n_items) break;
        const uint32_t j = D->item_job[item];
        const JobDesc& J = D->jobs[j];
        const uint32_t part = J.part_base + (item - J.item_base);
        const uint32_t n_sw = 1u << J.slice_log2;
        const uint32_t T = 1u << J.table_log2;
        const uint32_t tmask = T - 1;
        const int s2 = ONE ? 0 : J.n_samples - 1;  // a slot's counts: 1 << s2 of them
        const int a = J.part_bits;
        uint32_t* const sc = reinterpret_cast<uint32_t*>(sk + T);  // counts, then
        unsigned long long* const sb = sk + T;                     // the filter words
        if (J.ctr != last_ctr) {  // per-job candidate counters
            cand = warp_sum(cand);
            claimed = warp_sum(claimed);
            if (lane == 0 && last_ctr) {
                if (cand) atomicAdd(&last_ctr->candidates, (unsigned long long)cand);
                if (claimed) atomicAdd(&last_ctr->claimed, (unsigned long long)claimed);
            }
            cand = claimed = 0;
            last_ctr = J.ctr;
        }
        const uint64_t hpre = (uint64_t)part << (64 - a);
        const unsigned long long empty = hpre ^ (1ull << (64 - a));  // a hash of another partition
        int sl = max(min(hint, J.split_max), J.split_min);  // split level: the partition is taken as 2^sl sub-ranges
        uint32_t sub = 0;  // the sub-range being counted
        bool overflow = false;
        uint64_t h_left = 0;  // first hash left to the fallback
        for (;;) {
            const uint32_t w_n = n_sw >> sl;
            const uint32_t smask = (1u << sl) - 1u;
            const int sub_shift = 64 - a - sl;  // sub-range = h bits [sub_shift, 64 - a)
            // a window belongs to the (sub-range of the) partition iff the top
            // a + sl <= 32 bits of its hash equal those of `range`
            const uint64_t range = hpre | ((uint64_t)sub << sub_shift);
            const uint32_t rhi = (uint32_t)(range >> 32), rmask = ~0u << (32 - a - sl);
            for (uint32_t i = threadIdx.x; i < T / 2; i += THREADS)
                reinterpret_cast<ulonglong2*>(sk)[i] = make_ulonglong2(empty, empty);
            for (uint32_t i = threadIdx.x; i < (T << s2) / 4; i += THREADS)
                reinterpret_cast<uint4*>(sc)[i] = make_uint4(0u, 0u, 0u, 0u);
            if (threadIdx.x == 0) s_fail = 0;
            __syncthreads();
            bool stop = false;  // the same in all lanes of a warp
            for (int bt = 0; bt < J.n_batches && !stop; ++bt) {
                const uint64_t lo = J.starts[bt][part];
                const uint64_t n_all = J.starts[bt][part + 1] - lo;
                uint32_t* const scol = ONE ? sc : sc + J.samples[bt];  // this batch's count column
                unsigned q = 0;                             // entries in the warp's queue
                // The queue's last n (at most 32) windows, one per lane, take their
                // next two probes: slots home, home + 1, home + 3, home + 6, ... (every
                // slot of a power-of-two table in turn).
                const auto step = [&](unsigned n) {
                    __syncwarp();
                    q -= n;
                    bool again = false;
                    unsigned long long h = 0;
                    uint32_t next = 0;
                    if ((unsigned)lane < n) {
                        h = wq[q + lane];
                        next = ws[q + lane];
                        const auto probe = [&](uint32_t slot) {
                            unsigned long long cur = sk[slot];
                            if (cur == empty) {
                                cur = atomicCAS(sk + slot, empty, h);
                                if (cur == empty) cur = h;
                            }
                            return cur == h;
                        };
                        uint32_t slot = next & tmask;
                        bool found = probe(slot);
                        if (!found) {
                            next += 0x10000u;
                            slot = (slot + (next >> 16)) & tmask;
                            found = probe(slot);
                        }
                        if (found) {
                            atomicAdd(scol + (slot << s2), 1u);
                        } else {
                            next = ((next & 0xffff0000u) + 0x10000u) | ((slot + (next >> 16) + 1) & tmask);
                            again = next < (unsigned)kProbeLimit << 16;
                            if (!again) s_fail = 1;
                        }
                    }
                    const unsigned back = __ballot_sync(kFull, again);
                    if (again) {
                        const unsigned pos = q + __popc(back & lt);
                        wq[pos] = h;
                        ws[pos] = next;
                    }
                    q += __popc(back);
                };
                // 32-bit indices within chunks of 2^31 hashes (one chunk, in practice)
                for (uint64_t c0 = 0; c0 < n_all && !stop; c0 += kChunk) {
                    const uint64_t* __restrict__ d = J.data[bt] + lo + c0;
                    const uint32_t n = (uint32_t)min(n_all - c0, (uint64_t)kChunk);
                    // each thread's next hashes are in flight while it handles the current ones
                    uint64_t hn[kAhead];
#pragma unroll
                    for (int e = 0; e < kAhead; ++e) {
                        const uint32_t i = e * THREADS + threadIdx.x;
                        hn[e] = i < n ? __ldcg(d + i) : empty;
                    }
                    for (uint32_t b = 0; b < n && !stop; b += kAhead * THREADS) {
                        uint64_t hc[kAhead];
#pragma unroll
                        for (int e = 0; e < kAhead; ++e) {
                            hc[e] = hn[e];
                            const uint32_t i = b + (kAhead + e) * THREADS + threadIdx.x;
                            hn[e] = i < n ? __ldcg(d + i) : empty;
                        }
#pragma unroll
                        for (int e = 0; e < kAhead; ++e) {
                            const uint64_t h = hc[e];
                            const bool in = ((((uint32_t)(h >> 32)) ^ rhi) & rmask) == 0u;  // else run padding, or another sub-range
                            const uint32_t s = (uint32_t)h & tmask;
                            unsigned long long cur = sk[s];
                            if (kClaimAtOnce && in && cur == empty) {
                                cur = atomicCAS(sk + s, empty, h);
                                if (cur == empty) cur = h;
                            }
                            const bool hit = in && cur == h;  // (padding may hold the empty mark)
                            if (hit) atomicAdd(scol + (s << s2), 1u);
                            const unsigned miss = __ballot_sync(kFull, in && !hit);
                            if (miss) {
                                if (in && !hit) {
                                    const unsigned pos = q + __popc(miss & lt);
                                    wq[pos] = h;
                                    ws[pos] = !kClaimAtOnce && cur == empty ? s : 0x10000u | ((s + 1) & tmask);
                                }
                                q += __popc(miss);
                                while (q >= 32) step(32);
                            }
                        }
                        stop = __any_sync(kFull, *(volatile int*)&s_fail);  // a warp overflowed: give up early
                    }
                }
                while (q) step(min(q, 32u));
                stop = __any_sync(kFull, *(volatile int*)&s_fail);
            }
            __syncthreads();
            if (s_fail) {
                __syncthreads();  // s_fail is cleared for the next attempt
                if (sl < J.split_max) {
                    ++sl;
                    sub <<= 1;
                    continue;
                }
                overflow = true;
                h_left = range;
                break;
            }
            // emit: each warp its slots [wid * T / kWarps, ...), at most 32 rows of 32
            const uint32_t rows = T / THREADS;  // T >= 1024
            const uint32_t slot0 = wid * rows * 32 + lane;
            unsigned kept = 0, n_kept = 0, once = 0;  // kept, once: lane r has the ballot of row r
            uint64_t n_win = 0;
            const uint32_t min_count = J.min_count;
            for (uint32_t r = 0; r < rows; ++r) {
                const uint32_t i = slot0 + r * 32;
                const uint64_t sum = s2 ? (uint64_t)sc[2 * i] + sc[2 * i + 1] : (uint64_t)sc[i];
                n_win += sum;
                const unsigned ballot = __ballot_sync(kFull, sum != 0 && sum >= min_count);
                const unsigned ones = __ballot_sync(kFull, sum == 1);
                if (lane == (int)r) {
                    kept = ballot;
                    once = ones;
                }
                n_kept += __popc(ballot);
            }
            unsigned long long pos0 = 0;
            if (n_kept) {
                if (lane == 0) pos0 = atomicAdd(&D->counters[2 * j], (unsigned long long)n_kept);
                pos0 = __shfl_sync(kFull, pos0, 0);
                uint64_t* const sv_keys = J.sv_keys;
                uint64_t* const sv_vals = J.sv_vals;
                uint32_t* const hist = J.hist_job;
                const uint64_t sv_cap = J.sv_cap;
                const int key_bits = J.key_bits, hist_bits = J.fixed_bits;
                const bool even = even_buckets(key_bits, hist_bits);
                unsigned qn = 0;  // the slots of kept keys, taken 32 at a time
                const auto write = [&](unsigned n) {
                    __syncwarp();
                    qn -= n;
                    const uint64_t pos = pos0 + lane;
                    if ((unsigned)lane < n && pos < sv_cap) {
                        const uint32_t i = ws[qn + lane];
                        const uint64_t key = unmixer64(sk[i]);
                        sv_keys[pos] = key;
                        sv_vals[pos] = s2 ? (uint64_t)sc[2 * i] | ((uint64_t)sc[2 * i + 1] << 32) : (uint64_t)sc[i];
                        if (hist) atomicAdd(hist + key_bucket(key, key_bits, hist_bits, even), 1u);
                    }
                    pos0 += n;
                    __syncwarp();
                };
                for (uint32_t r = 0; r < rows; ++r) {
                    const unsigned ballot = __shfl_sync(kFull, kept, r);
                    if ((ballot >> lane) & 1u) ws[qn + __popc(ballot & lt)] = slot0 + r * 32;
                    qn += __popc(ballot);
                    if (qn >= 32) write(32);
                }
                if (qn) write(qn);
            }
            // filter: the words of the (sub-)range in the place of the counts
            __syncthreads();
            for (uint32_t i = threadIdx.x; i < w_n; i += THREADS) sb[i] = 0ull;
            __syncthreads();
            const int bloom_shift = J.bloom_shift, n_hashes = J.n_hashes;
            const bool all_cand = J.all_candidates != 0;
            uint64_t n_new = 0, n_seen = 0;  // keys that set a bit first, keys that were candidates
            unsigned qn = 0;  // the warp's keys, taken 32 at a time (the table's rows are up to three quarters empty)
            const auto set_bits = [&](unsigned n) {
                __syncwarp();
                qn -= n;
                if ((unsigned)lane < n) {
                    uint64_t h = wq[qn + lane];
                    const bool once = (h ^ hpre) & kTopBit;
                    if (once) h ^= kTopBit;
                    const uint64_t g = mixer64(h);
                    const uint64_t pat = n_hashes == 4 ? bloom_pattern_n<4>(g) : bloom_pattern_rt(g, n_hashes);  // (4: every configuration's)
                    // one 64-bit update, so that of the keys with equal bits one alone finds them new (an
                    // update a half, where two keys can each be first in one, saves 0.5 to 1 % of a job)
                    const unsigned long long old =
                        atomicOr(sb + ((uint32_t)(h >> bloom_shift) & (w_n - 1)), (unsigned long long)pat);
                    const bool fresh = (pat & ~old) != 0ull;
                    n_new += fresh;
                    n_seen += all_cand || !(fresh && once);
                }
                __syncwarp();
            };
            for (uint32_t r = 0; r < rows; ++r) {
                const uint64_t h = sk[slot0 + r * 32];
                const unsigned used = __ballot_sync(kFull, h != empty);
                // a key seen once is queued with its top bit flipped: the filter's
                // candidates do not count it if its bits are new
                const unsigned ones = __shfl_sync(kFull, once, r);
                if (h != empty) wq[qn + __popc(used & lt)] = (ones >> lane) & 1u ? h ^ kTopBit : h;
                qn += __popc(used);
                if (qn >= 32) set_bits(32);
            }
            if (qn) set_bits(qn);
            // windows reported as seen before: all but each key's first, if its bits were new
            cand += n_win - (all_cand ? 0 : n_new);
            claimed += n_seen;
            __syncthreads();
            unsigned long long* gb = J.bloom + (uint64_t)part * n_sw + sub * w_n;
            for (uint32_t i = threadIdx.x; i < w_n; i += THREADS) gb[i] = sb[i];
            __syncthreads();
            if (++sub > smask) break;
        }
        if (threadIdx.x == 0) {
            if (overflow) J.failed[atomicAdd(&D->counters[2 * j + 1], 1ull)] = h_left;
            else if (sl > J.split_min) atomicAdd(&J.ctr->split_parts, 1u);
            if (sl > hint) atomicMax(&J.ctr->split_hint, (unsigned)sl);
        }
    }
    cand = warp_sum(cand);
    claimed = warp_sum(claimed);
    if (lane == 0 && last_ctr) {
        if (cand) atomicAdd(&last_ctr->candidates, (unsigned long long)cand);
        if (claimed) atomicAdd(&last_ctr->claimed, (unsigned long long)claimed);
    }
}

// Start of a batch: the queue head, the sort error bits and every job's
// survivor and failed-partition counters at zero.
__global__ void k_reset_q(const BatchDesc* __restrict__ D) {
    for (uint32_t i = threadIdx.x; i < 2 * D->n_jobs; i += blockDim.x) D->counters[i] = 0ull;
    if (threadIdx.x == 0) {
        *D->head = 0u;
        *D->err = 0u;
    }
}

// Sort plan, on the device once the survivors are counted: per job, bucket
// bits for at most about 32 survivors a bucket and the job's first bucket in
// the flat arrays; the total into D->n_buckets.  More buckets than the arrays
// hold (never, when the host sized them from the survivor capacities) is an
// internal error and sorts nothing.
__device__ void plan_sort(BatchDesc* __restrict__ D) {
    JobDesc* jobs = const_cast<JobDesc*>(D->jobs);
    uint64_t total = 0, flat = 0;
    bool short_arrays = false;
    for (uint32_t j = 0; j < D->n_jobs; ++j) {
        JobDesc& J = jobs[j];
        uint64_t nsv = D->counters[2 * j];
        if (nsv > J.sv_cap) nsv = J.sv_cap;
        if (nsv > J.res_cap) {  // result arrays too short (a sort run ahead of the count): sort nothing
            short_arrays = true;
            nsv = 0;
        }
        J.flat_base = flat;
        flat += nsv;
        if (nsv < 1) nsv = 1;
        int bits = 0;
        if (J.fixed_bits >= 0) bits = J.fixed_bits;  // the consumer's histogram has these buckets
        else
            while (bits < 24 && bits < J.key_bits && (nsv >> bits) > 32) ++bits;
        J.sort_bits = bits;
        J.bucket_base = total;
        J.n_buckets = 1ull << bits;
        total += J.n_buckets;
        J.even = even_buckets(J.key_bits, bits) ? 1 : 0;
    }
    // short result arrays: no bucket and no survivor is sorted at all (a
    // histogram the consumer took may count that job's survivors), and the
    // host sorts again into larger arrays
    D->n_flat = short_arrays ? 0 : flat;
    *D->err = short_arrays ? DERR_INTERNAL : 0u;
    if (total > D->buckets_cap) {
        atomicOr(D->err, DERR_INTERNAL);
        total = 0;
    }
    D->n_buckets = short_arrays ? 0 : total;
}
__global__ void k_plan_q(BatchDesc* __restrict__ D) {
    if (threadIdx.x == 0) plan_sort(D);
    if (threadIdx.x >= 32)  // meanwhile the other warps clear the scan's state (all of it: the plan is not known yet)
        for (uint64_t i = threadIdx.x - 32; i <= D->n_tiles; i += blockDim.x - 32) D->tiles[i] = 0ull;
}

__global__ void k_zero_hist_q(const BatchDesc* __restrict__ D) {
    const uint64_t n = D->n_buckets;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) D->hist[i] = 0u;
}

// Job owning the batch's survivor number i (jobs are in survivor order).
__device__ __forceinline__ uint32_t job_of_survivor(const BatchDesc* D, uint64_t i) {
    uint32_t lo = 0, hi = D->n_jobs;  // invariant: jobs[lo].flat_base <= i
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (D->jobs[mid].flat_base <= i) lo = mid;
        else hi = mid;
    }
    return lo;
}

// A thread's view of the job that owns its current survivor: the fields the
// histogram and scatter use, reloaded only when the survivor index passes
// into a later job (a thread's indices only grow).
struct SurvivorJob {
    uint32_t j;
    uint64_t lo, hi;  // flat survivor range of job j
    const uint64_t* keys;
    const uint64_t* vals;
    int key_bits, bits;
    bool even;
    uint64_t n_buckets, bucket_base;
    uint64_t res_cap;
    __device__ void load(const BatchDesc* D, uint32_t jj) {
        j = jj;
        const JobDesc& J = D->jobs[jj];
        lo = J.flat_base;
        hi = jj + 1 < D->n_jobs ? D->jobs[jj + 1].flat_base : D->n_flat;
        keys = J.sv_keys;
        vals = J.sv_vals;
        key_bits = J.key_bits;
        bits = J.sort_bits;
        even = J.even != 0;
        n_buckets = J.n_buckets;
        bucket_base = J.bucket_base;
        res_cap = J.res_cap;
    }
    __device__ uint64_t bucket(uint64_t key) const { return key_bucket(key, key_bits, bits, even); }
    __device__ void seek(const BatchDesc* D, uint64_t i) {
        while (i >= hi && j + 1 < D->n_jobs) load(D, j + 1);
    }
};

// The survivors of all jobs as one flat range: every thread takes survivors
// across job boundaries, so one job or many keep the whole grid busy.
__global__ void k_prefix_hist_q(const BatchDesc* __restrict__ D) {
    const uint64_t n = D->n_flat;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    SurvivorJob S;
    S.load(D, job_of_survivor(D, i));
    for (; i < n; i += stride) {
        S.seek(D, i);
        const uint64_t b = S.bucket(S.keys[i - S.lo]);
        if (b < S.n_buckets) atomicAdd(D->hist + S.bucket_base + b, 1u);
        else atomicOr(D->err, DERR_INTERNAL);
    }
}

// Flat exclusive scan of D->hist over D->n_buckets counters (fixed grid of D's
// tile capacity; CTAs past the end exit).  One launch in place of a sum per
// tile, a scan of the sums and a second pass: 65,536 counters
// 5 us, 15 in three.
__global__ void __launch_bounds__(kScanThreads) k_scan_q(const BatchDesc* __restrict__ D) {
    if (blockIdx.x * kScanTile >= D->n_buckets) return;
    scan_lookback(D->hist, D->n_buckets, D->starts, D->cursor, D->tiles, D->tiles + D->n_tiles);
}

__global__ void __launch_bounds__(256) k_scatter_q(const BatchDesc* __restrict__ D) {
    const uint64_t n = D->n_flat;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    SurvivorJob S;
    S.load(D, job_of_survivor(D, i));
    uint64_t job0 = D->starts[S.bucket_base];
    for (; i < n; i += stride) {
        if (i >= S.hi) {
            S.seek(D, i);
            job0 = D->starts[S.bucket_base];
        }
        const uint64_t k = i - S.lo;
        const uint64_t key = S.keys[k];
        const uint64_t val = S.vals[k];
        const uint64_t b = S.bucket(key);
        if (b >= S.n_buckets) {
            atomicOr(D->err, DERR_INTERNAL);
            continue;
        }
        const uint64_t gpos = atomicAdd(reinterpret_cast<unsigned long long*>(D->cursor) + S.bucket_base + b, 1ull);
        if (gpos - job0 >= S.res_cap || gpos >= D->pairs_cap) {
            atomicOr(D->err, DERR_INTERNAL);
            continue;
        }
        D->pairs[gpos] = make_ulonglong2(key, val);  // one 16-byte store
    }
}

// Job owning flat bucket fb (jobs are in bucket order).
__device__ __forceinline__ uint32_t job_of_bucket(const BatchDesc* D, uint64_t fb) {
    uint32_t lo = 0, hi = D->n_jobs;  // invariant: jobs[lo].bucket_base <= fb
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (D->jobs[mid].bucket_base <= fb) lo = mid;
        else hi = mid;
    }
    return lo;
}

// Buckets of up to 64 keys (nearly all of them: the bits are chosen for 16 to
// 32 keys a bucket, and key_bucket's even shares keep them there): one warp
// each ranks the keys (warp_rank64) and stores every pair at its place.
// Bound by instruction issue (73 %) and shared-memory wavefronts (72 %) about
// equally; six 256-thread CTAs an SM in one wave, the next bucket's bounds
// loaded ahead.  6.8 M keys: 76 us (bitonic networks 129), a batch of 12 jobs
// 347 us (665).
__global__ void __launch_bounds__(256, 6) k_warp_sort_q(const BatchDesc* __restrict__ D) {
    __shared__ __align__(16) WarpRankTile tiles[256 / 32];
    const int lane = threadIdx.x & 31;
    WarpRankTile& tile = tiles[threadIdx.x >> 5];
    *reinterpret_cast<uint2*>(&tile.count[2 * lane]) = make_uint2(0u, 0u);
    __syncwarp();
    const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    const uint64_t nb = D->n_buckets;
    if (warp >= nb) return;
    uint64_t g0 = D->starts[warp], g1 = D->starts[warp + 1];
    uint64_t job_end = 0, job0 = 0;  // the job's last bucket + 1 and its first pair
    uint64_t *rk = nullptr, *rv = nullptr;
    int key_bits = 0;
    for (uint64_t fb = warp; fb < nb; fb += n_warps) {
        const uint64_t next = fb + n_warps;
        const uint64_t f0 = next < nb ? D->starts[next] : 0ull, f1 = next < nb ? D->starts[next + 1] : 0ull;
        const uint64_t n64 = g1 - g0;
        const ulonglong2* __restrict__ src = D->pairs + g0;
        const bool in0 = lane < (int)min((unsigned long long)n64, 32ull);
        const bool two = n64 > 32;
        const bool in1 = n64 > 32 + (uint64_t)lane;
        const ulonglong2 q0 = in0 ? src[lane] : make_ulonglong2(0ull, 0ull);
        const ulonglong2 q1 = in1 ? src[32 + lane] : make_ulonglong2(0ull, 0ull);
        if (fb >= job_end) {
            const JobDesc& J = D->jobs[job_of_bucket(D, fb)];
            job_end = J.bucket_base + J.n_buckets;
            job0 = D->starts[J.bucket_base];
            rk = J.res_keys;
            rv = J.res_vals;
            key_bits = J.key_bits;
        }
        const uint64_t lo = g0 - job0;
        if (n64 > 64) {
            // sorted later in place (k_warp_sort_big_q): the pairs as they are
            if (lane == 0 && !(*(volatile unsigned*)D->err & DERR_SORT_BIG)) atomicOr(D->err, DERR_SORT_BIG);
            for (uint64_t i = lane; i < n64; i += 32) {
                const ulonglong2 q = src[i];
                rk[lo + i] = q.x;
                rv[lo + i] = q.y;
            }
        } else if (n64) {
            uint32_t r0 = lane, r1 = 0;
            if (n64 > 1) warp_rank64(tile, q0.x, q1.x, in0, in1, two, key_bits, lane, r0, r1);
            if (in0) {
                rk[lo + r0] = q0.x;
                rv[lo + r0] = q0.y;
            }
            if (in1) {
                rk[lo + r1] = q1.x;
                rv[lo + r1] = q1.y;
            }
        }
        g0 = f0;
        g1 = f1;
    }
}

// Buckets of 65..256 keys in registers of one warp; larger ones are flagged
// for the shared-memory sort.
// The lanes of a warp look at 32 buckets at once; the warp then sorts the
// ones it has to, one after the other.
__global__ void __launch_bounds__(256, 2) k_warp_sort_big_q(const BatchDesc* __restrict__ D) {
    const int lane = threadIdx.x & 31;
    const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    if (!(*D->err & DERR_SORT_BIG)) return;
    const uint64_t nb = D->n_buckets;
    for (uint64_t base = warp * 32; base < nb; base += n_warps * 32) {
        const uint64_t fb = base + (uint64_t)lane;
        const uint64_t m64 = fb < nb ? D->starts[fb + 1] - D->starts[fb] : 0ull;
        unsigned todo = __ballot_sync(kFull, m64 > 64);
        while (todo) {
            const int src = __ffs(todo) - 1;
            todo &= todo - 1;
            const uint64_t b = base + (uint64_t)src;
            const uint64_t n64 = __shfl_sync(kFull, m64, src);
            if (n64 > 256) {
                if (lane == 0) atomicOr(D->err, DERR_SORT_MEDIUM);
                continue;
            }
            const JobDesc& J = D->jobs[job_of_bucket(D, b)];
            const uint64_t lo = D->starts[b] - D->starts[J.bucket_base];
            const int n = (int)n64;
            if (n <= 128) warp_sort_bucket<4>(J.res_keys, J.res_vals, lo, n, lane);
            else warp_sort_bucket<8>(J.res_keys, J.res_vals, lo, n, lane);
        }
    }
}

// Buckets of 257..2048 keys: one CTA each, bitonic network in shared memory
// (mirror form, indices >= n act as +infinity).  Larger ones are flagged.
constexpr int kMedCap = 2048;

__global__ void __launch_bounds__(256) k_medium_sort_q(const BatchDesc* __restrict__ D) {
    __shared__ uint64_t sk[kMedCap];
    __shared__ uint64_t sv[kMedCap];
    for (uint64_t fb = blockIdx.x; fb < D->n_buckets; fb += gridDim.x) {
        const uint64_t n64 = D->starts[fb + 1] - D->starts[fb];
        if (n64 <= 256) continue;
        if (n64 > (uint64_t)kMedCap) {
            if (threadIdx.x == 0) atomicOr(D->err, DERR_SORT_BUCKET);
            continue;
        }
        const JobDesc& J = D->jobs[job_of_bucket(D, fb)];
        const uint64_t lo = D->starts[fb] - D->starts[J.bucket_base];
        const int n = (int)n64;
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            sk[i] = J.res_keys[lo + i];
            sv[i] = J.res_vals[lo + i];
        }
        int n2 = 1;
        while (n2 < n) n2 <<= 1;
        __syncthreads();
        for (int size = 2; size <= n2; size <<= 1) {
            const int half = size >> 1;
            for (int i = threadIdx.x; i < (n2 >> 1); i += blockDim.x) {
                const int blk = i / half, off = i % half;
                const int x = blk * size + off, y = blk * size + size - 1 - off;
                if (y < n && sk[x] > sk[y]) {
                    const uint64_t tk = sk[x], tv = sv[x];
                    sk[x] = sk[y];
                    sv[x] = sv[y];
                    sk[y] = tk;
                    sv[y] = tv;
                }
            }
            __syncthreads();
            for (int stride = size >> 2; stride > 0; stride >>= 1) {
                for (int i = threadIdx.x; i < (n2 >> 1); i += blockDim.x) {
                    const int x = 2 * i - (i & (stride - 1)), y = x + stride;
                    if (y < n && sk[x] > sk[y]) {
                        const uint64_t tk = sk[x], tv = sv[x];
                        sk[x] = sk[y];
                        sv[x] = sv[y];
                        sk[y] = tk;
                        sv[y] = tv;
                    }
                }
                __syncthreads();
            }
        }
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            J.res_keys[lo + i] = sk[i];
            J.res_vals[lo + i] = sv[i];
        }
        __syncthreads();
    }
}

}  // namespace
}  // namespace kc

using namespace kcapi;

struct kc_batch_ctx {
    cudaStream_t st = nullptr;
    bool own_stream = false;
    int device = 0, sm_count = 152, max_optin = 0, max_sm = 0;
    kc::BatchDesc* d_desc = nullptr;
    kc::JobDesc* d_jobs = nullptr;
    uint32_t* d_item_job = nullptr;
    unsigned long long* d_counters = nullptr;
    unsigned int* d_flags = nullptr;  // [0] queue head, [1] sort error bits
    size_t jobs_cap = 0, items_cap = 0;
    uint32_t* d_hist = nullptr;
    uint64_t* d_starts = nullptr;
    uint64_t* d_cursor = nullptr;
    unsigned long long* d_tiles = nullptr;
    uint64_t buckets_cap = 0, tiles_cap = 0;
    cudaGraphExec_t sort_graph[2] = {nullptr, nullptr};  // [1]: the consumer has counted the buckets
    // captured consumer launches, one per launch shape
    struct ConsumeGraph {
        bool one;  // one sample in every job
        int threads, n_ctas;
        size_t smem;
        cudaGraphExec_t exec;
    };
    std::vector<ConsumeGraph> consume_graphs;
    std::vector<kc::JobDesc> jobs;
    std::vector<uint32_t> item_job;
    uint64_t launches = 0;
    // pinned host memory the finalize reads its counters back into (so the
    // copies queue behind the kernels and one synchronisation waits for all)
    unsigned char* h_read = nullptr;
    size_t h_read_jobs = 0;
    // the scattered survivors of a batch, (key, value) pairs
    ulonglong2* d_pairs = nullptr;
    size_t pairs_cap = 0;
};

namespace {

template <class T>
kc_status grow(T*& p, size_t& cap, size_t need) {
    if (need <= cap) return KC_OK;
    size_t n = std::max<size_t>(need, cap * 2);
    std::lock_guard<std::mutex> lk(kc::sync_api_mutex());
    if (p) cudaFree(p);
    p = nullptr;
    cap = 0;
    KC_CUDA(kc::dev_alloc_fixed(&p, n * sizeof(T)));
    cap = n;
    return KC_OK;
}

kc_status ensure_jobs(kc_batch_ctx* b, size_t n_jobs, size_t n_items) {
    if (n_jobs > b->jobs_cap) {
        size_t n = std::max<size_t>(n_jobs, b->jobs_cap * 2);
        std::lock_guard<std::mutex> lk(kc::sync_api_mutex());
        if (b->d_jobs) cudaFree(b->d_jobs);
        if (b->d_counters) cudaFree(b->d_counters);
        b->d_jobs = nullptr;
        b->d_counters = nullptr;
        b->jobs_cap = 0;
        KC_CUDA(kc::dev_alloc_fixed(&b->d_jobs, n * sizeof(kc::JobDesc)));
        KC_CUDA(kc::dev_alloc_fixed(&b->d_counters, 2 * n * sizeof(unsigned long long)));
        b->jobs_cap = n;
    }
    size_t cap = b->items_cap;
    kc_status s = grow(b->d_item_job, cap, n_items);
    b->items_cap = cap;
    return s;
}

// Readback area for n jobs: the error word, then 2 n queue counters, then n
// device-counter blocks.
kc_status ensure_readback(kc_batch_ctx* b, size_t n) {
    if (n <= b->h_read_jobs) return KC_OK;
    const size_t m = std::max<size_t>(n, 2 * b->h_read_jobs);
    std::lock_guard<std::mutex> lk(kc::sync_api_mutex());  // pinning may synchronise the device
    if (b->h_read) cudaFreeHost(b->h_read);
    b->h_read = nullptr;
    b->h_read_jobs = 0;
    KC_CUDA(cudaMallocHost(&b->h_read, 64 + m * (16 + sizeof(kc::DevCounters))));
    b->h_read_jobs = m;
    return KC_OK;
}

kc_status ensure_buckets(kc_batch_ctx* b, uint64_t n_buckets) {
    if (n_buckets <= b->buckets_cap) return KC_OK;
    const uint64_t n = std::max<uint64_t>(n_buckets, 1ull << 16);
    std::lock_guard<std::mutex> lk(kc::sync_api_mutex());
    if (b->d_hist) cudaFree(b->d_hist);
    if (b->d_starts) cudaFree(b->d_starts);
    if (b->d_cursor) cudaFree(b->d_cursor);
    if (b->d_tiles) cudaFree(b->d_tiles);
    b->d_hist = nullptr;
    b->d_starts = b->d_cursor = nullptr;
    b->d_tiles = nullptr;
    b->buckets_cap = 0;
    const uint64_t tiles = (n + kc::kScanTile - 1) / kc::kScanTile;
    KC_CUDA(kc::dev_alloc_fixed(&b->d_hist, n * 4));
    KC_CUDA(kc::dev_alloc_fixed(&b->d_starts, (n + 1) * 8));
    KC_CUDA(kc::dev_alloc_fixed(&b->d_cursor, n * 8));
    KC_CUDA(kc::dev_alloc_fixed(&b->d_tiles, (tiles + 1) * 8));
    b->buckets_cap = n;
    b->tiles_cap = tiles;
    for (cudaGraphExec_t& g : b->sort_graph)
        if (g) {  // the graph holds the old capacities
            cudaGraphExecDestroy(g);
            g = nullptr;
        }
    return KC_OK;
}

// Capture the sort sequence once (early: without the histogram the consumer
// has taken); it reads everything else from d_desc.
kc_status capture_sort_graph(kc_batch_ctx* b, int early) {
    if (b->sort_graph[early]) return KC_OK;
    std::lock_guard<std::mutex> lk(kc::sync_api_mutex());
    cudaGraph_t g = nullptr;
    KC_CUDA(cudaStreamBeginCapture(b->st, cudaStreamCaptureModeThreadLocal));
    const unsigned grid2 = (unsigned)b->sm_count * 16;  // latency-bound atomics: many threads in flight
    kc::k_plan_q<<<1, 512, 0, b->st>>>(b->d_desc);
    if (!early) {
        kc::k_zero_hist_q<<<(unsigned)b->sm_count * 4, 256, 0, b->st>>>(b->d_desc);
        kc::k_prefix_hist_q<<<grid2, 256, 0, b->st>>>(b->d_desc);
    }
    kc::k_scan_q<<<(unsigned)b->tiles_cap, kc::kScanThreads, 0, b->st>>>(b->d_desc);
    kc::k_scatter_q<<<grid2, 256, 0, b->st>>>(b->d_desc);
    kc::k_warp_sort_q<<<(unsigned)b->sm_count * 6, 256, 0, b->st>>>(b->d_desc);
    kc::k_warp_sort_big_q<<<(unsigned)b->sm_count * 2, 256, 0, b->st>>>(b->d_desc);
    cudaError_t e = cudaStreamEndCapture(b->st, &g);
    if (e != cudaSuccess) return cuda_fail(e, "cudaStreamEndCapture(sort)");
    e = cudaGraphInstantiate(&b->sort_graph[early], g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGraphInstantiate(sort)");
    return KC_OK;
}

kc_status upload_desc(kc_batch_ctx* b, uint32_t n_jobs, uint32_t n_items, uint64_t n_buckets) {
    kc::BatchDesc d{};
    d.pairs = b->d_pairs;
    d.pairs_cap = b->pairs_cap;
    d.buckets_cap = b->buckets_cap;
    d.jobs = b->d_jobs;
    d.item_job = b->d_item_job;
    d.counters = b->d_counters;
    d.head = b->d_flags;
    d.err = b->d_flags + 1;
    d.n_jobs = n_jobs;
    d.n_items = n_items;
    d.n_buckets = n_buckets;
    d.hist = b->d_hist;
    d.starts = b->d_starts;
    d.cursor = b->d_cursor;
    d.tiles = b->d_tiles;
    d.n_tiles = b->tiles_cap;
    KC_CUDA(cudaMemcpyAsync(b->d_desc, &d, sizeof(d), cudaMemcpyHostToDevice, b->st));
    KC_CUDA(cudaMemcpyAsync(b->d_jobs, b->jobs.data(), n_jobs * sizeof(kc::JobDesc), cudaMemcpyHostToDevice, b->st));
    return KC_OK;
}

// Split levels a table of the library's own size may take beyond a limit set by
// the caller: up to 32 keys seen once for each that is not.
constexpr int kSplitLevelsForSingles = 5;

struct JobWork {
    kc_handle h;
    std::vector<uint64_t> hs;  // partition starts of every batch
    uint64_t total_w = 0, max_w = 0;
    // survivors: keys, then values, in one block of the handle's (take_block)
    uint64_t* sv_keys = nullptr;
    uint64_t* sv_vals = nullptr;
    uint64_t sv_cap = 0;
    size_t sv_bytes = 0;
    uint64_t* failed = nullptr;  // failed partitions, then the batches' pointers (meta)
    void* meta = nullptr;
};

// The jobs' blocks of one finalize, given back when it returns.  They go to the
// batch's stream, so that stream must be ordered after the handles' by then: a
// survivors' block may be the scratch of a grouping still queued on its handle's
// stream.  A finalize that fails before it has queued that order waits for the
// handles here.
struct WorkSet {
    kc_batch_ctx* b;
    std::vector<JobWork> jobs;
    bool ordered = false;
    WorkSet(kc_batch_ctx* batch, size_t n) : b(batch), jobs(n) {}
    WorkSet(const WorkSet&) = delete;
    WorkSet& operator=(const WorkSet&) = delete;
    JobWork& operator[](size_t j) { return jobs[j]; }
    ~WorkSet() {
        for (auto& x : jobs) {
            if (x.sv_keys && !ordered) cudaStreamSynchronize(x.h->stream);
            if (x.sv_keys) cudaFreeAsync(x.sv_keys, b->st);
            if (x.failed) cudaFreeAsync(x.failed, b->st);
        }
    }
};

// prepare: set the kernel's shared-memory limit (before any capture);
// otherwise launch it.
cudaError_t launch_consume(bool prepare, bool one, int threads, int n_ctas, size_t smem, const kc::BatchDesc* d, cudaStream_t st) {
    const auto go = [&](auto kern) {
        if (prepare) return kc::allow_max_dynamic_smem(kern);
        kern<<<n_ctas, threads, smem, st>>>(d);
        return cudaGetLastError();
    };
    if (threads == kc::kConsumeThreads)
        return one ? go(kc::k_consume_q<kc::kConsumeThreads, true>) : go(kc::k_consume_q<kc::kConsumeThreads, false>);
    return one ? go(kc::k_consume_q<kc::kConsumeThreadsWide, true>) : go(kc::k_consume_q<kc::kConsumeThreadsWide, false>);
}

// The batch's counters reset and its persistent consumer launch, captured
// once per launch shape (samples, CTA size, grid, shared memory); everything else
// they read comes from the device descriptor.
kc_status consume_graph(kc_batch_ctx* b, bool one, int threads, int n_ctas, size_t smem, cudaGraphExec_t* out) {
    for (const auto& g : b->consume_graphs)
        if (g.one == one && g.threads == threads && g.n_ctas == n_ctas && g.smem == smem) {
            *out = g.exec;
            return KC_OK;
        }
    KC_CUDA(launch_consume(true, one, threads, n_ctas, smem, b->d_desc, b->st));
    std::lock_guard<std::mutex> lk(kc::sync_api_mutex());
    cudaGraph_t g = nullptr;
    KC_CUDA(cudaStreamBeginCapture(b->st, cudaStreamCaptureModeThreadLocal));
    kc::k_reset_q<<<1, 256, 0, b->st>>>(b->d_desc);
    launch_consume(false, one, threads, n_ctas, smem, b->d_desc, b->st);
    cudaError_t e = cudaStreamEndCapture(b->st, &g);
    if (e != cudaSuccess) return cuda_fail(e, "cudaStreamEndCapture(consumer)");
    cudaGraphExec_t exec = nullptr;
    e = cudaGraphInstantiate(&exec, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGraphInstantiate(consumer)");
    b->consume_graphs.push_back({one, threads, n_ctas, smem, exec});
    *out = exec;
    return KC_OK;
}

// Bucket bits of a sort of at most n survivors (about 32 a bucket).
int sort_bits_for(uint64_t n, int key_bits) {
    int bits = 0;
    n = std::max<uint64_t>(1, n);
    while (bits < 24 && bits < key_bits && (n >> bits) > 32) ++bits;
    return bits;
}

// Partitions whose shared-memory table overflowed: rebuild their filter
// slice from zero and count them in a global table (kc_partition.cu kernels).
kc_status run_fallbacks(kc_batch_ctx* b, JobWork& x, uint32_t j, uint32_t n_failed) {
    kc_handle h = x.h;
    const kc::JobDesc& J = b->jobs[j];
    const uint64_t P = 1ull << h->part_bits;
    const size_t nb = h->batches.size();
    std::vector<uint64_t> fl(n_failed);  // first hash of each partition not yet counted
    KC_CUDA(cudaMemcpyAsync(fl.data(), x.failed, n_failed * 8, cudaMemcpyDeviceToHost, b->st));
    unsigned long long n_sv = 0;
    KC_CUDA(cudaMemcpyAsync(&n_sv, b->d_counters + 2 * j, 8, cudaMemcpyDeviceToHost, b->st));
    if (x.hs.empty()) {  // sized from the host's counts: the partition starts were not read yet
        x.hs.resize(nb * (P + 1));
        for (size_t t = 0; t < nb; ++t)
            KC_CUDA(cudaMemcpyAsync(x.hs.data() + t * (P + 1), h->batches[t].hstarts, (P + 1) * 8,
                                    cudaMemcpyDeviceToHost, b->st));
    }
    KC_CUDA(cudaStreamSynchronize(b->st));
    auto windows_of = [&](uint32_t p) {
        uint64_t w = 0;
        for (size_t t = 0; t < nb; ++t) w += x.hs[t * (P + 1) + p + 1] - x.hs[t * (P + 1) + p];
        return w;
    };
    const int a = h->part_bits;
    uint64_t extra = 0;
    for (uint64_t hl : fl) extra += windows_of((uint32_t)(hl >> (64 - a)));
    const uint64_t need = n_sv + extra;
    if (need > x.sv_cap) {
        uint64_t* nk = nullptr;
        cudaError_t e = kc::dev_alloc(&nk, need * 16, b->st);
        if (e != cudaSuccess) return cuda_fail(e, "cudaMallocAsync(fallback survivors)");
        uint64_t* nv = nk + need;
        const uint64_t have = std::min<uint64_t>(n_sv, x.sv_cap);
        KC_CUDA(cudaMemcpyAsync(nk, x.sv_keys, have * 8, cudaMemcpyDeviceToDevice, b->st));
        KC_CUDA(cudaMemcpyAsync(nv, x.sv_vals, have * 8, cudaMemcpyDeviceToDevice, b->st));
        cudaFreeAsync(x.sv_keys, b->st);
        x.sv_keys = nk;
        x.sv_vals = nv;
        x.sv_cap = need;
        x.sv_bytes = need * 16;
    }
    const uint64_t n_sw = 1ull << h->slice_log2;
    for (uint64_t hl : fl) {
        const uint32_t p = (uint32_t)(hl >> (64 - a));
        const uint64_t w_lo = (hl >> J.bloom_shift) & (n_sw - 1);  // sub-ranges below are finished
        uint64_t slots = 1024;
        while (slots < 2 * windows_of(p)) slots <<= 1;
        kc::Slot* table = nullptr;
        cudaError_t e = kc::dev_alloc(&table, slots * sizeof(kc::Slot), b->st);
        if (e != cudaSuccess) return cuda_fail(e, "cudaMallocAsync(fallback table)");
        KC_CUDA(cudaMemsetAsync(table, 0, slots * sizeof(kc::Slot), b->st));
        KC_CUDA(cudaMemsetAsync(h->bloom + p * n_sw + w_lo, 0, (n_sw - w_lo) * 8, b->st));
        kc::FallbackArgs F{};
        F.data = J.data;
        F.starts = J.starts;
        F.samples = J.samples;
        F.part = p;
        F.h_lo = hl;
        F.part_bits = h->part_bits;
        F.bloom_shift = J.bloom_shift;
        F.n_hashes = h->n_hashes;
        F.n_samples = h->n_samples;
        F.all_candidates = J.all_candidates;
        F.min_count = h->min_count;
        F.bloom = reinterpret_cast<unsigned long long*>(h->bloom);
        F.table = table;
        F.table_mask = slots - 1;
        F.out_keys = x.sv_keys;
        F.out_vals = x.sv_vals;
        F.out_cap = x.sv_cap;
        F.n_out = b->d_counters + 2 * j;
        F.ctr = h->ctr;
        for (size_t t = 0; t < nb; ++t) kc::launch_fb_claim(F, (int)t, b->st);
        for (size_t t = 0; t < nb; ++t) kc::launch_fb_recount(F, (int)t, b->st);
        kc::launch_fb_compact(F, b->st);
        h->launches += 2 * nb + 1;
        KC_LAUNCHED("fallback launches");
        cudaFreeAsync(table, b->st);
    }
    h->fallback_partitions += n_failed;
    return KC_OK;
}

}  // namespace

kc_status kc_batch_create_internal(cudaStream_t st, kc_batch_ctx** out) {
    *out = nullptr;
    kc_batch_ctx* b = new (std::nothrow) kc_batch_ctx();
    if (!b) return fail(KC_ERR_OOM_HOST, "host allocation");
    auto bail = [&](kc_status s) {
        kc_batch_destroy_internal(b);
        return s;
    };
    cudaError_t e = cudaGetDevice(&b->device);
    if (e != cudaSuccess) return bail(cuda_fail(e, "cudaGetDevice"));
    cudaDeviceGetAttribute(&b->sm_count, cudaDevAttrMultiProcessorCount, b->device);
    cudaDeviceGetAttribute(&b->max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, b->device);
    cudaDeviceGetAttribute(&b->max_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, b->device);
    if (st) {
        b->st = st;
    } else {
        if ((e = cudaStreamCreateWithFlags(&b->st, cudaStreamNonBlocking)) != cudaSuccess)
            return bail(cuda_fail(e, "cudaStreamCreate"));
        b->own_stream = true;
    }
    {
        std::lock_guard<std::mutex> lk(kc::sync_api_mutex());
        if ((e = kc::dev_alloc_fixed(&b->d_desc, sizeof(kc::BatchDesc))) == cudaSuccess)
            e = kc::dev_alloc_fixed(&b->d_flags, 2 * sizeof(unsigned int));
    }
    if (e != cudaSuccess) return bail(cuda_fail(e, "cudaMalloc(batch descriptor)"));  // after the lock: bail takes it again
    *out = b;
    return KC_OK;
}

void kc_batch_destroy_internal(kc_batch_ctx* b) {
    if (!b) return;
    if (b->st) cudaStreamSynchronize(b->st);
    for (cudaGraphExec_t g : b->sort_graph)
        if (g) cudaGraphExecDestroy(g);
    for (auto& g : b->consume_graphs) cudaGraphExecDestroy(g.exec);
    std::lock_guard<std::mutex> lk(kc::sync_api_mutex());
    cudaFree(b->d_desc);
    cudaFree(b->d_flags);
    cudaFree(b->d_jobs);
    cudaFree(b->d_counters);
    cudaFree(b->d_item_job);
    cudaFree(b->d_hist);
    cudaFree(b->d_starts);
    cudaFree(b->d_cursor);
    cudaFree(b->d_tiles);
    if (b->h_read) cudaFreeHost(b->h_read);
    cudaFree(b->d_pairs);
    if (b->own_stream && b->st) cudaStreamDestroy(b->st);
    delete b;
}

// Finalize partitions [part_lo, part_hi) of every job (clamped to the job's
// partition count); the handles become finalized only when `last`.
kc_status finalize_core(kc_batch_ctx* b, kc_handle* hs, int n, uint32_t part_lo, uint32_t part_hi, bool last) {
    if (!b || !hs || n < 0) return fail(KC_ERR_ARG, "null argument");
    if (n == 0) return KC_OK;
    cudaStream_t st = b->st;
    WorkSet work(b, (size_t)n);
    const bool one = n == 1 && hs[0]->stream == st;  // no cross-stream ordering needed
    const bool timed = n == 1;                         // phase times go to the only handle
    bool fast = true;  // every job whole: sized from host counts (below)
    for (int j = 0; j < n; ++j) {
        kc_handle h = hs[j];
        if (!h) return fail(KC_ERR_ARG, "null handle in batch");
        if (h->state == State::Poisoned) return fail(KC_ERR_STATE, "handle poisoned by an earlier error; call kc_reset");
        if (h->state != State::Open) return fail(KC_ERR_STATE, "handle already finalized");
        if (h->strategy != KC_STRATEGY_PARTITIONED) return fail(KC_ERR_ARG, "batched finalize needs the partitioned strategy");
        for (int i = 0; i < j; ++i)
            if (hs[i] == h) return fail(KC_ERR_ARG, "handle listed twice");
        work[j].h = h;
        fast = fast && part_lo == 0 && part_hi >= (1u << h->part_bits) && !h->owner && !h->deferred;
    }
    // order the batch after every handle's queued work: at once when the
    // setup reads the grouping back, else just before the consumer, so the
    // setup's uploads queue while the handles' grouping still runs
    const auto order_after_handles = [&]() -> kc_status {
        if (!one)
            for (int j = 0; j < n; ++j) {
                KC_CUDA(cudaEventRecord(hs[j]->ev_main, hs[j]->stream));
                KC_CUDA(cudaStreamWaitEvent(st, hs[j]->ev_main, 0));
            }
        work.ordered = true;
        return KC_OK;
    };
    if (!fast) {
        kc_status os = order_after_handles();
        if (os != KC_OK) return os;
    }
    // Partition sizes of every job, and each job's counters (ingest errors):
    // read back when the batch covers part of a job's partitions (spill
    // groups, owned ranges, hash ranges of kept reads).  A job counted whole
    // is sized from the host's counts instead (bases and reads added), so no
    // host round trip sits between its grouping and its consumer; its ingest
    // errors are read after the consumer.
    kc_status rs = ensure_readback(b, (size_t)n);
    if (rs != KC_OK) return rs;
    unsigned& err = *reinterpret_cast<unsigned*>(b->h_read);
    unsigned long long* cnt = reinterpret_cast<unsigned long long*>(b->h_read + 64);
    kc::DevCounters* hc = reinterpret_cast<kc::DevCounters*>(b->h_read + 64 + 16 * (size_t)n);
    if (!fast) {
        for (int j = 0; j < n; ++j) {
            kc_handle h = hs[j];
            const uint64_t P = 1ull << h->part_bits;
            work[j].hs.resize(h->batches.size() * (P + 1));
            for (size_t t = 0; t < h->batches.size(); ++t)
                KC_CUDA(cudaMemcpyAsync(work[j].hs.data() + t * (P + 1), h->batches[t].hstarts, (P + 1) * 8,
                                        cudaMemcpyDeviceToHost, st));
            KC_CUDA(cudaMemcpyAsync(&hc[j], h->ctr, sizeof(kc::DevCounters), cudaMemcpyDeviceToHost, st));
        }
        KC_CUDA(cudaStreamSynchronize(st));
        for (int j = 0; j < n; ++j) {
            hs[j]->host_ctr = hc[j];
            kc_status s = device_errors(hs[j]);
            if (s != KC_OK) return s;
        }
    }

    // per-job consumer setup
    b->jobs.assign((size_t)n, kc::JobDesc{});
    b->item_job.clear();
    size_t smem_max = 0;
    for (int j = 0; j < n; ++j) {
        JobWork& x = work[j];
        kc_handle h = x.h;
        const uint64_t P = 1ull << h->part_bits;
        // the requested partitions that the handle owns (kc_config.own_bits)
        const uint64_t p_lo = std::max<uint64_t>(std::min<uint64_t>(part_lo, P), h->own_plo);
        const uint64_t p_hi = std::max<uint64_t>(p_lo, std::min<uint64_t>(std::min<uint64_t>(part_hi, P), h->own_phi));
        const size_t nb = h->batches.size();
        if (fast) {
            // windows: at most one per base; about bases - reads (k - 1), spread
            // evenly over the partitions by the hash
            const uint64_t est = h->bases > h->reads * (uint64_t)(h->k - 1) ? h->bases - h->reads * (uint64_t)(h->k - 1) : 0;
            x.total_w = h->bases;
            x.max_w = est / P + est / P / 16 + 64;
        } else {
            for (uint64_t p = p_lo; p < p_hi; ++p) {
                uint64_t w = 0;
                for (size_t t = 0; t < nb; ++t) w += x.hs[t * (P + 1) + p + 1] - x.hs[t * (P + 1) + p];
                x.max_w = std::max(x.max_w, w);
                x.total_w += w;
            }
        }
        // Split level: a sub-range's filter words take at most 64 KiB.
        const int split_min = std::max(0, h->slice_log2 - kc::kConsumeSliceLog2);
        // Shared-memory table: twice the windows of the largest partition
        // (2^10..2^13 slots, or 2^14), so that small partitions never split; a
        // larger partition's distinct keys fit or it splits.
        int tl = (int)h->cfg.smem_table_log2;
        if (!tl) {
            tl = 10;
            while (tl < 13 && (1ull << tl) < 2 * (x.max_w >> split_min)) ++tl;
            // one-sample partitions beyond what 8192 slots take at 30x coverage
            // (one distinct key in six windows): 16384 slots and one wide CTA an
            // SM, instead of two passes (1.8e8 windows, 43,700 a partition: 1.48 -> 1.16 ms)
            if (h->n_samples == 1 && (x.max_w >> split_min) > 40960) tl = 14;
        }
        const size_t queue = kc::consume_queue_smem(kc::kConsumeThreadsWide) + 1024;
        while (tl > 10 && kc::consume_smem(h->slice_log2 - split_min, tl, h->n_samples) + queue > (size_t)b->max_optin) --tl;
        const size_t smem = kc::consume_smem(h->slice_log2 - split_min, tl, h->n_samples);
        if (smem + queue > (size_t)b->max_optin) {
            return fail(KC_ERR_INTERNAL, "partition does not fit shared memory");
        }
        smem_max = std::max(smem_max, smem);
        // survivors: a partition holds at most 2^split_max tables of keys and
        // one key per min_count of its windows
        // the consumer tells a window's sub-range by the top 32 bits of its hash
        // A limit set by the caller is about keys seen more than once; a table of the
        // library's own size holds those seen once too and may split that much further
        // (two samples of 30x coverage in 2048 partitions with KC_SPLIT_NONE: 76 ms in
        // global tables, 2.3 split)
        const bool limited = h->cfg.split_max != 0;
        int levels = h->cfg.split_max == KC_SPLIT_NONE ? 0 : limited ? (int)h->cfg.split_max : 8;
        if (limited && !h->cfg.smem_table_log2) levels += kSplitLevelsForSingles;
        const int split_max = std::max(split_min, std::min({h->slice_log2, 32 - h->part_bits, levels}));
        x.sv_cap = 0;
        if (fast) {  // every survivor has min_count windows, and no partition more than 2^split_max tables
            x.sv_cap = std::min<uint64_t>((p_hi - p_lo) << (tl + split_max), x.total_w / std::max<uint32_t>(1, h->min_count));
        } else {
            for (uint64_t p = p_lo; p < p_hi; ++p) {
                uint64_t w = 0;
                for (size_t t = 0; t < nb; ++t) w += x.hs[t * (P + 1) + p + 1] - x.hs[t * (P + 1) + p];
                x.sv_cap += std::min<uint64_t>(1ull << (tl + split_max), w / std::max<uint32_t>(1, h->min_count));
            }
        }
        x.sv_cap = std::max<uint64_t>(1, x.sv_cap);
        const size_t meta_bytes = std::max<size_t>(16, nb * 20);
        cudaError_t e;
        // (the survivors' block is first used by the consumer, after the
        // handle's stream; the other one is written at once)
        x.sv_bytes = x.sv_cap * 16;
        if ((e = take_block(h, reinterpret_cast<void**>(&x.sv_keys), &x.sv_bytes, st)) != cudaSuccess ||
            (e = kc::dev_alloc(&x.failed, P * 8 + meta_bytes, st)) != cudaSuccess) {
            return cuda_fail(e, "cudaMallocAsync(batch consumer)");
        }
        x.sv_vals = x.sv_keys + x.sv_cap;
        x.meta = x.failed + P;
        std::vector<unsigned char> hm(meta_bytes, 0);
        for (size_t t = 0; t < nb; ++t) {
            const uint64_t dp = (uint64_t)(uintptr_t)h->batches[t].hdata;
            const uint64_t sp = (uint64_t)(uintptr_t)h->batches[t].hstarts;
            const int smp = h->batches[t].sample;
            std::memcpy(hm.data() + t * 8, &dp, 8);
            std::memcpy(hm.data() + nb * 8 + t * 8, &sp, 8);
            std::memcpy(hm.data() + nb * 16 + t * 4, &smp, 4);
        }
        KC_CUDA(cudaMemcpyAsync(x.meta, hm.data(), meta_bytes, cudaMemcpyHostToDevice, st));
        kc::JobDesc& J = b->jobs[j];
        J.part_bits = h->part_bits;
        J.slice_log2 = h->slice_log2;
        J.table_log2 = tl;
        J.bloom_shift = 64 - h->log2_words;
        J.n_hashes = h->n_hashes;
        J.n_samples = h->n_samples;
        J.all_candidates = h->min_count <= 1 ? 1 : 0;
        J.key_bits = 2 * h->k;
        J.min_count = h->min_count;
        J.split_max = split_max;
        J.split_min = split_min;
        J.fixed_bits = -1;  // the plan chooses the bucket bits (unless set below)
        J.hist_job = nullptr;
        J.n_batches = (int)nb;
        J.item_base = (uint32_t)b->item_job.size();
        J.part_base = (uint32_t)p_lo;
        J.data = reinterpret_cast<const uint64_t* const*>(x.meta);
        J.starts = reinterpret_cast<const uint64_t* const*>(static_cast<char*>(x.meta) + nb * 8);
        J.samples = reinterpret_cast<const int*>(static_cast<char*>(x.meta) + nb * 16);
        J.bloom = reinterpret_cast<unsigned long long*>(h->bloom);
        J.sv_keys = x.sv_keys;
        J.sv_vals = x.sv_vals;
        J.sv_cap = x.sv_cap;
        J.failed = x.failed;
        J.ctr = h->ctr;
        for (uint64_t p = p_lo; p < p_hi; ++p) b->item_job.push_back((uint32_t)j);
    }
    const uint32_t n_items = (uint32_t)b->item_job.size();
    kc_status s = ensure_jobs(b, (size_t)n, n_items);
    if (s != KC_OK) {
        return s;
    }
    KC_CUDA(cudaMemcpyAsync(b->d_item_job, b->item_job.data(), n_items * 4, cudaMemcpyHostToDevice, st));
    // Whole jobs whose handles still hold result arrays from their last job:
    // the sort graph runs right behind the consumer into those arrays, with
    // bucket arrays for that many survivors, and one host round trip checks
    // both (no partition left to the fallback, every job's survivors within
    // its arrays); otherwise the sort runs again after the fallbacks, into
    // arrays of the right size.
    // The bucket bits are then fixed in advance (for the kept arrays' size),
    // so the consumer histograms the survivors as it writes them and the sort
    // graph skips its histogram pass.
    bool spec = fast;
    for (int j = 0; j < n && spec; ++j) spec = hs[j]->res_keys != nullptr && hs[j]->res_cap > 0;
    uint64_t spec_buckets = 0;
    if (spec) {
        for (int j = 0; j < n; ++j) {
            kc::JobDesc& J = b->jobs[j];
            J.fixed_bits = sort_bits_for(std::min<uint64_t>(hs[j]->res_cap, J.sv_cap), J.key_bits);
            spec_buckets += 1ull << J.fixed_bits;
            J.res_keys = hs[j]->res_keys;
            J.res_vals = hs[j]->res_vals;
            J.res_cap = hs[j]->res_cap;
        }
        uint64_t spec_pairs = 0;
        for (int j = 0; j < n; ++j) spec_pairs += hs[j]->res_cap;
        if ((s = ensure_buckets(b, spec_buckets)) != KC_OK || (s = grow(b->d_pairs, b->pairs_cap, spec_pairs)) != KC_OK ||
            (s = capture_sort_graph(b, 1)) != KC_OK) {
            return s;
        }
        uint64_t first = 0;  // the plan gives the jobs their buckets in this order
        for (int j = 0; j < n; ++j) {
            b->jobs[j].hist_job = b->d_hist + first;
            first += 1ull << b->jobs[j].fixed_bits;
        }
        KC_CUDA(cudaMemsetAsync(b->d_hist, 0, spec_buckets * 4, st));
    }
    if ((s = upload_desc(b, (uint32_t)n, n_items, 0)) != KC_OK) {
        return s;
    }
    bool one_sample = true;
    for (int j = 0; j < n; ++j) one_sample = one_sample && hs[j]->n_samples == 1;
    // a persistent grid (CTAs without an item exit at once), so the captured
    // launch depends on the samples and the shared memory alone
    const size_t smem_cta = smem_max + kc::consume_queue_smem(kc::kConsumeThreads);
    int per_sm = std::min(2, b->max_sm / (int)(smem_cta + 2048));
    const int threads = per_sm > 1 ? kc::kConsumeThreads : kc::kConsumeThreadsWide;
    per_sm = std::max(1, per_sm);
    smem_max += kc::consume_queue_smem(threads);
    const int n_ctas = b->sm_count * per_sm;
    cudaGraphExec_t cons = nullptr;
    if ((s = consume_graph(b, one_sample, threads, n_ctas, smem_max, &cons)) != KC_OK) {
        return s;
    }

    if (fast && (s = order_after_handles()) != KC_OK) {
        return s;
    }
    // consume: one persistent launch over the (job, partition) queue
    cudaEvent_t t0 = timed ? phase_begin(hs[0], st) : nullptr;
    KC_CUDA(cudaGraphLaunch(cons, st));
    if (timed) phase_end(hs[0], kPass2, t0, st);
    err = 0;
    if (spec) {
        t0 = timed ? phase_begin(hs[0], st) : nullptr;
        KC_CUDA(cudaGraphLaunch(b->sort_graph[1], st));
        if (timed) phase_end(hs[0], kSort, t0, st);
        KC_CUDA(cudaMemcpyAsync(&err, b->d_flags + 1, 4, cudaMemcpyDeviceToHost, st));
    }
    KC_CUDA(cudaMemcpyAsync(cnt, b->d_counters, 2 * (size_t)n * 8, cudaMemcpyDeviceToHost, st));
    if (fast)
        for (int j = 0; j < n; ++j) KC_CUDA(cudaMemcpyAsync(&hc[j], hs[j]->ctr, sizeof(kc::DevCounters), cudaMemcpyDeviceToHost, st));
    KC_CUDA(cudaStreamSynchronize(st));
    for (int j = 0; j < n; ++j) work[j].h->launches += spec ? 7 : 2;
    if (fast) {
        for (int j = 0; j < n; ++j) {
            hs[j]->host_ctr = hc[j];
            kc_status s = device_errors(hs[j]);
            if (s != KC_OK) {
                return s;
            }
        }
    }

    // partitions whose table overflowed (rare): counted in global tables
    bool any_fb = false;
    for (int j = 0; j < n; ++j) any_fb |= cnt[2 * j + 1] != 0;
    bool sorted = spec && !any_fb && !(err & kc::DERR_INTERNAL);
    for (int j = 0; j < n && sorted; ++j) sorted = std::min<uint64_t>(cnt[2 * j], b->jobs[j].sv_cap) <= hs[j]->res_cap;
    if (sorted)
        for (int j = 0; j < n; ++j) hs[j]->n_result = std::min<uint64_t>(cnt[2 * j], b->jobs[j].sv_cap);
    if (any_fb) {
        for (int j = 0; j < n; ++j) {
            if (!cnt[2 * j + 1]) continue;
            t0 = timed ? phase_begin(hs[0], st) : nullptr;
            s = run_fallbacks(b, work[j], (uint32_t)j, (uint32_t)cnt[2 * j + 1]);
            if (timed) phase_end(hs[0], kCompact, t0, st);
            if (s != KC_OK) {
                return s;
            }
            kc::JobDesc& J = b->jobs[j];
            J.sv_keys = work[j].sv_keys;
            J.sv_vals = work[j].sv_vals;
            J.sv_cap = work[j].sv_cap;
        }
        KC_CUDA(cudaMemcpyAsync(cnt, b->d_counters, 2 * (size_t)n * 8, cudaMemcpyDeviceToHost, st));
        for (int j = 0; j < n; ++j) KC_CUDA(cudaMemcpyAsync(&hc[j], hs[j]->ctr, sizeof(kc::DevCounters), cudaMemcpyDeviceToHost, st));
        KC_CUDA(cudaStreamSynchronize(st));
        for (int j = 0; j < n; ++j) {
            hs[j]->host_ctr = hc[j];
            if ((s = device_errors(hs[j])) != KC_OK) {
                return s;
            }
        }
    }

    // sort: result arrays of each job's survivor count (a job's arrays are
    // kept for its next job when large enough), bucket arrays for as many
    // buckets as the plan will give; the plan itself runs on the device
    if (!sorted) {
    for (int j = 0; j < n; ++j) {  // the plan chooses the bits and the sort histograms again
        b->jobs[j].fixed_bits = -1;
        b->jobs[j].hist_job = nullptr;
    }
    uint64_t bucket_need = 0, pairs_need = 0;
    for (int j = 0; j < n; ++j) {
        kc_handle h = hs[j];
        kc::JobDesc& J = b->jobs[j];
        const uint64_t nsv = std::min<uint64_t>(cnt[2 * j], J.sv_cap);
        bucket_need += 1ull << sort_bits_for(nsv, J.key_bits);
        pairs_need += nsv;
        const uint64_t cap = std::max<uint64_t>(1, nsv);
        if (!h->res_keys || h->res_cap < cap) {
            free_result(h);
            cudaError_t e;
            if ((e = kc::dev_alloc(&h->res_keys, cap * 8, st)) != cudaSuccess ||
                (e = kc::dev_alloc(&h->res_vals, cap * 8, st)) != cudaSuccess) {
                free_result(h);
                return cuda_fail(e, "cudaMallocAsync(result)");
            }
            h->res_cap = cap;
        }
        h->n_result = nsv;
        J.res_keys = h->res_keys;
        J.res_vals = h->res_vals;
        J.res_cap = h->res_cap;
    }
    if ((s = ensure_buckets(b, bucket_need)) != KC_OK ||
        (s = grow(b->d_pairs, b->pairs_cap, std::max<uint64_t>(1, pairs_need))) != KC_OK ||
        (s = upload_desc(b, (uint32_t)n, n_items, 0)) != KC_OK ||
        (s = capture_sort_graph(b, 0)) != KC_OK) {
        return s;
    }
    t0 = timed ? phase_begin(hs[0], st) : nullptr;
    KC_CUDA(cudaGraphLaunch(b->sort_graph[0], st));
    if (timed) phase_end(hs[0], kSort, t0, st);
    KC_CUDA(cudaMemcpyAsync(&err, b->d_flags + 1, 4, cudaMemcpyDeviceToHost, st));
    KC_CUDA(cudaStreamSynchronize(st));
    for (int j = 0; j < n; ++j) work[j].h->launches += 7;
    }  // !sorted
    if (err & kc::DERR_INTERNAL) {
        for (int j = 0; j < n; ++j) hs[j]->state = State::Poisoned;
        return fail(KC_ERR_INTERNAL, "sort: key outside its bucket range");
    }
    t0 = timed && (err & (kc::DERR_SORT_MEDIUM | kc::DERR_SORT_BUCKET)) ? phase_begin(hs[0], st) : nullptr;
    if (err & kc::DERR_SORT_MEDIUM) {
        kc::k_medium_sort_q<<<(unsigned)b->sm_count * 4, 256, 0, st>>>(b->d_desc);
        KC_LAUNCHED("batched medium sort launch");
        KC_CUDA(cudaMemcpyAsync(&err, b->d_flags + 1, 4, cudaMemcpyDeviceToHost, st));
        KC_CUDA(cudaStreamSynchronize(st));
        for (int j = 0; j < n; ++j) hs[j]->launches += 1;
    }
    if (err & kc::DERR_SORT_BUCKET) {  // buckets above 2048 keys, sorted in global memory
        // the plan is on the device: read back the jobs' bucket ranges and the starts
        std::vector<kc::JobDesc> jd((size_t)n);
        uint64_t nbk = 0;
        KC_CUDA(cudaMemcpyAsync(jd.data(), b->d_jobs, n * sizeof(kc::JobDesc), cudaMemcpyDeviceToHost, st));
        KC_CUDA(cudaStreamSynchronize(st));
        for (const auto& J : jd) nbk = std::max<uint64_t>(nbk, J.bucket_base + J.n_buckets);
        std::vector<uint64_t> starts(nbk + 1);
        KC_CUDA(cudaMemcpyAsync(starts.data(), b->d_starts, (nbk + 1) * 8, cudaMemcpyDeviceToHost, st));
        KC_CUDA(cudaStreamSynchronize(st));
        std::vector<kc::SortRange> large;
        for (int j = 0; j < n; ++j) {
            const kc::JobDesc& J = jd[j];
            const uint64_t job0 = starts[J.bucket_base];
            for (uint64_t q = 0; q < J.n_buckets; ++q) {
                const uint64_t lo = starts[J.bucket_base + q], m = starts[J.bucket_base + q + 1] - lo;
                if (m > (uint64_t)kc::kMedCap) large.push_back({J.res_keys + (lo - job0), J.res_vals + (lo - job0), m});
            }
        }
        uint64_t steps = 0;
        if ((s = sort_ranges(large, st, &steps)) != KC_OK) return s;
        for (int j = 0; j < n; ++j) hs[j]->launches += steps;
    }
    if (t0) phase_end(hs[0], kSort, t0, st);
    KC_CUDA(cudaStreamSynchronize(st));
    for (JobWork& x : work.jobs) {  // nothing uses them any more
        leave_block(x.h, x.sv_keys, x.sv_bytes, st);
        x.sv_keys = x.sv_vals = nullptr;
    }
    for (int j = 0; j < n; ++j) {
        kc_handle h = hs[j];
        h->host_ctr.survivors = h->n_result;
        if (!one) {  // the handle's later work is ordered after the batch
            KC_CUDA(cudaEventRecord(h->ev_copy, st));
            KC_CUDA(cudaStreamWaitEvent(h->stream, h->ev_copy, 0));
        }
        phase_collect(h);
        if (last) h->state = State::Finalized;
    }
    b->launches += 9;
    return KC_OK;
}

// Out-of-core finalize of one handle: the partitions are processed in
// kSpillGroups hash-prefix groups in turn; each group's sorted survivors are
// copied to pinned host memory on the handle's side stream while the next
// group runs, and recorded in the spill directory (first partition, number
// of partitions, host location, items).  kc_dump merges the sorted runs.
constexpr uint32_t kSpillGroups = 64;

// Finalize partitions [part_lo, part_hi) of h and copy their sorted result to
// pinned host memory on the handle's side stream (one spill run).
kc_status spill_group(kc_batch_ctx* b, kc_handle h, uint32_t part_lo, uint32_t part_hi, bool last) {
    kc_status s = finalize_core(b, &h, 1, part_lo, part_hi, last);
    if (s != KC_OK) return s;
    SpillRun run;
    run.first_part = part_lo;
    run.n_parts = part_hi - part_lo;
    run.n_items = h->n_result;
    if (run.n_items) {
        run.host = spill_alloc(h, 2 * run.n_items);
        if (!run.host) return fail(KC_ERR_OOM_HOST, "pinned host memory for a spilled run");
        // the copy waits for the group's sort; the next group runs meanwhile
        KC_CUDA(cudaEventRecord(h->ev_main, b->st));
        KC_CUDA(cudaStreamWaitEvent(h->copy_stream, h->ev_main, 0));
        KC_CUDA(cudaMemcpyAsync(run.host, h->res_keys, run.n_items * 8, cudaMemcpyDeviceToHost, h->copy_stream));
        KC_CUDA(cudaMemcpyAsync(run.host + run.n_items, h->res_vals, run.n_items * 8, cudaMemcpyDeviceToHost,
                                h->copy_stream));
    }
    if (h->res_keys) cudaFreeAsync(h->res_keys, h->copy_stream);
    if (h->res_vals) cudaFreeAsync(h->res_vals, h->copy_stream);
    h->res_keys = h->res_vals = nullptr;
    h->res_cap = 0;
    h->spill_dir.push_back(run);
    h->spilled_bytes += run.n_items * 16;
    return KC_OK;
}

kc_status finish_spill(kc_handle h) {
    KC_CUDA(cudaStreamSynchronize(h->copy_stream));
    uint64_t total = 0;
    for (const auto& r : h->spill_dir) total += r.n_items;
    h->n_result = total;
    h->host_ctr.survivors = total;
    h->spilled = true;
    return KC_OK;
}

// Spill groups of partitions [g * per, (g + 1) * per) that the handle owns.
std::vector<uint32_t> owned_groups(kc_handle h, uint32_t G, uint32_t per, uint32_t g_lo, uint32_t g_hi) {
    std::vector<uint32_t> out;
    for (uint32_t g = g_lo; g < g_hi; ++g)
        if ((g + 1) * per > h->own_plo && g * per < h->own_phi) out.push_back(g);
    return out;
}

kc_status finalize_spilled(kc_batch_ctx* b, kc_handle h) {
    const uint32_t P = 1u << h->part_bits;
    const uint32_t G = std::min(P, kSpillGroups), per = P / G;
    release_spill(h);
    const std::vector<uint32_t> groups = owned_groups(h, G, per, 0, G);
    for (size_t i = 0; i < groups.size(); ++i) {
        const uint32_t g = groups[i];
        kc_status s = spill_group(b, h, g * per, (g + 1) * per, i + 1 == groups.size());
        if (s != KC_OK) return s;
    }
    return finish_spill(h);
}

// Out-of-core finalize of a handle with batches kept as reads (their hashes
// would have passed the device budget).  The hash space is cut into S scan
// ranges, S a power of two chosen so that one range's grouped hashes fit the
// room left; for each range every kept batch is extracted and grouped again
// in pieces, keeping only the range's windows, and the range's spill groups
// are finalized and spilled as by finalize_spilled.  Batches grouped at
// kc_add_reads take part in every range as they are.
kc_status finalize_grouped(kc_batch_ctx* b, kc_handle h) {
    const uint32_t P = 1u << h->part_bits;
    const uint32_t G = std::min(P, kSpillGroups), per = P / G;
    uint64_t kept_bases = 0;
    for (const auto& bt : h->batches)
        if (bt.deferred) kept_bases += bt.n_units * 64;
    // one range: its grouped hashes (8 bytes per window) plus the linear
    // hashes of the piece being grouped, about as large, plus the survivors
    // of one spill group; S = G at most
    const uint64_t room = room_bytes(h);
    uint32_t S = 1;
    while (S < G && 3 * (8 * kept_bases / S) > room) S <<= 1;
    h->scan_groups = S;
    const uint64_t piece_units = std::max<uint64_t>(1ull << 16, (kept_bases / 64) / S + 1);
    release_spill(h);
    std::vector<Batch> kept = h->batches;
    std::vector<uint32_t> all_groups = owned_groups(h, G, per, 0, G);
    const uint32_t last_group = all_groups.empty() ? 0 : all_groups.back();
    cudaStream_t st = h->stream;
    kc_status s = KC_OK;
    for (uint32_t r = 0; r < S && s == KC_OK; ++r) {
        const std::vector<uint32_t> groups = owned_groups(h, G, per, r * (G / S), (r + 1) * (G / S));
        if (groups.empty()) continue;
        // hash range of scan range r, within the handle's own range
        const int pb = h->part_bits;
        const uint64_t p0 = (uint64_t)r * (P / S), p1 = (uint64_t)(r + 1) * (P / S);
        kc::PassParams base = h->params(0);
        base.h_lo = std::max<uint64_t>(h->own_h_lo, p0 << (64 - pb));
        base.h_hi = std::min<uint64_t>(h->own_h_hi, (p1 << (64 - pb)) - 1ull);  // p1 = P wraps to 0: ~0
        std::vector<Batch> pieces;
        cudaEvent_t t0 = phase_begin(h);
        for (const Batch& bt : kept) {
            if (!bt.deferred) {
                pieces.push_back(bt);
                continue;
            }
            for (uint64_t u0 = 0; u0 < bt.n_units && s == KC_OK; u0 += piece_units) {
                Batch pc;
                pc.sample = bt.sample;
                pc.pw = bt.pw + 2 * u0;  // the word after the piece is the next unit's first word (or padding)
                pc.vw = bt.vw + u0;
                pc.n_units = std::min(piece_units, bt.n_units - u0);
                kc::PassParams p = base;
                p.sample = bt.sample;
                s = bucket_batch(h, pc, pc.n_units * 64, st, p, Grouping::Exact);
                h->launches += 5;
                pc.pw = pc.vw = nullptr;  // the piece borrows the kept reads
                pc.deferred = true;       // marks hashes to free after the range
                if (s == KC_OK) pieces.push_back(pc);
            }
        }
        phase_end(h, kPass1, t0);
        if (s == KC_OK) {
            h->batches = pieces;
            for (uint32_t g : groups) {
                s = spill_group(b, h, g * per, (g + 1) * per, g == last_group);
                if (s != KC_OK) break;
            }
        }
        if (s != KC_OK) cudaStreamSynchronize(b->st);  // a failed group may have left fallback kernels that read the pieces
        for (Batch& pc : pieces)
            if (pc.deferred) {
                leave_hashes(h, pc);
            }
        h->batches = kept;
    }
    if (s != KC_OK) return s;
    return finish_spill(h);
}

// The batches kc_add_reads kept for the batched ingest, of every handle of
// the batch: extracted and grouped on the batch's stream, which waits for each
// handle's stream first; each handle's stream then waits for the grouping.
kc_status ingest_batches(kc_batch_ctx* b, kc_handle* hs, int n) {
    bool any = false;
    for (int j = 0; j < n; ++j) {
        kc_handle h = hs[j];
        if (!h || h->state != State::Open || h->strategy != KC_STRATEGY_PARTITIONED) continue;
        for (const Batch& bt : h->batches) any |= bt.pending;
    }
    if (!any) return KC_OK;
    std::vector<kc_handle> open;
    for (int j = 0; j < n; ++j) {
        kc_handle h = hs[j];
        if (!h || h->state != State::Open || h->strategy != KC_STRATEGY_PARTITIONED) continue;
        for (kc_handle o : open)
            if (o == h) return fail(KC_ERR_ARG, "handle listed twice");
        open.push_back(h);
        KC_CUDA(cudaEventRecord(h->ev_main, h->stream));
        KC_CUDA(cudaStreamWaitEvent(b->st, h->ev_main, 0));
    }
    std::vector<LeftBlock> left;
    kc_status s = ingest_pending(open.data(), (int)open.size(), b->st, b->sm_count, &left);
    for (kc_handle h : open) {
        KC_CUDA(cudaEventRecord(h->ev_main, b->st));
        KC_CUDA(cudaStreamWaitEvent(h->stream, h->ev_main, 0));
    }
    for (const LeftBlock& x : left) leave_block(x.h, x.p, x.bytes, x.h->stream);
    return s;
}

// A finalize of the handle has failed and it stays open: what its consumer and
// fallbacks have added to the handle's counts is taken back, since the next
// finalize counts every partition again.
static void uncount(kc_batch_ctx* b, kc_handle h) {
    h->fallback_partitions = 0;
    cudaMemsetAsync(&h->ctr->candidates, 0, 2 * sizeof(unsigned long long), b->st);  // and claimed
    cudaMemsetAsync(&h->ctr->split_parts, 0, sizeof(unsigned), b->st);
    cudaStreamSynchronize(b->st);
}

static kc_status finalize_jobs(kc_batch_ctx* b, kc_handle* hs, int n) {
    if (b && hs && n > 0) {
        kc_status s = ingest_batches(b, hs, n);
        if (s != KC_OK) return s;
    }
    if (n == 1 && hs && hs[0] && hs[0]->strategy == KC_STRATEGY_PARTITIONED && hs[0]->state == State::Open) {
        kc_handle h = hs[0];
        if (h->deferred) return finalize_grouped(b, h);
        if (h->cfg.spill) return finalize_spilled(b, h);
        // survivors and sorted result, 16 bytes each per key, at most one
        // key per min_count windows (and per base): spill when they would
        // not fit
        const uint64_t need = 32 * (h->bases / std::max<uint32_t>(1, h->min_count));
        if (!fits_device(h, need)) return finalize_spilled(b, h);
        kc_status s = finalize_core(b, hs, n, 0, 0xffffffffu, true);
        if (s != KC_ERR_OOM_DEVICE || !small_need(h, need)) return s;
        uncount(b, h);
        return finalize_spilled(b, h);  // no room after all: counted again, group by group
    }
    if (!hs || n <= 1) return finalize_core(b, hs, n, 0, 0xffffffffu, true);
    // handles whose reads passed the device budget are finalized alone, in
    // hash ranges; the others together
    std::vector<kc_handle> rest;
    for (int j = 0; j < n; ++j) {
        if (hs[j] && hs[j]->deferred && hs[j]->strategy == KC_STRATEGY_PARTITIONED && hs[j]->state == State::Open) {
            kc_status s = finalize_grouped(b, hs[j]);
            if (s != KC_OK) return s;
        } else {
            rest.push_back(hs[j]);
        }
    }
    return finalize_core(b, rest.data(), (int)rest.size(), 0, 0xffffffffu, true);
}

kc_status kc_batch_finalize_internal(kc_batch_ctx* b, kc_handle* hs, int n) {
    const kc_status s = finalize_jobs(b, hs, n);
    if (s != KC_OK && b && hs)
        for (int j = 0; j < n; ++j)
            if (hs[j] && hs[j]->state == State::Open && hs[j]->strategy == KC_STRATEGY_PARTITIONED) uncount(b, hs[j]);
    return s;
}

extern "C" {

kc_status kc_batch_create(void* stream, kc_batch* out) {
    if (!out) return fail(KC_ERR_ARG, "out is null");
    kc_batch_ctx* b = nullptr;
    kc_status s = kc_batch_create_internal((cudaStream_t)stream, &b);
    *out = b;
    return s;
}

kc_status kc_batch_finalize(kc_batch b, kc_handle* handles, int n) { return kc_batch_finalize_internal(b, handles, n); }

kc_status kc_batch_ingest(kc_batch b, kc_handle* handles, int n) {
    if (!b || (!handles && n > 0) || n < 0) return fail(KC_ERR_ARG, "null batch or handle list");
    for (int j = 0; j < n; ++j) {
        if (!handles[j]) return fail(KC_ERR_ARG, "null handle in batch");
        for (int i = 0; i < j; ++i)
            if (handles[i] == handles[j]) return fail(KC_ERR_ARG, "handle listed twice");
    }
    return ingest_batches(b, handles, n);
}

void kc_batch_destroy(kc_batch b) { kc_batch_destroy_internal(b); }

}  // extern "C"
