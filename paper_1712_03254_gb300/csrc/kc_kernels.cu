// Kernels of the k-mer counting path and their launchers (sm_103a).
//
// Ingest      read-start bits from the offsets, then one "valid window start"
//             bit per base (no unknown base inside, window inside one read).
// Pass 1      per valid window: canonical key, mixer hash, one 64-bit atomicOr
//             on the key's filter word; the returned old word tells whether all
//             of the key's bits were set before (Section III, Prune: "seen
//             before"), and such candidates are claimed in the table.
// Pass 2      exact recount: every valid window probes the table and counts its
//             key if the key is there (Section II-B, Count unit re-reading the
//             input).
// Compaction  keys whose summed count reaches min_count (this removes the
//             filter's false positives, Section III, Unify).
// Sort        bucket by key, then sort each bucket: a warp ranks up to 64 keys
//             by key range, larger ones take bitonic networks; ascending keys.

#include <algorithm>
#include <atomic>

#include "kc_internal.h"

namespace kc {

namespace {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ uint64_t cover_pair_hi(uint64_t hi, uint64_t lo, int len) {
    // Position p (MSB first over the 128-bit pair) of the result is the OR of
    // positions p .. p+len-1 of the input; only the first 64 positions are kept.
    int c = 1;
    while (2 * c <= len) {
        const uint64_t nh = hi | (hi << c) | (lo >> (64 - c));
        const uint64_t nl = lo | (lo << c);
        hi = nh;
        lo = nl;
        c *= 2;
    }
    if (len > c) {
        const int s = len - c;
        hi = hi | (hi << s) | (lo >> (64 - s));
    }
    return hi;
}

__global__ void k_mark_read_starts(const uint64_t* __restrict__ offsets, uint64_t n_reads, uint64_t base,
                                   uint64_t n_local, unsigned long long* __restrict__ bd,
                                   DevCounters* __restrict__ ctr) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t r = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; r <= n_reads; r += stride) {
        const uint64_t o = offsets[r];
        if (r < n_reads && offsets[r + 1] < o) atomicOr(&ctr->err, DERR_OFFSETS);
        if (o < base) {
            atomicOr(&ctr->err, DERR_OFFSETS);
            continue;
        }
        const uint64_t i = o - base;
        if (i < n_local) atomicOr(bd + (i >> 6), 0x8000000000000000ull >> (i & 63));
    }
}

// Words [w_begin, w_end) of the batch's n_vwords valid-window words.  A window at
// j is broken by an unknown base at j .. j + k - 1 or a read start at j + 1 ..
// j + k - 1: one OR over k - 1 positions of the unknown bases and of the starts
// moved up by one, and the unknown base at j + k - 1.  (Three ORs, one for the
// starts across the word's end alone, made about 200 instructions a word: 1.4 M
// words 25 us, now 15.)
__global__ void k_build_valid(const uint64_t* __restrict__ nmask, const uint64_t* __restrict__ bd,
                              uint64_t n_vwords, uint64_t w_begin, uint64_t w_end, uint64_t start_local,
                              uint64_t n_local, int k, uint64_t* __restrict__ vout, DevCounters* __restrict__ ctr) {
    unsigned long long local = 0;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t w = w_begin + (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; w < w_end; w += stride) {
        const uint64_t n_hi = nmask[w], n_lo = w + 1 < n_vwords ? nmask[w + 1] : 0ull;
        uint64_t bad = n_hi;
        if (k >= 2) {
            const uint64_t b_hi = bd[w], b_lo = w + 1 < n_vwords ? bd[w + 1] : 0ull;
            // (position 127 of the pair, whose start lies in the next word, is not reached: k <= 31)
            bad = cover_pair_hi(n_hi | (b_hi << 1) | (b_lo >> 63), n_lo | (b_lo << 1), k - 1);
            bad |= (n_hi << (k - 1)) | (n_lo >> (65 - k));
        }
        uint64_t valid = ~bad;
        const uint64_t p0 = w * 64;
        // windows must start at or after the first read's first base
        if (p0 + 64 <= start_local) valid = 0;
        else if (p0 < start_local) valid &= ~0ull >> (start_local - p0);
        // and end at or before the last read's last base
        if (n_local < (uint64_t)k || p0 > n_local - k) {
            valid = 0;
        } else {
            const uint64_t last = n_local - k - p0;  // last valid offset in this word
            if (last < 63) valid &= ~(~0ull >> (last + 1));
        }
        vout[w] = valid;
        local += __popcll(valid);
    }
    local = warp_sum(local);
    if ((threadIdx.x & 31) == 0 && local) atomicAdd(&ctr->windows, local);
}

__global__ void __launch_bounds__(256) k_pass1(const uint64_t* __restrict__ pw, const uint64_t* __restrict__ vw,
                                               uint64_t n_units, PassParams p,
                                               unsigned long long* __restrict__ bloom, Slot* __restrict__ table,
                                               DevCounters* __restrict__ ctr) {
    const int lane = threadIdx.x & 31;
    const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long cand = 0, claimed = 0;
    for (uint64_t base = warp * 32; base < n_units; base += n_warps * 32) {
        const UnitWords uw = load_unit(pw, vw, base + lane, n_units, lane);
        uint64_t vm = uw.v;
        // Warp-uniform trip count with a reconvergence point per window, so
        // the lanes stay together instead of splitting into sub-warps at the
        // candidate branch.
        const int n_iter = __reduce_max_sync(kFull, (unsigned)__popcll(vm));
        for (int it = 0; it < n_iter; ++it) {
            if (vm) {
                const int j = __clzll(vm);
                vm &= ~(0x8000000000000000ull >> j);
                const uint64_t key = canonical_key(window_code(uw.w0, uw.w1, uw.w2, j, p.rc_shift), p);
                const uint64_t h = mixer64(key);
                const uint64_t pat = bloom_pattern(mixer64(h), p.n_hashes);
                const unsigned long long old = atomicOr(bloom + (h >> p.bloom_shift), (unsigned long long)pat);
                if (p.all_candidates || (old & pat) == pat) {
                    ++cand;
                    claimed += table_claim(table, p.table_mask, h >> p.table_shift, key + 1, ctr);
                }
            }
            __syncwarp();
        }
    }
    cand = warp_sum(cand);
    claimed = warp_sum(claimed);
    if (lane == 0) {
        if (cand) atomicAdd(&ctr->candidates, cand);
        if (claimed) atomicAdd(&ctr->claimed, claimed);
    }
}

__global__ void __launch_bounds__(256) k_pass2(const uint64_t* __restrict__ pw, const uint64_t* __restrict__ vw,
                                               uint64_t n_units, PassParams p, Slot* __restrict__ table,
                                               DevCounters* __restrict__ ctr) {
    const int lane = threadIdx.x & 31;
    const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    for (uint64_t base = warp * 32; base < n_units; base += n_warps * 32) {
        const UnitWords uw = load_unit(pw, vw, base + lane, n_units, lane);
        uint64_t vm = uw.v;
        const int n_iter = __reduce_max_sync(kFull, (unsigned)__popcll(vm));
        for (int it = 0; it < n_iter; ++it) {
            if (vm) {
                const int j = __clzll(vm);
                vm &= ~(0x8000000000000000ull >> j);
                const uint64_t key = canonical_key(window_code(uw.w0, uw.w1, uw.w2, j, p.rc_shift), p);
                const uint64_t h = mixer64(key);
                table_count(table, p.table_mask, h >> p.table_shift, key + 1, p.sample, ctr);
            }
            __syncwarp();
        }
    }
}

__global__ void k_clear_counts(Slot* __restrict__ table, uint64_t n_slots) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_slots; i += stride)
        table[i].cnt[0] = table[i].cnt[1] = 0u;
}

// Survivors of the table.  A warp queues the kept slots of its rows in shared
// memory and writes 32 at a time behind one claim of the output: a claim a row
// of 32 slots was one atomic on one address for each of 2.6e5 rows (2^23 slots,
// 1.05 M kept: 179 us, now 40).
__global__ void __launch_bounds__(256) k_compact(const Slot* __restrict__ table, uint64_t n_slots, int n_samples,
                                                 uint32_t min_count, uint64_t* __restrict__ keys,
                                                 uint64_t* __restrict__ vals, DevCounters* __restrict__ ctr) {
    __shared__ ulonglong2 s_q[8][64];
    const int lane = threadIdx.x & 31;
    ulonglong2* const q = s_q[threadIdx.x >> 5];
    const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    const unsigned lt = (1u << lane) - 1u;
    unsigned n = 0;  // queued
    const auto write = [&](unsigned m) {
        __syncwarp();
        n -= m;
        unsigned long long pos = 0;
        if (lane == 0) pos = atomicAdd(&ctr->survivors, (unsigned long long)m);
        pos = __shfl_sync(kFull, pos, 0) + lane;
        if ((unsigned)lane < m) {
            const ulonglong2 v = q[n + lane];
            keys[pos] = v.x - 1;
            vals[pos] = v.y;
        }
        __syncwarp();
    };
    constexpr int kRows = 4;  // rows in flight
    for (uint64_t base = warp * 32; base < n_slots; base += n_warps * 32 * kRows) {
        ulonglong2 v[kRows];
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
            const uint64_t i = base + r * n_warps * 32 + lane;
            v[r] = i < n_slots ? __ldcs(reinterpret_cast<const ulonglong2*>(table) + i) : make_ulonglong2(0, 0);
        }
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
            uint64_t sum = (uint32_t)v[r].y;
            if (n_samples == 2) sum += (uint32_t)(v[r].y >> 32);
            const bool keep = v[r].x != 0ull && sum >= min_count;
            const unsigned ballot = __ballot_sync(kFull, keep);
            if (keep) q[n + __popc(ballot & lt)] = v[r];
            n += __popc(ballot);
            if (n >= 32) write(32);
        }
    }
    if (n) write(n);
}

// Exclusive scan of n <= 4096 counters with one CTA of 1024 threads, four
// consecutive ones a thread (all loads in flight at once).
__global__ void __launch_bounds__(1024) k_scan(const uint32_t* __restrict__ hist, uint64_t n,
                                               uint64_t* __restrict__ starts, uint64_t* __restrict__ cursor) {
    __shared__ unsigned long long warp_tot[32];
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const uint64_t lo = 4ull * t;
    uint32_t c[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) c[j] = lo + j < n ? hist[lo + j] : 0u;
    const unsigned long long sum = (unsigned long long)c[0] + c[1] + c[2] + c[3];
    // inclusive warp scan
    unsigned long long x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[wid] = x;
    __syncthreads();
    if (wid == 0) {
        unsigned long long w = lane < (int)(blockDim.x >> 5) ? warp_tot[lane] : 0ull;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(kFull, w, o);
            if (lane >= o) w += y;
        }
        warp_tot[lane] = w;  // inclusive over warps
    }
    __syncthreads();
    unsigned long long run = x - sum + (wid ? warp_tot[wid - 1] : 0ull);
    if (lo + 4 <= n && !((reinterpret_cast<uintptr_t>(starts) | reinterpret_cast<uintptr_t>(cursor)) & 15u)) {
        // 16-byte stores: 4096 counters 7.5 -> 5 us
        const ulonglong2 a = make_ulonglong2(run, run + c[0]);
        const ulonglong2 b = make_ulonglong2(a.y + c[1], a.y + c[1] + c[2]);
        reinterpret_cast<ulonglong2*>(starts + lo)[0] = a;
        reinterpret_cast<ulonglong2*>(starts + lo)[1] = b;
        reinterpret_cast<ulonglong2*>(cursor + lo)[0] = a;
        reinterpret_cast<ulonglong2*>(cursor + lo)[1] = b;
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (lo + j < n) {
                starts[lo + j] = run;
                cursor[lo + j] = run;
            }
            run += c[j];
        }
    }
    if (t == (int)blockDim.x - 1) starts[n] = warp_tot[(blockDim.x >> 5) - 1];
}

// The scan of longer arrays (scan_lookback); state: a word per tile and the ticket.
__global__ void __launch_bounds__(kScanThreads) k_scan_long(const uint32_t* __restrict__ hist, uint64_t n,
                                                            uint64_t* __restrict__ starts,
                                                            uint64_t* __restrict__ cursor, unsigned long long* state,
                                                            uint64_t n_tiles) {
    scan_lookback(hist, n, starts, cursor, state, state + n_tiles);
}

__global__ void k_scatter(const uint64_t* __restrict__ keys, const uint64_t* __restrict__ vals,
                          DevCounters* __restrict__ ctr, uint64_t cap, int key_bits, int bits,
                          unsigned long long* __restrict__ cursor, uint64_t* __restrict__ out_keys,
                          uint64_t* __restrict__ out_vals) {
    const uint64_t n = ctr->survivors < cap ? ctr->survivors : cap;
    const bool even = even_buckets(key_bits, bits);
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint64_t key = keys[i];
        const uint64_t b = key_bucket(key, key_bits, bits, even);
        if (b >> bits) {
            atomicOr(&ctr->err, DERR_INTERNAL);
            continue;
        }
        const uint64_t pos = atomicAdd(cursor + b, 1ull);
        if (pos >= cap) {
            atomicOr(&ctr->err, DERR_INTERNAL);
            continue;
        }
        out_keys[pos] = key;
        out_vals[pos] = vals[i];
    }
}

constexpr int kSortCap = 2048;    // keys per shared-memory tile
constexpr int kWarpSortMax = 256; // keys one warp sorts in registers
constexpr int kSortThreads = 256;

// Ascending bitonic network in the "mirror" form: every comparator puts the
// minimum at the lower index, so indices >= n behave as +infinity and need no
// padding.
__global__ void __launch_bounds__(kSortThreads) k_bucket_sort(uint64_t* __restrict__ keys,
                                                              uint64_t* __restrict__ vals,
                                                              const uint64_t* __restrict__ starts,
                                                              DevCounters* __restrict__ ctr) {
    extern __shared__ uint64_t smem[];
    uint64_t* sk = smem;
    uint64_t* sv = smem + kSortCap;
    const uint64_t lo = starts[blockIdx.x];
    const uint64_t n64 = starts[blockIdx.x + 1] - lo;
    if (n64 <= (uint64_t)kWarpSortMax) return;  // sorted by k_bucket_sort_warp
    if (n64 > (uint64_t)kSortCap) {
        if (threadIdx.x == 0) atomicOr(&ctr->err, DERR_SORT_BUCKET);
        return;
    }
    const int n = (int)n64;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        sk[i] = keys[lo + i];
        sv[i] = vals[lo + i];
    }
    int n2 = 1;
    while (n2 < n) n2 <<= 1;
    __syncthreads();
    for (int size = 2; size <= n2; size <<= 1) {
        const int half = size >> 1;
        for (int i = threadIdx.x; i < (n2 >> 1); i += blockDim.x) {
            const int blk = i / half, off = i % half;
            const int a = blk * size + off, b = blk * size + size - 1 - off;
            if (b < n && sk[a] > sk[b]) {
                const uint64_t tk = sk[a], tv = sv[a];
                sk[a] = sk[b];
                sv[a] = sv[b];
                sk[b] = tk;
                sv[b] = tv;
            }
        }
        __syncthreads();
        for (int stride = size >> 2; stride > 0; stride >>= 1) {
            for (int i = threadIdx.x; i < (n2 >> 1); i += blockDim.x) {
                const int a = 2 * i - (i & (stride - 1)), b = a + stride;
                if (b < n && sk[a] > sk[b]) {
                    const uint64_t tk = sk[a], tv = sv[a];
                    sk[a] = sk[b];
                    sv[a] = sv[b];
                    sk[b] = tk;
                    sv[b] = tv;
                }
            }
            __syncthreads();
        }
    }
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        keys[lo + i] = sk[i];
        vals[lo + i] = sv[i];
    }
}

// Buckets of up to 64 keys ranked (warp_rank64) and stored in place; larger
// ones set DERR_SORT_BIG.  1.05 M pairs: 11 us; one kernel with the networks
// for the larger buckets, at two CTAs an SM for their registers and on plain
// key prefixes (buckets of up to twice the mean), 40.
__global__ void __launch_bounds__(256, 6) k_bucket_sort_warp(uint64_t* keys, uint64_t* vals,
                                                             const uint64_t* __restrict__ starts, uint64_t n_buckets,
                                                             int key_bits, DevCounters* __restrict__ ctr) {
    __shared__ __align__(16) WarpRankTile tiles[256 / 32];
    const int lane = threadIdx.x & 31;
    WarpRankTile& tile = tiles[threadIdx.x >> 5];
    *reinterpret_cast<uint2*>(&tile.count[2 * lane]) = make_uint2(0u, 0u);
    __syncwarp();
    const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    for (uint64_t b = warp; b < n_buckets; b += n_warps) {
        const uint64_t lo = starts[b];
        const uint64_t n = starts[b + 1] - lo;
        if (n <= 1) continue;
        if (n > 64) {
            if (lane == 0 && !(*(volatile unsigned*)&ctr->err & DERR_SORT_BIG)) atomicOr(&ctr->err, DERR_SORT_BIG);
            continue;
        }
        const bool in0 = lane < (int)n, in1 = 32 + lane < (int)n;
        const uint64_t k0 = in0 ? keys[lo + lane] : 0ull, v0 = in0 ? vals[lo + lane] : 0ull;
        const uint64_t k1 = in1 ? keys[lo + 32 + lane] : 0ull, v1 = in1 ? vals[lo + 32 + lane] : 0ull;
        uint32_t r0 = 0, r1 = 0;
        // every pair is read before the first is stored: the ranks wait for all keys, and __syncwarp orders the values
        warp_rank64(tile, k0, k1, in0, in1, n > 32, key_bits, lane, r0, r1);
        __syncwarp();
        if (in0) {
            keys[lo + r0] = k0;
            vals[lo + r0] = v0;
        }
        if (in1) {
            keys[lo + r1] = k1;
            vals[lo + r1] = v1;
        }
    }
}

// The buckets of 65..256 keys by a network in one warp's registers; larger
// ones set DERR_SORT_MEDIUM.
__global__ void __launch_bounds__(256, 2) k_bucket_sort_warp_big(uint64_t* __restrict__ keys,
                                                                 uint64_t* __restrict__ vals,
                                                                 const uint64_t* __restrict__ starts,
                                                                 uint64_t n_buckets, DevCounters* __restrict__ ctr) {
    if (!(*(volatile unsigned*)&ctr->err & DERR_SORT_BIG)) return;
    const int lane = threadIdx.x & 31;
    const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    // a lane looks at a bucket, the warp sorts the ones it has to
    for (uint64_t base = warp * 32; base < n_buckets; base += n_warps * 32) {
        const uint64_t b = base + (uint64_t)lane;
        const uint64_t lo_b = b < n_buckets ? starts[b] : 0ull;
        const uint64_t n_b = b < n_buckets ? starts[b + 1] - lo_b : 0ull;
        unsigned todo = __ballot_sync(0xffffffffu, n_b > 64);
        while (todo) {
            const int src = __ffs(todo) - 1;
            todo &= todo - 1;
            const uint64_t lo = __shfl_sync(0xffffffffu, lo_b, src), n = __shfl_sync(0xffffffffu, n_b, src);
            if (n > (uint64_t)kWarpSortMax) {
                if (lane == 0) atomicOr(&ctr->err, DERR_SORT_MEDIUM);
            } else if (n <= 128) {
                warp_sort_bucket<4>(keys, vals, lo, (int)n, lane);
            } else {
                warp_sort_bucket<8>(keys, vals, lo, (int)n, lane);
            }
        }
    }
}

// One comparator stage of the same network over global memory, for every bucket
// of the list that still has stages of this size (a row of the grid each).
__global__ void __launch_bounds__(256) k_bitonic_step(const SortRange* __restrict__ ranges, uint64_t n_ranges,
                                                      uint64_t size, uint64_t stride, int mirror) {
    const uint64_t gstride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t r = blockIdx.y; r < n_ranges; r += gridDim.y) {
        const uint64_t n = ranges[r].n;
        uint64_t* const keys = ranges[r].keys;
        uint64_t* const vals = ranges[r].vals;
        if (size >= 2 * n) continue;  // the bucket's network, of the next power of two, ends before
        const uint64_t pairs = (n + size - 1) / size * (size >> 1);  // blocks of `size` that hold a key
        for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < pairs; i += gstride) {
            uint64_t a, b;
            if (mirror) {
                const uint64_t half = size >> 1, blk = i / half, off = i % half;
                a = blk * size + off;
                b = blk * size + size - 1 - off;
            } else {
                a = 2 * i - (i & (stride - 1));
                b = a + stride;
            }
            if (b < n && keys[a] > keys[b]) {
                const uint64_t tk = keys[a], tv = vals[a];
                keys[a] = keys[b];
                vals[a] = vals[b];
                keys[b] = tk;
                vals[b] = tv;
            }
        }
    }
}

__global__ void k_counts_narrow(const uint64_t* __restrict__ vals, uint64_t n, uint32_t* __restrict__ out) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) out[i] = (uint32_t)vals[i];
}

// The result table into device arrays: keys as they are, the packed counts as
// S 32-bit counts a key, in one pass (a copy of the keys and k_counts_narrow
// read and wrote the same bytes one after the other).  Four keys a thread, 16
// bytes at a time, where the caller's arrays are aligned for it.  Bound by the
// memory: 6.8 M keys 27 us, 12.3 M of two samples 67 us (5.9 TB/s); a dump call
// of 5.3 M keys 72 -> 58 us.
template <int S>
__global__ void __launch_bounds__(256) k_dump(const uint64_t* __restrict__ keys, const uint64_t* __restrict__ vals,
                                              uint64_t n, uint64_t* __restrict__ out_keys,
                                              uint32_t* __restrict__ out_counts) {
    const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    uint64_t done = 0;
    if (!((reinterpret_cast<uintptr_t>(out_keys) | reinterpret_cast<uintptr_t>(out_counts)) & 15u)) {
        const ulonglong2 *k2 = reinterpret_cast<const ulonglong2*>(keys), *v2 = reinterpret_cast<const ulonglong2*>(vals);
        ulonglong2* ok = reinterpret_cast<ulonglong2*>(out_keys);
        const uint64_t quads = n >> 2;
        for (uint64_t q = t; q < quads; q += stride) {
            const ulonglong2 a = k2[2 * q], b = k2[2 * q + 1], x = v2[2 * q], y = v2[2 * q + 1];
            ok[2 * q] = a;
            ok[2 * q + 1] = b;
            if (S == 1) {
                reinterpret_cast<uint4*>(out_counts)[q] =
                    make_uint4((uint32_t)x.x, (uint32_t)x.y, (uint32_t)y.x, (uint32_t)y.y);
            } else {
                reinterpret_cast<ulonglong2*>(out_counts)[2 * q] = x;
                reinterpret_cast<ulonglong2*>(out_counts)[2 * q + 1] = y;
            }
        }
        done = quads << 2;
    }
    for (uint64_t i = done + t; i < n; i += stride) {
        const uint64_t v = vals[i];
        out_keys[i] = keys[i];
        out_counts[S * i] = (uint32_t)v;
        if (S == 2) out_counts[S * i + 1] = (uint32_t)(v >> 32);
    }
}

unsigned grid_for(uint64_t work, int block, int max_ctas) {
    uint64_t g = (work + block - 1) / block;
    if (g < 1) g = 1;
    if (g > (uint64_t)max_ctas) g = (uint64_t)max_ctas;
    return (unsigned)g;
}

}  // namespace

void launch_mark_read_starts(const uint64_t* offsets, uint64_t n_reads, uint64_t base, uint64_t n_local,
                             uint64_t* bd, DevCounters* ctr, cudaStream_t st) {
    k_mark_read_starts<<<grid_for(n_reads + 1, 256, 4096), 256, 0, st>>>(
        offsets, n_reads, base, n_local, reinterpret_cast<unsigned long long*>(bd), ctr);
}

void launch_build_valid(const uint64_t* nmask, const uint64_t* bd, uint64_t n_vwords, uint64_t start_local,
                        uint64_t n_local, int k, uint64_t* vout, DevCounters* ctr, const Grid& g, cudaStream_t st) {
    launch_build_valid_range(nmask, bd, n_vwords, 0, n_vwords, start_local, n_local, k, vout, ctr, g, st);
}

void launch_build_valid_range(const uint64_t* nmask, const uint64_t* bd, uint64_t n_vwords, uint64_t w_begin,
                              uint64_t w_end, uint64_t start_local, uint64_t n_local, int k, uint64_t* vout,
                              DevCounters* ctr, const Grid& g, cudaStream_t st) {
    k_build_valid<<<grid_for(w_end - w_begin, 256, g.sm_count * 8), 256, 0, st>>>(nmask, bd, n_vwords, w_begin, w_end,
                                                                                   start_local, n_local, k, vout, ctr);
}

void launch_pass1(const uint64_t* pw, const uint64_t* vw, uint64_t n_units, const PassParams& p, uint64_t* bloom,
                  Slot* table, DevCounters* ctr, const Grid& g, cudaStream_t st) {
    k_pass1<<<grid_for(n_units, 256, g.ctas()), 256, 0, st>>>(
        pw, vw, n_units, p, reinterpret_cast<unsigned long long*>(bloom), table, ctr);
}

void launch_pass2(const uint64_t* pw, const uint64_t* vw, uint64_t n_units, const PassParams& p, Slot* table,
                  DevCounters* ctr, const Grid& g, cudaStream_t st) {
    k_pass2<<<grid_for(n_units, 256, g.ctas()), 256, 0, st>>>(pw, vw, n_units, p, table, ctr);
}

void launch_clear_counts(Slot* table, uint64_t n_slots, const Grid& g, cudaStream_t st) {
    k_clear_counts<<<grid_for(n_slots, 256, g.sm_count * 8), 256, 0, st>>>(table, n_slots);
}

void launch_compact(const Slot* table, uint64_t n_slots, int n_samples, uint32_t min_count, uint64_t* keys,
                    uint64_t* vals, DevCounters* ctr, const Grid& g, cudaStream_t st) {
    k_compact<<<grid_for(n_slots, 256, g.sm_count * 8), 256, 0, st>>>(table, n_slots, n_samples, min_count, keys,
                                                                       vals, ctr);
}

cudaError_t launch_scan(const uint32_t* hist, uint64_t n, uint64_t* starts, uint64_t* cursor, cudaStream_t st) {
    if (n <= 4096) {
        k_scan<<<1, 1024, 0, st>>>(hist, n, starts, cursor);
        return cudaSuccess;
    }
    const uint64_t n_tiles = (n + kScanTile - 1) / kScanTile;
    unsigned long long* state = nullptr;
    cudaError_t e = dev_alloc(&state, (n_tiles + 1) * 8, st);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(state, 0, (n_tiles + 1) * 8, st);
    if (e == cudaSuccess) k_scan_long<<<(unsigned)n_tiles, kScanThreads, 0, st>>>(hist, n, starts, cursor, state, n_tiles);
    const cudaError_t f = cudaFreeAsync(state, st);
    return e != cudaSuccess ? e : f;
}

void launch_scatter(const uint64_t* keys, const uint64_t* vals, DevCounters* ctr, uint64_t cap, int key_bits,
                    int bits, uint64_t* cursor, uint64_t* out_keys, uint64_t* out_vals, const Grid& g,
                    cudaStream_t st) {
    k_scatter<<<g.sm_count * 8, 256, 0, st>>>(keys, vals, ctr, cap, key_bits, bits,
                                               reinterpret_cast<unsigned long long*>(cursor), out_keys, out_vals);
}

int bucket_sort_capacity() { return kSortCap; }

void launch_bucket_sort_warp(uint64_t* keys, uint64_t* vals, const uint64_t* starts, uint64_t n_buckets, int key_bits,
                             DevCounters* ctr, const Grid& g, cudaStream_t st) {
    const uint64_t warps = n_buckets;
    unsigned grid = (unsigned)((warps + 7) / 8);
    const unsigned cap = (unsigned)g.sm_count * 6;  // one wave
    if (grid > cap) grid = cap;
    if (grid < 1) grid = 1;
    k_bucket_sort_warp<<<grid, 256, 0, st>>>(keys, vals, starts, n_buckets, key_bits, ctr);
    grid = (unsigned)std::min<uint64_t>((n_buckets + 255) / 256, (uint64_t)g.sm_count * 2);
    k_bucket_sort_warp_big<<<grid, 256, 0, st>>>(keys, vals, starts, n_buckets, ctr);
}

int warp_sort_capacity() { return kWarpSortMax; }

void launch_bucket_sort(uint64_t* keys, uint64_t* vals, const uint64_t* starts, uint64_t n_buckets,
                        DevCounters* ctr, cudaStream_t st) {
    const size_t smem = 2 * sizeof(uint64_t) * kSortCap;
    static bool attr_set = false;
    if (!attr_set) {
        allow_max_dynamic_smem(k_bucket_sort);
        attr_set = true;
    }
    k_bucket_sort<<<(unsigned)n_buckets, kSortThreads, smem, st>>>(keys, vals, starts, ctr);
}

uint64_t launch_bitonic_global(const SortRange* ranges, uint64_t n_ranges, uint64_t largest, cudaStream_t st) {
    uint64_t n2 = 1, launches = 0;
    while (n2 < largest) n2 <<= 1;
    const unsigned rows = (unsigned)std::min<uint64_t>(n_ranges, 4096);
    const dim3 grid(grid_for(n2 >> 1, 256, std::max(1, 152 * 16 / (int)rows)), rows);
    for (uint64_t size = 2; size <= n2; size <<= 1) {
        k_bitonic_step<<<grid, 256, 0, st>>>(ranges, n_ranges, size, 0, 1);
        ++launches;
        for (uint64_t stride = size >> 2; stride > 0; stride >>= 1, ++launches)
            k_bitonic_step<<<grid, 256, 0, st>>>(ranges, n_ranges, size, stride, 0);
    }
    return launches;
}

void launch_dump(const uint64_t* keys, const uint64_t* vals, uint64_t n, int n_samples, uint64_t* out_keys,
                 uint32_t* out_counts, const Grid& g, cudaStream_t st) {
    const unsigned grid = grid_for((n + 3) / 4, 256, g.sm_count * 8);
    if (n_samples == 2) k_dump<2><<<grid, 256, 0, st>>>(keys, vals, n, out_keys, out_counts);
    else k_dump<1><<<grid, 256, 0, st>>>(keys, vals, n, out_keys, out_counts);
}

void launch_counts_narrow(const uint64_t* vals, uint64_t n, uint32_t* out, cudaStream_t st) {
    if (n == 0) return;
    k_counts_narrow<<<grid_for(n, 256, 152 * 8), 256, 0, st>>>(vals, n, out);
}

int max_optin_smem() {
    static std::atomic<int> cache[64];  // per device; 0 = not queried yet
    int dev = 0;
    cudaGetDevice(&dev);
    int v = dev >= 0 && dev < 64 ? cache[dev].load(std::memory_order_relaxed) : 0;
    if (!v) {
        cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        if (dev >= 0 && dev < 64) cache[dev].store(v, std::memory_order_relaxed);
    }
    return v;
}

}  // namespace kc
