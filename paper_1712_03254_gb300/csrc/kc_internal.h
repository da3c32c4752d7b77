// Host-side declarations shared by the C-ABI layer and the kernel launchers.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>
#include <string>

#include "kc_device.cuh"

namespace kc {

// Message returned by kc_last_error() on this thread.
void set_last_error(const std::string& msg);

// Held while a stream is being captured into a graph and around every CUDA
// call that may synchronise the device or the legacy stream (cudaMalloc,
// cudaFree, cudaMallocHost, cudaFreeHost, cudaMemcpy), so that none of them
// lands inside another host thread's capture.
std::mutex& sync_api_mutex();

// Every device allocation of the library: stream-ordered from the pool, and
// fixed (cudaMalloc, with sync_api_mutex() held).  One that finds no memory has
// all handles give back their idle blocks and is tried once more.  A failure
// leaves no error behind for a later cudaGetLastError to find.  (Not with
// sync_api_mutex() held, and never during a capture: dev_alloc.)
cudaError_t dev_alloc_bytes(void** p, size_t bytes, cudaStream_t st);
cudaError_t dev_alloc_fixed_bytes(void** p, size_t bytes);
template <class T>
cudaError_t dev_alloc(T** p, size_t bytes, cudaStream_t st) {
    return dev_alloc_bytes(reinterpret_cast<void**>(p), bytes, st);
}
template <class T>
cudaError_t dev_alloc_fixed(T** p, size_t bytes) {
    return dev_alloc_fixed_bytes(reinterpret_cast<void**>(p), bytes);
}

struct Grid {
    int sm_count = 152;
    int block = 256;
    int ctas_per_sm = 8;
    int ctas() const { return sm_count * ctas_per_sm; }
};

// Ingest: read-start bits from offsets, then valid-window-start bits.
void launch_mark_read_starts(const uint64_t* offsets, uint64_t n_reads, uint64_t base, uint64_t n_local,
                             uint64_t* bd, DevCounters* ctr, cudaStream_t st);
void launch_build_valid(const uint64_t* nmask, const uint64_t* bd, uint64_t n_vwords, uint64_t start_local,
                        uint64_t n_local, int k, uint64_t* vout, DevCounters* ctr, const Grid& g, cudaStream_t st);
// The same for words [w_begin, w_end) only (a chunk whose N-mask words up to
// w_end, inclusive when w_end < n_vwords, are on the device).
void launch_build_valid_range(const uint64_t* nmask, const uint64_t* bd, uint64_t n_vwords, uint64_t w_begin,
                              uint64_t w_end, uint64_t start_local, uint64_t n_local, int k, uint64_t* vout,
                              DevCounters* ctr, const Grid& g, cudaStream_t st);

// Pass 1: filter update, candidates claimed in the table.
void launch_pass1(const uint64_t* pw, const uint64_t* vw, uint64_t n_units, const PassParams& p, uint64_t* bloom,
                  Slot* table, DevCounters* ctr, const Grid& g, cudaStream_t st);
// Pass 2: exact recount of the keys held in the table.
void launch_pass2(const uint64_t* pw, const uint64_t* vw, uint64_t n_units, const PassParams& p, Slot* table,
                  DevCounters* ctr, const Grid& g, cudaStream_t st);

// The table's counts set back to zero, its keys kept.
void launch_clear_counts(Slot* table, uint64_t n_slots, const Grid& g, cudaStream_t st);

// Compaction of slots with summed count >= min_count.
void launch_compact(const Slot* table, uint64_t n_slots, int n_samples, uint32_t min_count, uint64_t* keys,
                    uint64_t* vals, DevCounters* ctr, const Grid& g, cudaStream_t st);
// starts[0..n] = exclusive scan of hist[0..n); cursor[0..n) = starts[0..n).
// Above 4096 counters one launch with look-back (scan_lookback) and a small
// stream-ordered temporary.
cudaError_t launch_scan(const uint32_t* hist, uint64_t n, uint64_t* starts, uint64_t* cursor, cudaStream_t st);
// Scatter survivors (at most cap of them) into their buckets; keys whose
// bucket or position would fall outside the arrays set DERR_INTERNAL.
void launch_scatter(const uint64_t* keys, const uint64_t* vals, DevCounters* ctr, uint64_t cap, int key_bits,
                    int bits, uint64_t* cursor, uint64_t* out_keys, uint64_t* out_vals, const Grid& g,
                    cudaStream_t st);
// Sort every bucket of at most warp_sort_capacity() keys in place, one warp
// per bucket (two launches: up to 64 keys, and the larger ones if there are any,
// told by DERR_SORT_BIG); larger buckets set DERR_SORT_MEDIUM and are left alone.
void launch_bucket_sort_warp(uint64_t* keys, uint64_t* vals, const uint64_t* starts, uint64_t n_buckets, int key_bits,
                             DevCounters* ctr, const Grid& g, cudaStream_t st);
int warp_sort_capacity();
// Sort buckets of warp_sort_capacity()+1 .. bucket_sort_capacity() keys in
// shared memory, one CTA per bucket; larger buckets set DERR_SORT_BUCKET and
// are left for launch_bitonic_global.
void launch_bucket_sort(uint64_t* keys, uint64_t* vals, const uint64_t* starts, uint64_t n_buckets,
                        DevCounters* ctr, cudaStream_t st);
int bucket_sort_capacity();
struct SortRange {
    uint64_t* keys;
    uint64_t* vals;
    uint64_t n;
};
// Sort ranges of about the same size (the largest has `largest` pairs) in global
// memory, all of them with the same launches; returns how many.
uint64_t launch_bitonic_global(const SortRange* ranges, uint64_t n_ranges, uint64_t largest, cudaStream_t st);

void launch_counts_narrow(const uint64_t* vals, uint64_t n, uint32_t* out, cudaStream_t st);
// The result's keys and counts into device arrays (result arrays 16-byte aligned).
void launch_dump(const uint64_t* keys, const uint64_t* vals, uint64_t n, int n_samples, uint64_t* out_keys,
                 uint32_t* out_counts, const Grid& g, cudaStream_t st);

// ---- partitioned strategy (kc_partition.cu) --------------------------------

struct FallbackArgs {
    const uint64_t* const* data;
    const uint64_t* const* starts;
    const int* samples;
    uint32_t part;
    uint64_t h_lo;  // hashes of the partition below h_lo are already counted
    int part_bits;
    int bloom_shift;
    int n_hashes;
    int n_samples;
    int all_candidates;
    uint32_t min_count;
    unsigned long long* bloom;
    Slot* table;
    uint64_t table_mask;
    uint64_t* out_keys;
    uint64_t* out_vals;
    uint64_t out_cap;
    unsigned long long* n_out;
    DevCounters* ctr;
};

size_t bucket_pass_smem(int a);
void launch_bucket_count(const uint64_t* pw, const uint64_t* vw, uint64_t n_units, uint64_t units_per_cta,
                         int n_ctas, const PassParams& p, int a, uint32_t* counts, cudaStream_t st);
void launch_bucket_offsets(const uint32_t* counts, int n_ctas, int a, int pad4, uint64_t* rel, uint32_t* total,
                           cudaStream_t st);
void launch_bucket_base(uint64_t* rel, const uint64_t* starts, int n_ctas, int a, cudaStream_t st);
size_t staged_scatter_smem(int a);
size_t staged_seg_smem(int a);
// A run of hashes handled by one CTA: src + off .. src + off + len; group =
// the level-1 group the run belongs to (0 with a single level).
struct SegDesc {
    uint64_t off, len, group, pad;
};
// mode 4: the extraction pass writes every CTA's hashes to its own segment of
// a linear array (plus counts); the staged scatter then moves the segments.
// accumulate: add the CTAs' counts to their rows (a later piece of the same
// segments, launched with the same number of CTAs).
// Windows outside [p.h_lo, p.h_hi] are dropped (their number kept goes to
// ctr->kept when the range is not the whole hash space).
void launch_extract_count(const uint64_t* pw, const uint64_t* vw, uint64_t n_units, uint64_t units_per_cta,
                          int n_ctas, const PassParams& p, int a, uint32_t* counts, uint64_t* g_cursor, SegDesc* seg,
                          uint64_t* lin, DevCounters* ctr, cudaStream_t st,
                          bool accumulate = false);
// Two grouping levels with a first one of a1 <= kStreamBits bits: CTA c's hashes
// of group g go to a stream of at most cap hashes at lin_off + (c 2^a1 + g) cap
// (segment seg[c 2^a1 + g]); counts rows over all 2^a partitions.  *overflow is
// set when a stream had no room for all.
constexpr int kStreamBits = 2;
uint32_t extract_groups_cap(uint64_t units_per_cta, int a1);
void launch_extract_groups(const uint64_t* pw, const uint64_t* vw, uint64_t n_units, uint64_t units_per_cta,
                           int n_ctas, const PassParams& p, int a1, int a, uint32_t* counts, uint32_t cap,
                           SegDesc* seg, uint64_t lin_off, uint64_t* lin, unsigned* overflow, cudaStream_t st,
                           bool accumulate);
// Staged scatter of segment c into its runs (base: within their buckets,
// which begin at starts): bucket (h >> (64 - a1 - a2)) mod
// 2^a2; with a1 > 0 only hashes of the segment's level-1 group.  Segment c
// comes in n_pieces pieces segs[c], segs[c + n_segs], ...  Nothing is moved where
// *skip is set by then.
void launch_scatter_staged_seg(const uint64_t* src, const SegDesc* segs, int n_segs, int n_pieces, int a1, int a2,
                               const uint64_t* base, const uint64_t* starts, uint64_t* out, cudaStream_t st,
                               const unsigned* skip = nullptr);
// Batched ingest: the read batches of several jobs extracted and grouped by
// one set of launches.  Each batch is cut into items of whole units; the
// extraction and the staged scatter are persistent kernels over the item
// queue, the per-bucket offsets and scans cover every batch in one launch each.  Per batch: histogram rows and segments of its items, its
// linear hashes, the runs' bases in their buckets, its bucket totals and starts
// (the batch's partition starts) and its grouped hashes.
struct IngestBatch {
    const uint64_t* pw;
    const uint64_t* vw;
    uint64_t n_units;
    PassParams p;
    int a;             // bucket bits (the first grouping level)
    uint32_t item0;    // first item of the batch in the queue
    uint32_t n_items;  // items of upi units (the last one shorter)
    uint64_t upi;
    uint32_t* counts;   // [n_items][2^a]
    SegDesc* seg;       // [n_items]
    uint64_t* lin;      // linear hashes
    unsigned long long* g_cursor;
    DevCounters* ctr;
    uint64_t* rel;      // [n_items][2^a]: run starts within their bucket
    uint32_t* total;    // [2^a]
    uint64_t* starts;   // [2^a + 1]
    uint64_t* out;      // grouped hashes
    uint64_t bucket_off;  // first (batch, bucket) index of the batch: sum of 2^a over earlier batches
};
struct IngestPlan {
    const IngestBatch* batches;
    const uint32_t* item_batch;  // batch of every item
    unsigned int* head;          // [0] extraction queue, [1] scatter queue
    uint32_t n_batches, n_items;
    uint64_t n_buckets;  // sum of 2^a
    int max_a;
};
size_t ingest_scatter_smem(int max_a);
// The four launches; `plan` is on the device, its arrays too.  ranged: some
// batch keeps only a hash range; all_k31: every batch has k = 31.
void launch_ingest(const IngestPlan* plan, const IngestPlan& host_plan, bool ranged, bool all_k31, int sm_count,
                   cudaStream_t st);
// Level-2 re-bucketing of level-1 groups: per-segment counts, per-(group,
// partition) offsets and totals (padded to 4).
void launch_count_seg(const uint64_t* src, const SegDesc* segs, int n_segs, int a1, int a2, uint32_t* counts,
                      cudaStream_t st);
void launch_regroup_offsets(const uint32_t* counts, const uint32_t* vlo, int a1, int a2, uint64_t* rel,
                            uint32_t* total, cudaStream_t st);
void launch_bucket_scatter(const uint64_t* pw, const uint64_t* vw, uint64_t n_units, uint64_t units_per_cta,
                           int n_ctas, const PassParams& p, int a, int mode, const uint64_t* base, uint64_t* cursor,
                           uint64_t* out, cudaStream_t st);
// Dynamic shared memory of a consumer CTA: the table and filter words of one
// (sub-range of a) partition, and its warps' queues.
constexpr int kConsumeSliceLog2 = 13;  // filter words of a sub-range, at most
constexpr int kWarpQueue = 64;         // windows a consumer warp's queue holds (under 32, plus a step's)
size_t consume_smem(int slice_log2, int table_log2, int n_samples);
size_t consume_queue_smem(int threads);
void launch_fb_claim(const FallbackArgs& F, int bt, cudaStream_t st);
void launch_fb_recount(const FallbackArgs& F, int bt, cudaStream_t st);
void launch_fb_compact(const FallbackArgs& F, cudaStream_t st);
void launch_prefix_hist(const uint64_t* keys, DevCounters* ctr, uint64_t cap, int key_bits, int bits,
                        uint32_t* hist, const Grid& g, cudaStream_t st);

// The device's opt-in shared memory per block (cached per device).
int max_optin_smem();

// Let func launch with as much dynamic shared memory as the device allows
// beside its static shared memory.  The attribute belongs to the function and
// is shared by every host thread, so it is always set to the same value, the
// maximum, never to one launch's need: jobs launching on other threads cannot
// lower it under each other.
template <typename F>
inline cudaError_t allow_max_dynamic_smem(F func) {
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, func);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                max_optin_smem() - (int)fa.sharedSizeBytes);
}

}  // namespace kc
