// The paper's two-filter Prune chain (Section III, Prune and Count units) on
// the direct strategy's resident reads (sm_103a).
//
// Prune  every valid window ORs its bit pattern into the first filter; a
//        window whose bits were all set already (the key was seen before, or
//        the filter answers with a false positive) ORs the same pattern into
//        the second filter, at the same word.  The second filter then holds
//        every key seen at least twice, plus some false positives.
// Count  every valid window whose key is in the second filter is claimed in
//        the table and counted there in the same step: the second filter is
//        complete before counting starts, so one pass gives exact counts, and
//        the compaction (count >= min_count) removes the false positives, as
//        the paper's Unify unit does.
// With min_count <= 1 every window is counted.

#include "kc_ctx.h"

namespace kc {
namespace {

constexpr unsigned kFullMask = 0xffffffffu;

// Both kernels are bound by the latency of random accesses to the filters and
// the table, one after the other for each window: a lane has two windows of
// its unit in flight, and a warp takes a quarter of 32 units at a time, so that
// the last items spread over the SMs.  2.4e7 windows, 2^28-bit filters: Prune
// 0.295 ms, Count 0.479; with one window in flight, whole units, and the table
// probed once to claim and once more to count 0.315 and 0.688.
constexpr int kParts = 4;  // items of 64 / kParts window starts a lane

// The next window of the lane's item: its key's hash and bit pattern.
struct Probe {
    bool has;
    uint64_t key, h;
    unsigned long long pat;
};

__device__ __forceinline__ Probe next_probe(const UnitWords& uw, uint64_t& vm, const PassParams& p) {
    Probe r{vm != 0ull, 0, 0, 0};
    if (r.has) {
        const int j = __clzll(vm);
        vm &= ~(0x8000000000000000ull >> j);
        r.key = canonical_key(window_code(uw.w0, uw.w1, uw.w2, j, p.rc_shift), p);
        r.h = mixer64(r.key);
        r.pat = bloom_pattern(mixer64(r.h), p.n_hashes);
    }
    return r;
}

// Valid-window bits of part `part` of a unit.
__device__ __forceinline__ uint64_t part_bits(uint64_t v, int part) {
    constexpr int w = 64 / kParts;
    return v & (~0ull << (64 - w)) >> (part * w);
}

__global__ void __launch_bounds__(256, 6) k_prune(const uint64_t* __restrict__ pw, const uint64_t* __restrict__ vw,
                                               uint64_t n_units, PassParams p, unsigned long long* __restrict__ bf1,
                                               unsigned long long* __restrict__ bf2, DevCounters* __restrict__ ctr) {
    const int lane = threadIdx.x & 31;
    const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    const uint64_t n_items = (n_units + 31) / 32 * kParts;
    unsigned long long promoted = 0;
    for (uint64_t item = warp; item < n_items; item += n_warps) {
        const UnitWords uw = load_unit(pw, vw, item / kParts * 32 + lane, n_units, lane);
        uint64_t vm = part_bits(uw.v, (int)(item % kParts));
        const int n_iter = __reduce_max_sync(kFullMask, (unsigned)__popcll(vm));
        for (int it = 0; it < n_iter; it += 2) {
            const Probe a = next_probe(uw, vm, p), b = next_probe(uw, vm, p);
            unsigned long long old_a = 0, old_b = 0;
            if (a.has) old_a = atomicOr(bf1 + (a.h >> p.bloom_shift), a.pat);
            if (b.has) old_b = atomicOr(bf1 + (b.h >> p.bloom_shift), b.pat);
            if (a.has && (old_a & a.pat) == a.pat) {
                atomicOr(bf2 + (a.h >> p.bloom_shift), a.pat);
                ++promoted;
            }
            if (b.has && (old_b & b.pat) == b.pat) {
                atomicOr(bf2 + (b.h >> p.bloom_shift), b.pat);
                ++promoted;
            }
            __syncwarp();
        }
    }
    promoted = warp_sum(promoted);
    if (lane == 0 && promoted) atomicAdd(&ctr->candidates, promoted);
}

__global__ void __launch_bounds__(256, 6) k_count_chain(const uint64_t* __restrict__ pw,
                                                     const uint64_t* __restrict__ vw, uint64_t n_units, PassParams p,
                                                     const unsigned long long* __restrict__ bf2,
                                                     Slot* __restrict__ table, DevCounters* __restrict__ ctr) {
    const int lane = threadIdx.x & 31;
    const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    const uint64_t n_items = (n_units + 31) / 32 * kParts;
    unsigned long long claimed = 0;
    for (uint64_t item = warp; item < n_items; item += n_warps) {
        const UnitWords uw = load_unit(pw, vw, item / kParts * 32 + lane, n_units, lane);
        uint64_t vm = part_bits(uw.v, (int)(item % kParts));
        const int n_iter = __reduce_max_sync(kFullMask, (unsigned)__popcll(vm));
        for (int it = 0; it < n_iter; it += 2) {
            const Probe a = next_probe(uw, vm, p), b = next_probe(uw, vm, p);
            // the filter words, then the home slots of the windows they let through
            unsigned long long word_a = ~0ull, word_b = ~0ull;
            if (a.has && !p.all_candidates) word_a = __ldg(bf2 + (a.h >> p.bloom_shift));
            if (b.has && !p.all_candidates) word_b = __ldg(bf2 + (b.h >> p.bloom_shift));
            const bool in_a = a.has && (word_a & a.pat) == a.pat, in_b = b.has && (word_b & b.pat) == b.pat;
            const uint64_t home_a = a.h >> p.table_shift, home_b = b.h >> p.table_shift;
            unsigned long long cur_a = 0, cur_b = 0;
            if (in_a) cur_a = __ldcg(&table[home_a].key1);
            if (in_b) cur_b = __ldcg(&table[home_b].key1);
            if (in_a) claimed += table_add(table, p.table_mask, home_a, a.key + 1, cur_a, p.sample, ctr);
            if (in_b) claimed += table_add(table, p.table_mask, home_b, b.key + 1, cur_b, p.sample, ctr);
            __syncwarp();
        }
    }
    claimed = warp_sum(claimed);
    if (lane == 0 && claimed) atomicAdd(&ctr->claimed, claimed);
}

// Four times the resident CTAs and more: with 6 or 7 items a warp in 1.6 waves
// the last ones ran on a half-empty chip, now CTAs of one or two items a warp
// follow each other as SMs come free.  2.4e7 windows, as many as are resident:
// Count 0.55 ms; 18, 24, 32 an SM, unbounded: 0.486, 0.495, 0.479, 0.483.
unsigned grid_for_units(uint64_t n_units, const Grid& g) {
    uint64_t blocks = (n_units * kParts + 255) / 256;
    if (blocks < 1) blocks = 1;
    if (blocks > 4 * (uint64_t)g.ctas()) blocks = 4 * (uint64_t)g.ctas();
    return (unsigned)blocks;
}

}  // namespace

void launch_prune(const uint64_t* pw, const uint64_t* vw, uint64_t n_units, const PassParams& p, uint64_t* bf1,
                  uint64_t* bf2, DevCounters* ctr, const Grid& g, cudaStream_t st) {
    k_prune<<<grid_for_units(n_units, g), 256, 0, st>>>(pw, vw, n_units, p,
                                                         reinterpret_cast<unsigned long long*>(bf1),
                                                         reinterpret_cast<unsigned long long*>(bf2), ctr);
}

void launch_count_chain(const uint64_t* pw, const uint64_t* vw, uint64_t n_units, const PassParams& p,
                        const uint64_t* bf2, Slot* table, DevCounters* ctr, const Grid& g, cudaStream_t st) {
    k_count_chain<<<grid_for_units(n_units, g), 256, 0, st>>>(
        pw, vw, n_units, p, reinterpret_cast<const unsigned long long*>(bf2), table, ctr);
}

}  // namespace kc
