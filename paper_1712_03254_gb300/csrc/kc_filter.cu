// Downstream of the count (sm_103a): the result in the paper's 16-byte k-mer
// item form, its joint count spectrum, and the Filter unit.
//
// Items     Section III-D: one k-mer item is 8 bytes of k-mer, 4 bytes holding
//           the two samples' counts and 4 bytes of padding.  Counts are kept
//           as uint32 by the library; the item stores each as 16 bits,
//           clamped to 65535.
// Spectrum  number of result keys per pair of clamped counts: the per-sample
//           imbalance summary of a joint normal/tumoral table.
// Filter    Section II-B: the Filter unit selects the k-mers whose
//           frequencies differ between the normal and the tumoral sample,
//           then reads the input again and looks every k-mer up in the table
//           to find the reads that carry selected k-mers.  Selection:
//           count[t] >= min_tumor, count[n] <= max_normal, count[t] >=
//           ratio * count[n] (the paper gives no threshold).  The selected
//           keys are compacted in key order and both orientations of each are
//           stored in a lookup table of 16-byte buckets of four fingerprints;
//           the rescan rolls every valid window's forward code and probes
//           the table; hits are marked per 64-base unit and then counted per
//           read.

#include <algorithm>
#include <atomic>
#include <cstring>

#include "kc_ctx.h"

namespace kc {
namespace {

constexpr int kTileThreads = 256;
constexpr int kTileRounds = 16;
constexpr uint64_t kTileItems = (uint64_t)kTileThreads * kTileRounds;

struct SelSpec {
    int tumor;
    uint32_t min_tumor, max_normal, ratio;
};

// Packed counts: sample 0 in the low 32 bits, sample 1 in the high 32 bits.
__device__ __forceinline__ bool is_selected(uint64_t v, const SelSpec& s) {
    const uint64_t c0 = (uint32_t)v, c1 = v >> 32;
    const uint64_t t = s.tumor ? c1 : c0, n = s.tumor ? c0 : c1;
    return t >= s.min_tumor && n <= s.max_normal && t >= (uint64_t)s.ratio * n;
}

// Ordered compaction in tiles of kTileItems: the first kernel counts a tile's
// kept items, a scan gives each tile its output start, the second kernel
// writes the kept items of a tile in their input order.
struct SelectPred {
    const uint64_t* vals;
    SelSpec spec;
    __device__ bool operator()(uint64_t i) const { return is_selected(vals[i], spec); }
};

struct HitPred {
    const uint32_t* hits;
    __device__ bool operator()(uint64_t i) const { return hits[i] != 0u; }
};

// Sum of a value over the CTA's THREADS threads, in thread 0.
template <int THREADS>
__device__ __forceinline__ uint32_t tile_sum(uint32_t v) {
    __shared__ uint32_t s_sum[THREADS / 32];
    v = __reduce_add_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < THREADS / 32; ++w) v += s_sum[w];
    return v;
}

template <typename Pred>
__global__ void __launch_bounds__(kTileThreads) k_tile_count(Pred pred, uint64_t n, uint32_t* __restrict__ counts) {
    const uint64_t base = (uint64_t)blockIdx.x * kTileItems;
    uint32_t mine = 0;
#pragma unroll 8
    for (int r = 0; r < kTileRounds; ++r) {
        const uint64_t i = base + (uint64_t)r * kTileThreads + threadIdx.x;
        mine += i < n && pred(i);
    }
    const uint32_t total = tile_sum<kTileThreads>(mine);
    if (threadIdx.x == 0) counts[blockIdx.x] = total;
}

// Writer for the selection: key and packed counts.
struct SelectWrite {
    const uint64_t* keys;
    const uint64_t* vals;
    uint64_t* out_keys;
    uint64_t* out_vals;
    __device__ void operator()(uint64_t i, uint64_t pos) const {
        out_keys[pos] = keys[i];
        out_vals[pos] = vals[i];
    }
};

// Writer for candidate reads: the read's index.
struct IndexWrite {
    uint64_t* out;
    __device__ void operator()(uint64_t i, uint64_t pos) const { out[pos] = i; }
};

// Each warp a row of kTileRounds * 32 items of the tile: the ballots of its
// rounds stay in its lanes (lane r: round r), one barrier gives the warps their
// output starts, then the kept items are written in order.  (A barrier pair
// and a prefix a round took 40 us where this takes 37 for 5.5 M keys, 151 k
// kept, and 13 against 5 for the candidates of 600 k reads.)
template <typename Pred, typename Write>
__global__ void __launch_bounds__(kTileThreads) k_tile_write(Pred pred, Write write, uint64_t n,
                                                             const uint64_t* __restrict__ starts) {
    __shared__ uint32_t warp_n[kTileThreads / 32];
    static_assert(kTileRounds <= 32, "a lane per round");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t base = (uint64_t)blockIdx.x * kTileItems + (uint64_t)warp * (kTileRounds * 32) + lane;
    unsigned mine = 0;
#pragma unroll 8
    for (int r = 0; r < kTileRounds; ++r) {
        const uint64_t i = base + r * 32;
        const unsigned ballot = __ballot_sync(0xffffffffu, i < n && pred(i));
        if (lane == r) mine = ballot;
    }
    const uint32_t total = __reduce_add_sync(0xffffffffu, (unsigned)__popc(mine));
    if (lane == 0) warp_n[warp] = total;
    __syncthreads();
    uint64_t out = starts[blockIdx.x];
    for (int w = 0; w < warp; ++w) out += warp_n[w];
    if (total == 0) return;
    for (int r = 0; r < kTileRounds; ++r) {
        const unsigned ballot = __shfl_sync(0xffffffffu, mine, r);
        if ((ballot >> lane) & 1u) write(base + r * 32, out + (uint32_t)__popc(ballot & ((1u << lane) - 1u)));
        out += __popc(ballot);
    }
}

// Selection table.  It holds both orientations of every selected k-mer (the
// forward code of a window then finds its canonical key without the reverse
// complement): 2^lb buckets of four slots.  A slot is a 32-bit fingerprint
// (0 = free) in the bucket's 16-byte fingerprint word, with the 64-bit code
// in a parallel array, read only when a fingerprint matches; at most a
// quarter of the slots are taken.  A code goes to the first free slot of its
// bucket or of the buckets after it, so slots fill in order and a bucket
// whose last slot is free ends every probe through it.
// Hash: Fibonacci hashing, h = code * 2^64/golden ratio; bucket = top lb bits
// of h, fingerprint = the 32 bits below them with the lowest bit set.
//
// Small selections also get a prefilter that the rescan keeps in shared
// memory: kPreWords 32-bit words, each entry setting two bits of one word
// (word from the top 32 bits of h, bits from h's bits 14..18 and 20..24).  A
// window whose two bits are not both set is not in the table, and most
// windows are rejected there instead of by a random global load.
constexpr uint32_t kPreWords = 49152;                 // 192 KiB of shared memory
constexpr uint64_t kPreMaxEntries = kPreWords * 32 / 4;  // at most a quarter of its bits per entry pair

struct SelTable {
    unsigned int* fp;      // 4 per bucket
    unsigned long long* code;  // 4 per bucket
    unsigned int* pre;     // kPreWords prefilter words (null: no prefilter)
    int lb;
    uint64_t mask;         // buckets - 1
};

__device__ __forceinline__ uint64_t sel_h(uint64_t code) { return code * 0x9e3779b97f4a7c15ull; }

// Bucket and fingerprint of a hash, 8 <= lb <= 32: both from 32-bit shifts.
__device__ __forceinline__ uint32_t sel_bucket(uint64_t h, int lb) { return (uint32_t)(h >> 32) >> (32 - lb); }
__device__ __forceinline__ unsigned sel_fp(uint64_t h, int lb) {
    return __funnelshift_rc((uint32_t)h, (uint32_t)(h >> 32), 32 - lb) | 1u;  // never 0 (0 marks a free slot)
}

__device__ __forceinline__ void sel_hash(uint64_t code, int lb, uint64_t& bucket, unsigned& fp) {
    const uint64_t h = sel_h(code);
    bucket = sel_bucket(h, lb);
    fp = sel_fp(h, lb);
}

__device__ __forceinline__ uint32_t pre_word(uint64_t h) {
    return (uint32_t)(((h >> 32) * (uint64_t)kPreWords) >> 32);
}

__device__ __forceinline__ uint32_t pre_bits(uint64_t h) {
    return (1u << ((uint32_t)(h >> 20) & 31u)) | (1u << ((uint32_t)(h >> 14) & 31u));
}

__device__ __forceinline__ bool sel_insert(const SelTable& T, uint64_t code) {
    uint64_t b;
    unsigned fp;
    sel_hash(code, T.lb, b, fp);
    if (T.pre) {
        const uint64_t h = sel_h(code);
        atomicOr(T.pre + pre_word(h), pre_bits(h));
    }
    for (uint64_t probe = 0; probe <= T.mask; ++probe) {
        for (int s = 0; s < 4; ++s)
            if (atomicCAS(T.fp + 4 * b + s, 0u, fp) == 0u) {
                T.code[4 * b + s] = code;
                return true;
            }
        b = (b + 1) & T.mask;
    }
    return false;
}

// Both orientations of every selected canonical key.
__global__ void k_sel_insert(const uint64_t* __restrict__ keys, uint64_t n, SelTable T, PassParams p,
                             DevCounters* __restrict__ ctr) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint64_t key = keys[i];
        const uint64_t rc = reverse_pairs(key ^ p.kmask) >> p.rc_shift;
        bool ok = sel_insert(T, key);
        if (rc != key) ok = ok && sel_insert(T, rc);  // an even-k palindrome is its own reverse complement
        if (!ok) atomicOr(&ctr->err, DERR_INTERNAL);  // cannot happen: the table is at most half full
    }
}

// Matching slots of a bucket word: confirm against the stored codes.
__device__ __forceinline__ bool sel_confirm(const SelTable& T, uint64_t b, uint4 q, unsigned fp, uint64_t code) {
    const unsigned f[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int s = 0; s < 4; ++s)
        if (f[s] == fp && __ldg(T.code + 4 * b + s) == code) return true;
    return false;
}

// Probe from the bucket after b on (rare: b's slots are all taken).
__device__ __forceinline__ bool sel_probe_rest(const SelTable& T, uint64_t b, unsigned fp, uint64_t code) {
    for (uint64_t probe = 0; probe < T.mask; ++probe) {
        b = (b + 1) & T.mask;
        const uint4 q = __ldg(reinterpret_cast<const uint4*>(T.fp) + b);
        if ((q.x == fp || q.y == fp || q.z == fp || q.w == fp) && sel_confirm(T, b, q, fp, code)) return true;
        if (q.w == 0u) return false;
    }
    return false;
}

// Whether both prefilter bits of h are set in word (in bit 0): the word rotated
// by the two bit numbers.
__device__ __forceinline__ uint32_t pre_test(uint32_t word, uint64_t h) {
    return __funnelshift_r(word, word, (uint32_t)h >> 20) & __funnelshift_r(word, word, (uint32_t)h >> 14);
}

// Filter rescan: one lane per 64-base unit; the lane cuts the forward codes of
// its unit's 64 window starts out of the unit's words (forward_code) and probes
// the selection for four windows at a time (four 16-byte bucket loads in flight).  PRE: one
// 1024-thread CTA per SM holds the prefilter in shared memory and loads a
// bucket only for windows that pass it.  Hits go to the unit's hit mask (bit
// 63 - j: the window starting at base j of the unit, as the valid-window
// bits), written once per unit; k_read_hits turns the masks into hits per
// read.
constexpr int kFilterThreads = 256;
constexpr int kFilterThreadsPre = 1024;

template <bool PRE, int K, int J0>
__device__ __forceinline__ void filter_four(const WindowWords& w, unsigned valid, int rc_shift, const SelTable& T,
                                            const uint32_t* s_pre, unsigned& hits) {
    const uint64_t code[4] = {forward_code<K, J0>(w, rc_shift), forward_code<K, J0 + 1>(w, rc_shift),
                              forward_code<K, J0 + 2>(w, rc_shift), forward_code<K, J0 + 3>(w, rc_shift)};
    uint64_t h[4];
    bool probe[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        h[t] = sel_h(code[t]);
        probe[t] = (valid >> (7 - J0 - t)) & 1u;
        if (PRE && probe[t]) probe[t] = pre_test(s_pre[pre_word(h[t])], h[t]) & 1u;
    }
    if (!(probe[0] || probe[1] || probe[2] || probe[3])) return;
    uint4 q[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        q[t] = make_uint4(0u, 0u, 0u, 0u);
        if (probe[t]) q[t] = __ldg(reinterpret_cast<const uint4*>(T.fp) + sel_bucket(h[t], T.lb));
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const unsigned fp = sel_fp(h[t], T.lb);
        const bool match = q[t].x == fp || q[t].y == fp || q[t].z == fp || q[t].w == fp;
        if (!match && q[t].w == 0u) continue;  // not in the table (skipped windows read as empty)
        const uint64_t b = sel_bucket(h[t], T.lb);
        bool hit = match && sel_confirm(T, b, q[t], fp, code[t]);
        if (!hit && q[t].w != 0u) hit = sel_probe_rest(T, b, fp, code[t]);
        if (hit) hits |= 1u << (7 - J0 - t);
    }
}

template <bool PRE, int K>
__global__ void __launch_bounds__(PRE ? kFilterThreadsPre : kFilterThreads, PRE ? 1 : 4)
    k_filter_hits(const uint64_t* __restrict__ pw, uint64_t n_words, const uint64_t* __restrict__ vw, uint64_t n_units,
                  PassParams p, SelTable T, uint64_t* __restrict__ hitmask, DevCounters* __restrict__ ctr) {
    extern __shared__ uint4 s_pre4[];
    const uint32_t* s_pre = reinterpret_cast<const uint32_t*>(s_pre4);
    if (PRE) {
        const uint4* g = reinterpret_cast<const uint4*>(T.pre);
        for (uint32_t i = threadIdx.x; i < kPreWords / 4; i += blockDim.x) s_pre4[i] = __ldg(g + i);
        __syncthreads();
    }
    const int lane = threadIdx.x & 31;
    const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long found = 0;
    // The units in whole rounds of the grid's lanes, then the rest, whose lanes take
    // a half to an eighth of a unit each if they are few (9.03 rounds: 188 -> 176 us
    // and 285 -> 278, no hits and 1.5 M).
    const uint64_t rest = n_units / (n_warps * 32) * (n_warps * 32);
    for (int lp = 0, at_rest = rest == 0; at_rest < 2; ++at_rest) {
    if (at_rest) lp = parts_log2(n_units - rest, n_warps * 32);
    const uint64_t end = at_rest ? n_units : rest;
    for (uint64_t base = ((at_rest ? rest : 0) << lp) + warp * 32; base < end << lp; base += n_warps * 32) {
        const uint64_t u = base + lane;
        UnitWords uw{0, 0, 0, 0};
        if (lp == 0) uw = load_unit(pw, vw, u, end, lane, n_words);
        else if (u < end << lp) uw = load_part(pw, vw, u >> lp, (int)u & ((1 << lp) - 1), lp, n_words);
        uint64_t vm = uw.v, hm = 0;
        WindowWords w = window_words(uw.w0, uw.w1, uw.w2);
        for (int j0 = 0; j0 < 64 >> lp; j0 += 8, vm <<= 8) {  // eight windows: their bits on top of vm
            unsigned hits = 0;
            const unsigned valid = (unsigned)(vm >> 56);
            if (valid) {
                filter_four<PRE, K, 0>(w, valid, p.rc_shift, T, s_pre, hits);
                filter_four<PRE, K, 4>(w, valid, p.rc_shift, T, s_pre, hits);
            }
            hm = (hm << 8) | hits;
            next_windows(w);
        }
        if (u < end << lp) {  // the first window's bit is the unit's highest: part 0 is its last bytes
            if (lp == 0) hitmask[u] = hm;
            else if (lp == 1) reinterpret_cast<uint32_t*>(hitmask)[u ^ 1] = (uint32_t)hm;
            else if (lp == 2) reinterpret_cast<uint16_t*>(hitmask)[u ^ 3] = (uint16_t)hm;
            else reinterpret_cast<uint8_t*>(hitmask)[u ^ 7] = (uint8_t)hm;
        }
        found += __popcll(hm);
    }
    }
    found = warp_sum(found);
    if (lane == 0 && found) atomicAdd(&ctr->candidates, found);
}

// hits[r] = hit-mask bits inside read r's bases (local positions o0 .. o1 - 1;
// the mask has bits only at valid window starts, which lie inside reads), and
// per tile of kTileItems reads how many of them have hits (the compaction's
// counts).  Thread per read, CTA per tile.
constexpr int kReadThreads = 1024;

__global__ void __launch_bounds__(kReadThreads) k_read_hits(const uint64_t* __restrict__ offsets, uint64_t n_reads,
                                                            uint64_t base, uint64_t n_units,
                                                            const uint64_t* __restrict__ hitmask,
                                                            unsigned int* __restrict__ hits,
                                                            uint32_t* __restrict__ counts) {
    uint32_t mine = 0;
#pragma unroll 4
    for (int round = 0; round < (int)(kTileItems / kReadThreads); ++round) {
        const uint64_t r = (uint64_t)blockIdx.x * kTileItems + (uint64_t)round * kReadThreads + threadIdx.x;
        unsigned n = 0;
        if (r < n_reads) {
            const uint64_t o0 = offsets[r] - base, o1 = offsets[r + 1] - base;
            if (o1 > o0) {
                const uint64_t u0 = o0 >> 6, u1 = (o1 - 1) >> 6;
                for (uint64_t u = u0; u <= u1 && u < n_units; ++u) {
                    uint64_t m = hitmask[u];
                    if (u == u0) m &= ~0ull >> (o0 & 63);                 // from base o0 on
                    const int e = (int)((o1 - 1) & 63);
                    if (u == u1 && e < 63) m &= ~(~0ull >> (e + 1));      // up to base o1 - 1
                    n += (unsigned)__popcll(m);
                }
            }
            hits[r] = n;
        }
        mine += n != 0u;
    }
    const uint32_t total = tile_sum<kReadThreads>(mine);
    if (threadIdx.x == 0) counts[blockIdx.x] = total;
}

__global__ void k_items16(const uint64_t* __restrict__ keys, const uint64_t* __restrict__ vals, uint64_t n,
                          int n_samples, ulonglong2* __restrict__ out) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint64_t v = vals[i];
        const uint64_t lo = (uint32_t)v, hi = n_samples == 2 ? v >> 32 : 0ull;
        const uint64_t c0 = lo < 65535u ? lo : 65535u, c1 = hi < 65535u ? hi : 65535u;
        out[i] = make_ulonglong2(keys[i], c0 | (c1 << 16));  // padding (bytes 12..15) zero
    }
}

// Spectrum with a per-CTA shared-memory histogram (n_bins <= kSmemBins) or
// straight global atomics.
constexpr int kSmemBins = 8192;

__device__ __forceinline__ uint64_t spectrum_bin(uint64_t v, int n_samples, uint64_t cap) {
    const uint64_t lo = (uint32_t)v, hi = v >> 32;
    const uint64_t c0 = lo < cap ? lo : cap;
    if (n_samples == 1) return c0;
    return c0 * (cap + 1) + (hi < cap ? hi : cap);
}

__global__ void __launch_bounds__(256) k_spectrum(const uint64_t* __restrict__ vals, uint64_t n, int n_samples,
                                                  uint64_t cap, uint64_t n_bins,
                                                  unsigned long long* __restrict__ hist) {
    __shared__ unsigned int local[kSmemBins];
    const bool shared = n_bins <= (uint64_t)kSmemBins;
    if (shared)
        for (uint64_t b = threadIdx.x; b < n_bins; b += blockDim.x) local[b] = 0u;
    __syncthreads();
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint64_t b = spectrum_bin(vals[i], n_samples, cap);
        if (shared) atomicAdd(local + b, 1u);
        else atomicAdd(hist + b, 1ull);
    }
    __syncthreads();
    if (shared)
        for (uint64_t b = threadIdx.x; b < n_bins; b += blockDim.x)
            if (local[b]) atomicAdd(hist + b, (unsigned long long)local[b]);
}

// Stem-grouped items.  A result key K = x S y (first base x, stem S of k-2
// bases, last base y) fills entry (x, y) of stem S when S is canonical (not
// above its reverse complement S'); otherwise its reverse complement
// y' S' x' (complements y', x') fills entry (y', x') of stem S'.  A stem that
// is its own reverse complement gets both entries.  One record per entry:
// key = stem << 4 | entry, value = the key's packed counts; records are
// claimed with one atomic per CTA and round (one per warp, all on one address,
// took 35 us for 1.2 M keys, this 12).
__global__ void __launch_bounds__(kTileThreads) k_stem_records(const uint64_t* __restrict__ keys,
                                                               const uint64_t* __restrict__ vals, uint64_t n, int k,
                                                               uint64_t* __restrict__ rec_keys,
                                                               uint64_t* __restrict__ rec_vals,
                                                               DevCounters* __restrict__ ctr) {
    const int lane = threadIdx.x & 31;
    const int sb = 2 * (k - 2);  // stem bits, 2..58
    const uint64_t smask = (1ull << sb) - 1ull;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    __shared__ uint32_t warp_n[kTileThreads / 32];
    __shared__ unsigned long long s_base;
    const uint64_t n_round = (n + kTileThreads - 1) / kTileThreads * kTileThreads;  // whole CTAs in every round
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_round; i += stride) {
        uint64_t r0 = 0, r1 = 0, v = 0;
        int cnt = 0;
        if (i < n) {
            const uint64_t K = keys[i];
            v = vals[i];
            const uint64_t x = K >> (2 * k - 2), y = K & 3ull;
            const uint64_t S = (K >> 2) & smask;
            const uint64_t Sr = reverse_pairs(S ^ smask) >> (64 - sb);
            const uint64_t e_fwd = 4 * x + y, e_rev = 4 * (3 - y) + (3 - x);
            if (S < Sr) {
                r0 = (S << 4) | e_fwd;
                cnt = 1;
            } else if (S > Sr) {
                r0 = (Sr << 4) | e_rev;
                cnt = 1;
            } else {
                r0 = (S << 4) | e_fwd;
                r1 = (S << 4) | e_rev;
                cnt = e_rev == e_fwd ? 1 : 2;  // equal only for a k-mer that is its own reverse complement
            }
        }
        // claim of cnt slots per lane for the CTA
        unsigned incl = (unsigned)cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) warp_n[threadIdx.x >> 5] = incl;
        __syncthreads();
        unsigned before = 0, total = 0;
#pragma unroll
        for (int w = 0; w < kTileThreads / 32; ++w) {
            if (w < (int)(threadIdx.x >> 5)) before += warp_n[w];
            total += warp_n[w];
        }
        if (threadIdx.x == 0) s_base = total ? atomicAdd(&ctr->survivors, (unsigned long long)total) : 0ull;
        __syncthreads();
        const uint64_t pos = s_base + before + incl - cnt;
        if (cnt >= 1) {
            rec_keys[pos] = r0;
            rec_vals[pos] = v;
        }
        if (cnt == 2) {
            rec_keys[pos + 1] = r1;
            rec_vals[pos + 1] = v;
        }
    }
}

// A sorted record starts an item when its stem differs from the previous one.
struct StemStartPred {
    const uint64_t* rec_keys;
    __device__ bool operator()(uint64_t i) const { return i == 0 || (rec_keys[i] >> 4) != (rec_keys[i - 1] >> 4); }
};

// One thread per item: its records are starts[j] .. starts[j+1] - 1 (n_rec
// for the last); 72 bytes = stem, 16 counts of sample 0, 16 of sample 1, as
// nine 64-bit words (count e of a sample in bits 16 (e % 4) of word e / 4).
// The CTA's items are put together in shared memory and leave as one
// contiguous block: nine stores 72 bytes apart a thread took 61 us for 1.2 M
// items (88 MB), this 39.
__global__ void __launch_bounds__(kTileThreads) k_stem_items(const uint64_t* __restrict__ rec_keys,
                                                             const uint64_t* __restrict__ rec_vals, uint64_t n_rec,
                                                             const uint64_t* __restrict__ starts, uint64_t n_items,
                                                             int n_samples, uint64_t* __restrict__ out) {
    __shared__ uint64_t s_out[9 * kTileThreads];
    for (uint64_t j0 = (uint64_t)blockIdx.x * kTileThreads; j0 < n_items; j0 += (uint64_t)gridDim.x * kTileThreads) {
        const uint64_t j = j0 + threadIdx.x;
        const unsigned here = (unsigned)(n_items - j0 < kTileThreads ? n_items - j0 : kTileThreads);
        if (threadIdx.x < here) {
            const uint64_t s0 = starts[j], s1 = j + 1 < n_items ? starts[j + 1] : n_rec;
            uint64_t w[8] = {0, 0, 0, 0, 0, 0, 0, 0};
            for (uint64_t r = s0; r < s1; ++r) {
                const int e = (int)(rec_keys[r] & 15ull);
                const uint64_t v = rec_vals[r];
                const uint64_t lo = (uint32_t)v, hi = n_samples == 2 ? v >> 32 : 0ull;
                const uint64_t c0 = lo < 65535u ? lo : 65535u, c1 = hi < 65535u ? hi : 65535u;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if ((e >> 2) == q) {  // registers stay registers: the word is chosen by unrolled compares
                        w[q] |= c0 << (16 * (e & 3));
                        w[4 + q] |= c1 << (16 * (e & 3));
                    }
            }
            uint64_t* o = s_out + 9 * threadIdx.x;  // nine words apart: no bank conflicts
            o[0] = rec_keys[s0] >> 4;
#pragma unroll
            for (int q = 0; q < 8; ++q) o[1 + q] = w[q];
        }
        __syncthreads();
        for (unsigned i = threadIdx.x; i < 9 * here; i += kTileThreads) out[9 * j0 + i] = s_out[i];
        __syncthreads();
    }
}

unsigned grid_of(uint64_t n, unsigned block, unsigned cap) {
    uint64_t g = (n + block - 1) / block;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (unsigned)g;
}

// Resident CTAs of k_filter_hits<false, K> per SM: its grid fills the SMs
// once, no partial second wave.
int filter_blocks_per_sm() {
    static std::atomic<int> cached{0};
    int v = cached.load(std::memory_order_relaxed);
    if (!v) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, k_filter_hits<false, 31>, kFilterThreads, 0) !=
                cudaSuccess ||
            v < 1) {
            cudaGetLastError();
            v = 4;
        }
        cached.store(v, std::memory_order_relaxed);
    }
    return v;
}

// k_filter_hits<true, K> takes 192 KiB of dynamic shared memory (set once per
// device; the value is the same for every caller).
cudaError_t filter_pre_smem_attr() {
    static std::atomic<int> done[64];
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && done[dev].load(std::memory_order_relaxed)) return cudaSuccess;
    cudaError_t e = allow_max_dynamic_smem(k_filter_hits<true, 31>);
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_filter_hits<true, 0>);
    if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev].store(1, std::memory_order_relaxed);
    return e;
}

}  // namespace
}  // namespace kc

namespace kcapi {

void free_selection(kc_handle h) {
    if (h->sel_keys) cudaFreeAsync(h->sel_keys, h->stream);
    if (h->sel_vals) cudaFreeAsync(h->sel_vals, h->stream);
    if (h->sel_table) cudaFreeAsync(h->sel_table, h->stream);
    h->sel_keys = h->sel_vals = h->sel_table = nullptr;
    h->n_sel = 0;
    h->sel_buckets_log2 = 0;
    h->sel_pre = false;
    h->has_selection = false;
}

void free_stems(kc_handle h) {
    if (h->stem_items) cudaFreeAsync(h->stem_items, h->stream);
    h->stem_items = nullptr;
    h->n_stems = 0;
    h->has_stems = false;
}

namespace {

// Bytes per selection bucket: four 32-bit fingerprints and four 64-bit codes.
constexpr uint64_t kSelBucketBytes = 16 + 32;

kc::SelTable sel_table_of(kc_handle h) {
    kc::SelTable T;
    const uint64_t n_buckets = 1ull << h->sel_buckets_log2;
    T.fp = reinterpret_cast<unsigned int*>(h->sel_table);
    T.code = reinterpret_cast<unsigned long long*>(reinterpret_cast<char*>(h->sel_table) + 16 * n_buckets);
    T.pre = h->sel_pre ? reinterpret_cast<unsigned int*>(reinterpret_cast<char*>(h->sel_table) +
                                                          kSelBucketBytes * n_buckets)
                       : nullptr;
    T.lb = h->sel_buckets_log2;
    T.mask = n_buckets - 1;
    return T;
}

// The result on the device: a spilled result is copied back and sorted there.
kc_status device_result(kc_handle h, const char* who) {
    kc_status s = check_open(h);
    if (s != KC_OK) return s;
    if (h->state != State::Finalized) return fail(KC_ERR_STATE, std::string(who) + " before kc_finalize");
    if (!h->spilled || h->n_result == 0) return KC_OK;
    s = resort_spilled(h);
    if (s == KC_ERR_OOM_DEVICE)
        return fail(KC_ERR_OOM_DEVICE, std::string(who) + ": the spilled result does not fit on the device");
    return s;
}

// The tiles of an ordered compaction of n items: per tile its kept items and
// the output start (one block; starts[n_tiles] is the total).
struct Tiles {
    uint64_t n = 0;
    uint64_t *starts = nullptr, *cursor = nullptr;
    uint32_t* counts = nullptr;
    cudaError_t take(uint64_t items, cudaStream_t st) {
        n = std::max<uint64_t>(1, (items + kc::kTileItems - 1) / kc::kTileItems);
        cudaError_t e = kc::dev_alloc(&starts, (n + 1) * 8 + n * 12, st);
        if (e != cudaSuccess) return e;
        cursor = starts + n + 1;
        counts = reinterpret_cast<uint32_t*>(cursor + n);
        return cudaSuccess;
    }
    void leave(cudaStream_t st) {
        if (starts) cudaFreeAsync(starts, st);
        starts = nullptr;
    }
};

// Ordered compaction of n items into the writer's arrays; *kept = how many.
template <typename Pred, typename Write>
kc_status compact_ordered(kc_handle h, Pred pred, Write write, uint64_t n, uint64_t* kept) {
    cudaStream_t st = h->stream;
    Tiles t;
    cudaError_t e = t.take(n, st);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMallocAsync(compaction tiles)");
    kc::k_tile_count<Pred><<<(unsigned)t.n, kc::kTileThreads, 0, st>>>(pred, n, t.counts);
    e = kc::launch_scan(t.counts, t.n, t.starts, t.cursor, st);
    if (e != cudaSuccess) {
        t.leave(st);
        return cuda_fail(e, "tile scan");
    }
    kc::k_tile_write<Pred, Write><<<(unsigned)t.n, kc::kTileThreads, 0, st>>>(pred, write, n, t.starts);
    h->launches += 3;
    KC_LAUNCHED("ordered compaction launches");
    KC_CUDA(cudaMemcpyAsync(kept, t.starts + t.n, 8, cudaMemcpyDeviceToHost, st));
    t.leave(st);
    KC_CUDA(cudaStreamSynchronize(st));
    return KC_OK;
}

}  // namespace
}  // namespace kcapi

using namespace kcapi;

extern "C" {

kc_status kc_export_items(kc_handle h, kc_item16* items, uint64_t capacity, uint64_t* n_out) {
    kc_status s = device_result(h, "kc_export_items");
    if (s != KC_OK) return s;
    if (n_out) *n_out = h->n_result;
    if (!items) return KC_OK;
    if (capacity < h->n_result) return fail(KC_ERR_CAPACITY, "item capacity smaller than the result");
    const uint64_t n = h->n_result;
    if (n == 0) return KC_OK;
    cudaStream_t st = h->stream;
    const bool dev = is_device_ptr(items);
    if (dev && reinterpret_cast<uintptr_t>(items) % 16 != 0) return fail(KC_ERR_ARG, "device items must be 16-byte aligned");
    ulonglong2* out = reinterpret_cast<ulonglong2*>(items);
    if (!dev) KC_CUDA(kc::dev_alloc(&out, n * 16, st));
    kc::k_items16<<<kc::grid_of(n, 256, h->grid.sm_count * 8), 256, 0, st>>>(h->res_keys, h->res_vals, n,
                                                                             h->n_samples, out);
    h->launches += 1;
    KC_LAUNCHED("item export launch");
    if (!dev) {
        KC_CUDA(cudaMemcpyAsync(items, out, n * 16, cudaMemcpyDeviceToHost, st));
        cudaFreeAsync(out, st);
    }
    KC_CUDA(cudaStreamSynchronize(st));
    return KC_OK;
}

kc_status kc_spectrum(kc_handle h, uint32_t cap, uint64_t* hist) {
    kc_status s = device_result(h, "kc_spectrum");
    if (s != KC_OK) return s;
    if (cap < 1 || cap > KC_SPECTRUM_MAX_CAP || !hist) return fail(KC_ERR_ARG, "spectrum cap out of range or null hist");
    const uint64_t side = (uint64_t)cap + 1;
    const uint64_t n_bins = h->n_samples == 2 ? side * side : side;
    cudaStream_t st = h->stream;
    const bool dev = is_device_ptr(hist);
    uint64_t* out = hist;
    if (!dev) KC_CUDA(kc::dev_alloc(&out, n_bins * 8, st));
    KC_CUDA(cudaMemsetAsync(out, 0, n_bins * 8, st));
    if (h->n_result) {
        kc::k_spectrum<<<kc::grid_of(h->n_result, 256, h->grid.sm_count * 2), 256, 0, st>>>(
            h->res_vals, h->n_result, h->n_samples, cap, n_bins, reinterpret_cast<unsigned long long*>(out));
        h->launches += 1;
        KC_LAUNCHED("spectrum launch");
    }
    if (!dev) {
        KC_CUDA(cudaMemcpyAsync(hist, out, n_bins * 8, cudaMemcpyDeviceToHost, st));
        cudaFreeAsync(out, st);
    }
    KC_CUDA(cudaStreamSynchronize(st));
    return KC_OK;
}

// Build the stem items of the result on the device (kept until kc_reset).
static kc_status build_stems(kc_handle h) {
    cudaStream_t st = h->stream;
    const uint64_t n = h->n_result;
    const uint64_t cap = std::max<uint64_t>(1, 2 * n);
    uint64_t *rk = nullptr, *rv = nullptr, *sk = nullptr, *sv = nullptr, *starts = nullptr;
    kc::DevCounters* sctr = nullptr;
    auto release = [&]() {
        for (void* q : {(void*)rk, (void*)rv, (void*)sk, (void*)sv, (void*)starts, (void*)sctr})
            if (q) cudaFreeAsync(q, st);
    };
    cudaError_t e;
    if ((e = kc::dev_alloc(&rk, cap * 8, st)) != cudaSuccess || (e = kc::dev_alloc(&rv, cap * 8, st)) != cudaSuccess ||
        (e = kc::dev_alloc(&sk, cap * 8, st)) != cudaSuccess || (e = kc::dev_alloc(&sv, cap * 8, st)) != cudaSuccess ||
        (e = kc::dev_alloc(&sctr, sizeof(kc::DevCounters), st)) != cudaSuccess) {
        release();
        return cuda_fail(e, "cudaMallocAsync(stem records)");
    }
    auto run = [&]() -> kc_status {
        KC_CUDA(cudaMemsetAsync(sctr, 0, sizeof(kc::DevCounters), st));
        cudaEvent_t t0 = phase_begin(h);
        if (n)
            kc::k_stem_records<<<kc::grid_of(n, kc::kTileThreads, h->grid.sm_count * 8), kc::kTileThreads, 0, st>>>(
                h->res_keys, h->res_vals, n, h->k, rk, rv, sctr);
        phase_end(h, kStems, t0);
        h->launches += 1;
        KC_LAUNCHED("stem record launch");
        uint64_t n_rec = 0;
        KC_CUDA(cudaMemcpyAsync(&n_rec, &sctr->survivors, 8, cudaMemcpyDeviceToHost, st));
        KC_CUDA(cudaStreamSynchronize(st));
        if (n_rec > cap) {
            h->state = State::Poisoned;
            return fail(KC_ERR_INTERNAL, "stem records: more than two per key");
        }
        kc_status s = sort_pairs(h, rk, rv, n_rec, 2 * (h->k - 2) + 4, sctr, sk, sv, kStems);
        if (s != KC_OK) return s;
        KC_CUDA(kc::dev_alloc(&starts, std::max<uint64_t>(1, n_rec) * 8, st));
        uint64_t n_items = 0;
        t0 = phase_begin(h);
        s = compact_ordered(h, kc::StemStartPred{sk}, kc::IndexWrite{starts}, n_rec, &n_items);
        if (s != KC_OK) return s;
        KC_CUDA(kc::dev_alloc(&h->stem_items, std::max<uint64_t>(1, n_items) * sizeof(kc_stem_item), st));
        if (n_items)
            kc::k_stem_items<<<kc::grid_of(n_items, kc::kTileThreads, h->grid.sm_count * 8), kc::kTileThreads, 0, st>>>(
                sk, sv, n_rec, starts, n_items, h->n_samples, reinterpret_cast<uint64_t*>(h->stem_items));
        phase_end(h, kStems, t0);
        h->launches += 1;
        KC_LAUNCHED("stem item launch");
        KC_CUDA(cudaStreamSynchronize(st));
        phase_collect(h);
        h->n_stems = n_items;
        h->has_stems = true;
        return KC_OK;
    };
    kc_status s = run();
    if (s != KC_OK) {
        cudaStreamSynchronize(st);
        free_stems(h);
    }
    release();
    return s;
}

kc_status kc_export_stems(kc_handle h, kc_stem_item* items, uint64_t capacity, uint64_t* n_out) {
    kc_status s = device_result(h, "kc_export_stems");
    if (s != KC_OK) return s;
    if (h->k < 3) return fail(KC_ERR_STATE, "kc_export_stems needs k >= 3 (a stem is the middle k - 2 bases)");
    if (!h->has_stems && (s = build_stems(h)) != KC_OK) return s;
    if (n_out) *n_out = h->n_stems;
    if (!items) return KC_OK;
    if (capacity < h->n_stems) return fail(KC_ERR_CAPACITY, "item capacity smaller than the stem table");
    if (h->n_stems == 0) return KC_OK;
    KC_CUDA(cudaMemcpyAsync(items, h->stem_items, h->n_stems * sizeof(kc_stem_item), cudaMemcpyDefault, h->stream));
    KC_CUDA(cudaStreamSynchronize(h->stream));
    return KC_OK;
}

kc_status kc_filter_select(kc_handle h, const kc_filter_spec* spec, uint64_t* n_selected) {
    kc_status s = device_result(h, "kc_filter_select");
    if (s != KC_OK) return s;
    if (h->n_samples != 2) return fail(KC_ERR_STATE, "kc_filter_select needs a two-sample (normal/tumoral) job");
    if (!spec || spec->tumor < 0 || spec->tumor > 1) return fail(KC_ERR_ARG, "filter spec: tumor must be 0 or 1");
    free_selection(h);
    cudaStream_t st = h->stream;
    const uint64_t n = h->n_result;
    kc::SelSpec ss{spec->tumor, spec->min_tumor, spec->max_normal, spec->ratio};
    kc::SelectPred pred{h->res_vals, ss};
    uint64_t kept = 0;
    cudaEvent_t t0 = phase_begin(h);
    // count first, then allocate exactly and write
    Tiles tiles;
    cudaError_t e = tiles.take(n, st);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMallocAsync(compaction tiles)");
    kc::k_tile_count<kc::SelectPred><<<(unsigned)tiles.n, kc::kTileThreads, 0, st>>>(pred, n, tiles.counts);
    if ((e = kc::launch_scan(tiles.counts, tiles.n, tiles.starts, tiles.cursor, st)) != cudaSuccess) {
        tiles.leave(st);
        return cuda_fail(e, "tile scan");
    }
    h->launches += 2;
    KC_LAUNCHED("selection count launches");
    KC_CUDA(cudaMemcpyAsync(&kept, tiles.starts + tiles.n, 8, cudaMemcpyDeviceToHost, st));
    KC_CUDA(cudaStreamSynchronize(st));
    const uint64_t cap = std::max<uint64_t>(1, kept);
    // buckets of four slots for both orientations of every key, at most a
    // quarter full: about 2 % of the buckets are full and make a miss probe on
    int lb = 8;
    while ((1ull << lb) < 2 * kept) ++lb;
    if (lb > 32) {
        tiles.leave(st);
        return fail(KC_ERR_CAPACITY, "selection larger than 2^31 keys");
    }
    const uint64_t n_buckets = 1ull << lb;
    const bool pre = 2 * kept <= kc::kPreMaxEntries;
    const uint64_t table_bytes = n_buckets * kSelBucketBytes + (pre ? kc::kPreWords * 4ull : 0);
    if ((e = kc::dev_alloc(&h->sel_keys, cap * 8, st)) != cudaSuccess ||
        (e = kc::dev_alloc(&h->sel_vals, cap * 8, st)) != cudaSuccess ||
        (e = kc::dev_alloc(&h->sel_table, table_bytes, st)) != cudaSuccess) {
        tiles.leave(st);
        free_selection(h);
        return cuda_fail(e, "cudaMallocAsync(selection)");
    }
    h->sel_buckets_log2 = lb;
    h->sel_pre = pre;
    KC_CUDA(cudaMemsetAsync(h->sel_table, 0, n_buckets * 16, st));  // fingerprints: all slots free
    if (pre)
        KC_CUDA(cudaMemsetAsync(reinterpret_cast<char*>(h->sel_table) + n_buckets * kSelBucketBytes, 0,
                                kc::kPreWords * 4ull, st));
    if (kept) {
        kc::k_tile_write<kc::SelectPred, kc::SelectWrite><<<(unsigned)tiles.n, kc::kTileThreads, 0, st>>>(
            pred, kc::SelectWrite{h->res_keys, h->res_vals, h->sel_keys, h->sel_vals}, n, tiles.starts);
        kc::k_sel_insert<<<kc::grid_of(kept, 256, h->grid.sm_count * 8), 256, 0, st>>>(
            h->sel_keys, kept, sel_table_of(h), h->params(0), h->ctr);
        h->launches += 2;
        KC_LAUNCHED("selection table launches");
    }
    tiles.leave(st);
    phase_end(h, kFilterSelect, t0);
    s = read_counters(h);
    if (s != KC_OK) return s;
    phase_collect(h);
    if (h->host_ctr.err & kc::DERR_INTERNAL) {
        h->state = State::Poisoned;
        return fail(KC_ERR_INTERNAL, "selection table: no free slot");
    }
    h->n_sel = kept;
    h->has_selection = true;
    if (n_selected) *n_selected = kept;
    return KC_OK;
}

kc_status kc_filter_keys(kc_handle h, uint64_t* keys, uint32_t* counts, uint64_t capacity, uint64_t* n_out) {
    kc_status s = check_open(h);
    if (s != KC_OK) return s;
    if (!h->has_selection) return fail(KC_ERR_STATE, "kc_filter_keys before kc_filter_select");
    if (n_out) *n_out = h->n_sel;
    if (!keys) return KC_OK;
    if (capacity < h->n_sel) return fail(KC_ERR_CAPACITY, "key capacity smaller than the selection");
    if (h->n_sel == 0) return KC_OK;
    KC_CUDA(cudaMemcpyAsync(keys, h->sel_keys, h->n_sel * 8, cudaMemcpyDefault, h->stream));
    if (counts) KC_CUDA(cudaMemcpyAsync(counts, h->sel_vals, h->n_sel * 8, cudaMemcpyDefault, h->stream));
    KC_CUDA(cudaStreamSynchronize(h->stream));
    return KC_OK;
}

kc_status kc_filter_reads(kc_handle h, const uint64_t* packed_reads, const uint64_t* offsets, const uint64_t* n_mask,
                          uint64_t n_reads, uint32_t* hits, uint64_t* candidates, uint64_t* n_candidates) {
    kc_status s = check_open(h);
    if (s != KC_OK) return s;
    if (!h->has_selection) return fail(KC_ERR_STATE, "kc_filter_reads before kc_filter_select");
    if (n_candidates) *n_candidates = 0;
    if (n_reads == 0) return KC_OK;
    if (!offsets || !hits) return fail(KC_ERR_ARG, "offsets or hits is null");
    cudaStream_t st = h->stream;

    const bool off_dev = is_device_ptr(offsets);
    uint64_t b0, b1;
    if (off_dev) {
        KC_CUDA(pinned_words(h));
        KC_CUDA(cudaMemcpyAsync(h->pinned + 1, offsets, 8, cudaMemcpyDeviceToHost, st));
        KC_CUDA(cudaMemcpyAsync(h->pinned + 2, offsets + n_reads, 8, cudaMemcpyDeviceToHost, st));
        KC_CUDA(cudaStreamSynchronize(st));
        b0 = h->pinned[1];
        b1 = h->pinned[2];
    } else {
        b0 = offsets[0];
        b1 = offsets[n_reads];
        for (uint64_t r = 0; r < n_reads; ++r)
            if (offsets[r + 1] < offsets[r]) return fail(KC_ERR_ARG, "read offsets decrease");
    }
    if (b1 < b0) return fail(KC_ERR_ARG, "read offsets decrease");
    if (b1 > b0 && (!packed_reads || !n_mask)) return fail(KC_ERR_ARG, "packed_reads or n_mask is null");
    if (n_reads >= (1ull << 32)) return fail(KC_ERR_ARG, "at most 2^32 - 1 reads per kc_filter_reads call");

    const bool hits_dev = is_device_ptr(hits);
    const bool cand_dev = candidates && is_device_ptr(candidates);
    const uint64_t B = (b0 / 64) * 64;
    const uint64_t n_local = b1 - B;
    const uint64_t n_units = std::max<uint64_t>(1, (n_local + 63) / 64);
    const bool any = b1 > b0;  // else no word is read
    const uint64_t n_pwords_src = any ? (n_local + 31) / 32 : 0;
    const uint64_t n_pwords = 2 * n_units + 2;

    // Device arrays are read where they are (the packed words where 16-byte
    // loads can reach them), host ones copied; everything of this call lies in
    // one block.
    const uint64_t* const src_pw = any ? packed_reads + B / 32 : nullptr;
    const bool own_pw = !any || !is_local_device_ptr(packed_reads, h->device) || reinterpret_cast<uintptr_t>(src_pw) % 16 != 0;
    const bool own_nm = !any || !words_in_place(n_mask, h->device);
    const bool own_off = !words_in_place(offsets, h->device);
    const bool own_cand = candidates && !cand_dev;
    char* block = nullptr;
    uint64_t* hmask = nullptr;  // pinned words the call's small readbacks land in
    Tiles tiles;
    auto release = [&]() {
        if (block) cudaFreeAsync(block, st);
        tiles.leave(st);
    };
    const size_t bytes = (own_pw ? n_pwords * 8 : 0) + n_units * 8 * (3 + (own_nm ? 1 : 0)) + (own_off ? (n_reads + 1) * 8 : 0) +
                         (own_cand ? n_reads * 8 : 0) + (hits_dev ? 0 : n_reads * 4) + sizeof(kc::DevCounters) + 16;
    cudaError_t e = cudaSuccess;
    if ((e = kc::dev_alloc(&block, bytes, st)) != cudaSuccess || (e = tiles.take(n_reads, st)) != cudaSuccess ||
        (e = pinned_words(h)) != cudaSuccess) {
        release();
        return cuda_fail(e, "cudaMallocAsync(filter reads)");
    }
    hmask = h->pinned;
    char* q = block;
    const auto part = [&](size_t n) {
        char* p = q;
        q += n;
        return p;
    };
    kc::DevCounters* fctr = reinterpret_cast<kc::DevCounters*>(part(sizeof(kc::DevCounters)));
    uint64_t* bd = reinterpret_cast<uint64_t*>(part(n_units * 8));  // (cleared with the counters)
    uint64_t* pw = own_pw ? reinterpret_cast<uint64_t*>(part(n_pwords * 8 + (n_units % 2 ? 8 : 0))) : nullptr;
    if (pw && reinterpret_cast<uintptr_t>(pw) % 16 != 0) ++pw;  // 16-byte loads
    uint64_t* vw = reinterpret_cast<uint64_t*>(part(n_units * 8));
    uint64_t* hitmask = reinterpret_cast<uint64_t*>(part(n_units * 8));
    uint64_t* nm = own_nm ? reinterpret_cast<uint64_t*>(part(n_units * 8)) : nullptr;
    uint64_t* doff = own_off ? reinterpret_cast<uint64_t*>(part((n_reads + 1) * 8)) : nullptr;
    uint64_t* dcand = own_cand ? reinterpret_cast<uint64_t*>(part(n_reads * 8)) : candidates;
    uint32_t* dhits = hits_dev ? hits : reinterpret_cast<uint32_t*>(part(n_reads * 4));
    auto run = [&]() -> kc_status {
        KC_CUDA(cudaMemsetAsync(fctr, 0, sizeof(kc::DevCounters) + n_units * 8, st));
        if (own_pw) {
            KC_CUDA(cudaMemsetAsync(pw + n_pwords_src, 0, (n_pwords - n_pwords_src) * 8, st));
            if (n_pwords_src) KC_CUDA(cudaMemcpyAsync(pw, src_pw, n_pwords_src * 8, cudaMemcpyDefault, st));
        }
        if (own_nm) {
            if (any) KC_CUDA(cudaMemcpyAsync(nm, n_mask + B / 64, n_units * 8, cudaMemcpyDefault, st));
            else KC_CUDA(cudaMemsetAsync(nm, 0, n_units * 8, st));
        }
        if (own_off) KC_CUDA(cudaMemcpyAsync(doff, offsets, (n_reads + 1) * 8, cudaMemcpyDefault, st));
        const uint64_t* off_in = own_off ? doff : offsets;
        const uint64_t* pw_in = own_pw ? pw : src_pw;
        const uint64_t n_words = own_pw ? n_pwords : n_pwords_src;
        kc::launch_mark_read_starts(off_in, n_reads, B, n_local, bd, fctr, st);
        kc::launch_build_valid(own_nm ? nm : n_mask + B / 64, bd, n_units, b0 - B, n_local, h->k, vw, fctr, h->grid, st);
        const kc::SelTable T = sel_table_of(h);
        const auto rescan = [&](auto kern, unsigned grid, int threads, size_t smem) {
            cudaEvent_t t0 = phase_begin(h);
            kern<<<grid, threads, smem, st>>>(pw_in, n_words, vw, n_units, h->params(0), T, hitmask, fctr);
            phase_end(h, kFilterReads, t0);
        };
        // k = 31 (the longest k, the one the paper's configurations use): constant shifts
        if (T.pre) {
            KC_CUDA(kc::filter_pre_smem_attr());
            const unsigned grid = kc::grid_of(n_units, kc::kFilterThreadsPre, (unsigned)h->grid.sm_count);
            if (h->k == 31) rescan(kc::k_filter_hits<true, 31>, grid, kc::kFilterThreadsPre, kc::kPreWords * 4);
            else rescan(kc::k_filter_hits<true, 0>, grid, kc::kFilterThreadsPre, kc::kPreWords * 4);
        } else {
            const unsigned grid = kc::grid_of(n_units, kc::kFilterThreads,
                                              (unsigned)(h->grid.sm_count * kc::filter_blocks_per_sm()));
            if (h->k == 31) rescan(kc::k_filter_hits<false, 31>, grid, kc::kFilterThreads, 0);
            else rescan(kc::k_filter_hits<false, 0>, grid, kc::kFilterThreads, 0);
        }
        kc::k_read_hits<<<(unsigned)tiles.n, kc::kReadThreads, 0, st>>>(off_in, n_reads, B, n_units, hitmask, dhits, tiles.counts);
        h->launches += 4;
        KC_LAUNCHED("filter rescan launches");
        KC_CUDA(kc::launch_scan(tiles.counts, tiles.n, tiles.starts, tiles.cursor, st));
        h->launches += 1;
        if (candidates) {
            kc::k_tile_write<kc::HitPred, kc::IndexWrite><<<(unsigned)tiles.n, kc::kTileThreads, 0, st>>>(
                kc::HitPred{dhits}, kc::IndexWrite{dcand}, n_reads, tiles.starts);
            h->launches += 1;
        }
        KC_LAUNCHED("candidate list launches");
        // one readback: windows, hits and error bits, the number of candidates
        KC_CUDA(cudaMemcpyAsync(hmask, fctr, 2 * sizeof(uint64_t), cudaMemcpyDeviceToHost, st));
        KC_CUDA(cudaMemcpyAsync(hmask + 2, &fctr->err, sizeof(unsigned), cudaMemcpyDeviceToHost, st));
        KC_CUDA(cudaMemcpyAsync(hmask + 3, tiles.starts + tiles.n, sizeof(uint64_t), cudaMemcpyDeviceToHost, st));
        KC_CUDA(cudaStreamSynchronize(st));
        const unsigned err = *reinterpret_cast<unsigned*>(hmask + 2);
        const uint64_t n_cand = hmask[3];
        if (err & kc::DERR_OFFSETS) return fail(KC_ERR_ARG, "read offsets decrease or start before the first word");
        h->filter_windows += hmask[0];
        h->filter_hits += hmask[1];
        if (!hits_dev) KC_CUDA(cudaMemcpyAsync(hits, dhits, n_reads * 4, cudaMemcpyDeviceToHost, st));
        if (own_cand && n_cand) KC_CUDA(cudaMemcpyAsync(candidates, dcand, n_cand * 8, cudaMemcpyDeviceToHost, st));
        if (!hits_dev || (own_cand && n_cand)) KC_CUDA(cudaStreamSynchronize(st));
        phase_collect(h);
        if (n_candidates) *n_candidates = n_cand;
        return KC_OK;
    };
    s = run();
    if (s != KC_OK) cudaStreamSynchronize(st);  // nothing in flight may touch the caller's arrays after return
    release();
    return s;
}

}  // extern "C"
