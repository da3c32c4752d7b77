// Device-side building blocks of the k-mer counting path (sm_103a).
//
// Reads are kept on the device as 2-bit codes, 32 bases per 64-bit word,
// first base in the most significant bits, plus one "valid window start" bit
// per base (V).  A window of k <= 31 bases starting inside a 64-base unit
// never reaches past the first word of the next unit, so a lane that owns one
// unit (two packed words, one V word) only needs the next lane's first word,
// which it gets with a warp shuffle.
#pragma once

#include <cstdint>

namespace kc {

struct __align__(16) Slot {
    unsigned long long key1;  // key + 1; 0 marks an empty slot
    unsigned int cnt[2];      // per-sample counts (cnt[1] unused with one sample)
};
static_assert(sizeof(Slot) == 16, "a table item is 8 bytes of key and 8 of counts (Section III-D)");

// Device-wide counters and error bits of one job.
struct DevCounters {
    unsigned long long windows;     // valid windows (V bits) of all batches
    unsigned long long candidates;  // windows whose filter bits were all set already
    unsigned long long claimed;     // keys inserted into the table
    unsigned long long survivors;   // keys written by the compaction
    unsigned int err;               // DERR_* bits
    unsigned int split_parts;       // partitions counted in sub-ranges
    unsigned int split_hint;        // split level the job's partitions start at
    unsigned int pad0;
    unsigned long long kept;        // windows kept by hash-range restricted extractions
    unsigned int pad[2];
};
static_assert(sizeof(DevCounters) == 64, "device counters: 64 bytes");

enum : unsigned int {
    DERR_TABLE_FULL = 1u,      // a probe sequence visited every slot
    DERR_COUNT_OVERFLOW = 2u,  // a per-sample count passed 2^32 - 1
    DERR_OFFSETS = 4u,         // decreasing read offsets
    DERR_SORT_BUCKET = 8u,     // a sort bucket exceeded the shared-memory tile
    DERR_INTERNAL = 16u,       // a self-check failed (index out of range)
    DERR_SORT_MEDIUM = 32u,    // a sort bucket exceeded one warp's registers
    DERR_SORT_BIG = 64u,       // a sort bucket is left to the second warp sort (not an error)
};

// Parameters shared by the extraction passes.
struct PassParams {
    int k;
    int rc_shift;            // 64 - 2k
    unsigned long long kmask;  // 2k low bits
    int bloom_shift;         // 64 - log2(words)
    int n_hashes;
    int table_shift;         // 64 - log2(slots)
    unsigned long long table_mask;
    int all_candidates;      // min_count <= 1: every window goes to the table
    int sample;
    // Hash range kept by the partitioned extraction: a window is kept iff
    // h_lo <= h <= h_hi (0 and ~0: every window).  It restricts a handle to the
    // keys it owns, or to one hash range of an out-of-core job at a time.
    unsigned long long h_lo, h_hi;
};

// SplitMix64 output function (Steele, Lea & Flood, OOPSLA 2014): golden-ratio
// increment, then two xor-shift-multiply rounds and a closing xor-shift.
__device__ __forceinline__ uint64_t mixer64(uint64_t x) {
    uint64_t z = x + 0x9e3779b97f4a7c15ull;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

// Inverse of mixer64: undo the closing xor-shift, the two multiplies (by the
// multipliers' inverses modulo 2^64) and xor-shifts, then the increment.
// x ^= x >> s is undone by x ^ (x >> s) ^ (x >> 2s) ^ ... while the shift fits.
__device__ __forceinline__ uint64_t unmixer64(uint64_t z) {
    z ^= (z >> 31) ^ (z >> 62);
    z *= 0x319642b2d24d8ec3ull;  // inverse of 0x94d049bb133111eb
    z ^= (z >> 27) ^ (z >> 54);
    z *= 0x96de1b173f119089ull;  // inverse of 0xbf58476d1ce4e5b9
    z ^= (z >> 30) ^ (z >> 60);
    return z - 0x9e3779b97f4a7c15ull;
}
static_assert(0x319642b2d24d8ec3ull * 0x94d049bb133111ebull == 1ull, "multiplier inverse");
static_assert(0x96de1b173f119089ull * 0xbf58476d1ce4e5b9ull == 1ull, "multiplier inverse");

// Reverse the order of the 32 two-bit groups of x.
__device__ __forceinline__ uint64_t reverse_pairs(uint64_t x) {
    x = __brevll(x);
    return ((x >> 1) & 0x5555555555555555ull) | ((x & 0x5555555555555555ull) << 1);
}

// Forward 2k-bit code of the window starting at base j (0..63) of a unit whose
// words are w0, w1 and the following word w2.
__device__ __forceinline__ uint64_t window_code(uint64_t w0, uint64_t w1, uint64_t w2, int j, int rc_shift) {
    const bool second = j >= 32;
    const uint64_t hi = second ? w1 : w0;
    const uint64_t lo = second ? w2 : w1;
    const int off = 2 * (j & 31);
    const uint64_t x = off ? (hi << off) | (lo >> (64 - off)) : hi;
    return x >> rc_shift;
}

// Canonical key: the smaller of the forward code and the code of the reverse
// complement (complement = code ^ 3, then reverse the base order).
__device__ __forceinline__ uint64_t canonical_key(uint64_t fwd, const PassParams& p) {
    const uint64_t rc = reverse_pairs(fwd ^ p.kmask) >> p.rc_shift;
    return fwd < rc ? fwd : rc;
}

// Codes of eight windows at a time, cut out of the unit's bases at constant
// places: f holds the bases from the first of the eight windows on, as 32-bit
// words, first base on top.  Two funnel shifts and a mask a window (K = k at
// compile time; K = 0: one 64-bit shift by rc_shift more), where the rolling
// code takes nine operations.
struct WindowWords {
    uint32_t f[6];
};

// The reverse complements of the same windows: r holds the reverse complement
// of all bases from the first of the eight windows on, its lowest word first,
// so that window J's code begins at bit 2 J.
struct ReverseWords {
    uint32_t r[6];
};

__device__ __forceinline__ ReverseWords reverse_words(uint64_t w0, uint64_t w1, uint64_t w2) {
    const uint64_t a = reverse_pairs(~w0), b = reverse_pairs(~w1), c = reverse_pairs(~w2);
    return ReverseWords{{(uint32_t)a, (uint32_t)(a >> 32), (uint32_t)b, (uint32_t)(b >> 32), (uint32_t)c,
                         (uint32_t)(c >> 32)}};
}

__device__ __forceinline__ void next_windows(ReverseWords& w) {
#pragma unroll
    for (int i = 0; i < 5; ++i) w.r[i] = __funnelshift_r(w.r[i], w.r[i + 1], 16);
    w.r[5] >>= 16;
}

template <int K, int J>
__device__ __forceinline__ uint64_t reverse_code(const ReverseWords& w, uint64_t kmask) {
    uint32_t lo, hi;
    if constexpr (J == 0) {
        lo = w.r[0];
        hi = w.r[1];
    } else {
        lo = __funnelshift_r(w.r[0], w.r[1], 2 * J);
        hi = __funnelshift_r(w.r[1], w.r[2], 2 * J);
    }
    if constexpr (K > 16) return ((uint64_t)(hi & (0xffffffffu >> (64 - 2 * K))) << 32) | lo;
    else return (((uint64_t)hi << 32) | lo) & kmask;
}

__device__ __forceinline__ WindowWords window_words(uint64_t w0, uint64_t w1, uint64_t w2) {
    return WindowWords{{(uint32_t)(w0 >> 32), (uint32_t)w0, (uint32_t)(w1 >> 32), (uint32_t)w1, (uint32_t)(w2 >> 32),
                        (uint32_t)w2}};
}

__device__ __forceinline__ void next_windows(WindowWords& w) {
#pragma unroll
    for (int i = 0; i < 5; ++i) w.f[i] = __funnelshift_l(w.f[i + 1], w.f[i], 16);
    w.f[5] <<= 16;
}

// Window J (0..7) of the eight.
template <int K, int J>
__device__ __forceinline__ uint64_t forward_code(const WindowWords& w, int rc_shift) {
    constexpr int drop = K > 16 ? 64 - 2 * K : 0;  // bits after the window in the 64 cut out
    constexpr int off = 2 * J - drop;
    uint32_t hi, lo;
    if constexpr (off > 0) {
        hi = __funnelshift_l(w.f[1], w.f[0], off);
        lo = __funnelshift_l(w.f[2], w.f[1], off);
    } else if constexpr (off == 0) {
        hi = w.f[0];
        lo = w.f[1];
    } else {
        hi = w.f[0] >> -off;
        lo = __funnelshift_r(w.f[1], w.f[0], -off);
    }
    if constexpr (K > 16) return ((uint64_t)(hi & (0xffffffffu >> drop)) << 32) | lo;
    else return (((uint64_t)hi << 32) | lo) >> rc_shift;
}

// shl.b32 clamps its shift amount at 32: x << b is 0 for b >= 32.
__device__ __forceinline__ uint32_t shl_clamped(uint32_t x, uint32_t b) {
    uint32_t r;
    asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(b));
    return r;
}

// Bits of one key in its filter word: bit (g >> 6i) & 63 for i < n_hashes,
// assembled in two 32-bit halves (bit b >= 32 is bit b ^ 32 of the high half).
template <int NH>
__device__ __forceinline__ uint64_t bloom_pattern_n(uint64_t g) {
    uint32_t lo = 0, hi = 0;
#pragma unroll
    for (int i = 0; i < NH; ++i) {
        const uint32_t bit = (uint32_t)(g >> (6 * i)) & 63u;
        lo |= shl_clamped(1u, bit);
        hi |= shl_clamped(1u, bit ^ 32u);
    }
    return ((uint64_t)hi << 32) | lo;
}

__device__ __forceinline__ uint64_t bloom_pattern(uint64_t g, int n_hashes) {
    uint64_t pat = 0;
#pragma unroll
    for (int i = 0; i < 10; ++i)
        if (i < n_hashes) pat |= 1ull << ((g >> (6 * i)) & 63);
    return pat;
}

// Load the unit's words; lanes of a warp hold consecutive units, so the word
// after the unit comes from the next lane (the last lane loads it itself).
// The packed buffer is padded to 2 * n_units + 2 zero-filled words, so every
// unit has both of its words and a successor word in bounds.
struct UnitWords {
    uint64_t w0, w1, w2, v;
};

// Units at or beyond u_end are inactive (zero words); the last active lane
// loads its successor word itself, since that unit may belong to another
// lane group or CTA.  All 32 lanes must call this together.
// n_words: the words there are at pw (a caller's array read in place, without
// the padding); words past them read as zero.
__device__ __forceinline__ UnitWords load_unit(const uint64_t* __restrict__ pw, const uint64_t* __restrict__ vw,
                                               uint64_t u, uint64_t u_end, int lane, uint64_t n_words = ~0ull) {
    UnitWords r{0, 0, 0, 0};
    const bool in = u < u_end;
    if (in) {
        r.v = __ldg(vw + u);
        if (2 * u + 1 < n_words) {
            const ulonglong2 p = __ldg(reinterpret_cast<const ulonglong2*>(pw) + u);
            r.w0 = p.x;
            r.w1 = p.y;
        } else if (2 * u < n_words) {
            r.w0 = __ldg(pw + 2 * u);
        }
    }
    r.w2 = __shfl_down_sync(0xffffffffu, r.w0, 1);
    if (in && (lane == 31 || u + 1 >= u_end)) r.w2 = 2 * u + 2 < n_words ? __ldg(pw + 2 * u + 2) : 0ull;
    return r;
}

// Part `part` of 2^lp of unit u: the windows that start in its 64 >> lp bases,
// moved to the front.  n_words as above.
__device__ __forceinline__ UnitWords load_part(const uint64_t* __restrict__ pw, const uint64_t* __restrict__ vw,
                                               uint64_t u, int part, int lp, uint64_t n_words = ~0ull) {
    UnitWords r{0, 0, 0, __ldg(vw + u)};
    if (2 * u + 1 < n_words) {
        const ulonglong2 p = __ldg(reinterpret_cast<const ulonglong2*>(pw) + u);
        r.w0 = p.x;
        r.w1 = p.y;
        if (2 * u + 2 < n_words) r.w2 = __ldg(pw + 2 * u + 2);
    } else if (2 * u < n_words) {
        r.w0 = __ldg(pw + 2 * u);
    }
    int skip = part << (6 - lp);  // bases
    r.v = (r.v << skip) & (~0ull << (64 - (64 >> lp)));
    if (skip >= 32) {
        r.w0 = r.w1;
        r.w1 = r.w2;
        r.w2 = 0;
        skip -= 32;
    }
    if (skip) {
        r.w0 = r.w0 << 2 * skip | r.w1 >> (64 - 2 * skip);
        r.w1 = r.w1 << 2 * skip | r.w2 >> (64 - 2 * skip);
        r.w2 <<= 2 * skip;
    }
    return r;
}

// log2 of the parts, at most eight a unit, that give n units' lanes something to
// do without passing `lanes`.
__device__ __forceinline__ int parts_log2(uint64_t n, uint64_t lanes) {
    int lp = 0;
    while (lp < 3 && n << (lp + 1) <= lanes) ++lp;
    return lp;
}

// Insert key (stored as key + 1) by linear probing.  Returns 1 if this call
// claimed a new slot.  A probe sequence that wraps the whole table sets
// DERR_TABLE_FULL and gives up.
__device__ __forceinline__ int table_claim(Slot* __restrict__ table, uint64_t mask, uint64_t s, uint64_t stored,
                                           DevCounters* ctr) {
    for (uint64_t i = 0; i <= mask; ++i) {
        const unsigned long long cur = __ldcg(&table[s].key1);
        if (cur == stored) return 0;
        if (cur == 0ull) {
            const unsigned long long prev = atomicCAS(&table[s].key1, 0ull, (unsigned long long)stored);
            if (prev == 0ull) return 1;
            if (prev == stored) return 0;
        }
        s = (s + 1) & mask;
    }
    atomicOr(&ctr->err, DERR_TABLE_FULL);
    return 0;
}

// Insert key (stored as key + 1) and add one occurrence to it, from slot s on,
// whose key1 the caller has read as cur.  Returns 1 if this call claimed a new
// slot.
__device__ __forceinline__ int table_add(Slot* __restrict__ table, uint64_t mask, uint64_t s, uint64_t stored,
                                         unsigned long long cur, int sample, DevCounters* ctr) {
    for (uint64_t i = 0;; ) {
        int claimed = 0;
        if (cur == 0ull) {
            cur = atomicCAS(&table[s].key1, 0ull, (unsigned long long)stored);
            claimed = cur == 0ull;
        }
        if (claimed || cur == stored) {
            if (atomicAdd(&table[s].cnt[sample], 1u) == 0xffffffffu) atomicOr(&ctr->err, DERR_COUNT_OVERFLOW);
            return claimed;
        }
        if (++i > mask) break;
        s = (s + 1) & mask;
        cur = __ldcg(&table[s].key1);
    }
    atomicOr(&ctr->err, DERR_TABLE_FULL);
    return 0;
}

// Add one occurrence of key to its slot if the key is in the table.
__device__ __forceinline__ void table_count(Slot* __restrict__ table, uint64_t mask, uint64_t s, uint64_t stored,
                                            int sample, DevCounters* ctr) {
    for (uint64_t i = 0; i <= mask; ++i) {
        const unsigned long long cur = __ldcg(&table[s].key1);
        if (cur == stored) {
            const unsigned int old = atomicAdd(&table[s].cnt[sample], 1u);
            if (old == 0xffffffffu) atomicOr(&ctr->err, DERR_COUNT_OVERFLOW);
            return;
        }
        if (cur == 0ull) return;
        s = (s + 1) & mask;
    }
}

// Warp-per-bucket sort: the bucket's keys sit in registers, R per lane
// (element r*32 + lane), padded with ~0 keys; a bitonic network runs with
// register compare-exchanges for strides >= 32 and shuffles below.
template <int R>
__device__ __forceinline__ void warp_bitonic(uint64_t (&k)[R], uint64_t (&v)[R], int lane) {
#pragma unroll
    for (int size = 2; size <= 32 * R; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            if (stride >= 32) {
                const int rs = stride >> 5;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    if ((r & rs) == 0) {  // compile-time: pairs within the lane
                        const int q = r | rs;
                        const bool asc = (((r << 5) | lane) & size) == 0;
                        const bool sw = (k[r] > k[q]) == asc;  // selects, no branch: lanes stay converged
                        const uint64_t ka = k[r], kb = k[q], va = v[r], vb = v[q];
                        k[r] = sw ? kb : ka;
                        k[q] = sw ? ka : kb;
                        v[r] = sw ? vb : va;
                        v[q] = sw ? va : vb;
                    }
                }
            } else {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int i = (r << 5) | lane;
                    const uint64_t ok = __shfl_xor_sync(0xffffffffu, k[r], stride);
                    const uint64_t ov = __shfl_xor_sync(0xffffffffu, v[r], stride);
                    const bool asc = (i & size) == 0;
                    const bool lower = (i & stride) == 0;
                    // keep the smaller key when this lane's end of the pair should hold it
                    const bool want_min = lower == asc;
                    const bool take_other = want_min ? ok < k[r] : ok > k[r];
                    k[r] = take_other ? ok : k[r];
                    v[r] = take_other ? ov : v[r];
                }
            }
        }
    }
}

template <int R>
__device__ __forceinline__ void warp_sort_bucket(uint64_t* __restrict__ keys, uint64_t* __restrict__ vals,
                                                 uint64_t lo, int n, int lane) {
    uint64_t k[R], v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = (r << 5) | lane;
        k[r] = i < n ? keys[lo + i] : ~0ull;
        v[r] = i < n ? vals[lo + i] : 0ull;
    }
    warp_bitonic<R>(k, v, lane);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = (r << 5) | lane;
        if (i < n) {
            keys[lo + i] = k[r];
            vals[lo + i] = v[r];
        }
    }
}

// Bucket of a key among 2^bits buckets in key order.  Canonical keys, the
// smaller of two orientations, are not uniform: with x the key as a fraction
// of the key space their density is 2 (1 - x), so plain key prefixes give
// buckets from twice the mean down to none.  even: the buckets are equal parts
// of the distribution function x (2 - x), from the key's top 32 bits (the
// floor of x^2 grows by at most 2 a step, so the map never decreases).
__device__ __forceinline__ uint32_t key_bucket(uint64_t key, int key_bits, int bits, bool even) {
    if (!even) return (uint32_t)(key >> (key_bits - bits));
    const uint32_t x = (uint32_t)(key >> (key_bits - 32));
    const uint64_t y = 2ull * x - __umulhi(x, x);
    return (uint32_t)(y >> 32 ? 0xffffffffull : y) >> (32 - bits);
}
// The map needs the 32 bits; one bucket needs no map.
__host__ __device__ __forceinline__ bool even_buckets(int key_bits, int bits) {
    return key_bits >= 32 && bits >= 1;
}

// Exclusive scan of n counters into starts (and starts[n], the total) and
// cursor, in one launch: each CTA takes the next tile by ticket, adds it up,
// publishes the sum and looks back over the tiles before it, 32 at a time,
// until one has published its whole prefix (Merrill and Garland's decoupled
// look-back).  A tile waits only for tiles of smaller tickets, whose CTAs run
// already; the wait is bounded all the same, and a tile that gives up adds the
// counters before it itself.  state, a word per tile, and ticket are zero
// before.
constexpr int kScanThreads = 256;
constexpr uint64_t kScanTile = 4 * kScanThreads;
constexpr int kScanPolls = 1 << 22;
__device__ __forceinline__ void scan_lookback(const uint32_t* __restrict__ hist, uint64_t n,
                                              uint64_t* __restrict__ starts, uint64_t* __restrict__ cursor,
                                              unsigned long long* state, unsigned long long* ticket) {
    constexpr unsigned long long kSum = 1ull << 62, kPrefix = 2ull << 62, kValue = kSum - 1;
    constexpr int nw = kScanThreads / 32;
    __shared__ unsigned long long s_w[nw];
    __shared__ unsigned long long s_prefix, s_tile;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1ull);
    __syncthreads();
    const uint64_t tile = s_tile;
    if (tile * kScanTile >= n) return;
    const uint64_t i0 = tile * kScanTile + 4 * threadIdx.x;
    const bool wide = i0 + 4 <= n && !((reinterpret_cast<uintptr_t>(hist) | reinterpret_cast<uintptr_t>(starts) |
                                        reinterpret_cast<uintptr_t>(cursor)) & 15u);
    uint32_t c[4];
    if (wide) {
        const uint4 q = *reinterpret_cast<const uint4*>(hist + i0);
        c[0] = q.x, c[1] = q.y, c[2] = q.z, c[3] = q.w;
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) c[j] = i0 + j < n ? hist[i0 + j] : 0u;
    }
    const unsigned long long sum = (unsigned long long)c[0] + c[1] + c[2] + c[3];
    unsigned long long incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) s_w[wid] = incl;
    __syncthreads();
    unsigned long long before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < nw; ++w) {
        if (w < wid) before += s_w[w];
        total += s_w[w];
    }
    volatile unsigned long long* const st = state;
    if (wid == 0) {
        if (lane == 0) st[tile] = (tile ? kSum : kPrefix) | total;
        unsigned long long prefix = 0;
        for (uint64_t at = tile; at > 0;) {  // tiles [0, at) are still to be added
            unsigned long long v = kPrefix;  // before the first tile: nothing
            for (int polls = 0; polls < kScanPolls; ++polls) {
                if ((uint64_t)lane < at) v = st[at - 1 - lane];
                if (__all_sync(0xffffffffu, v >> 62)) break;
            }
            if (__any_sync(0xffffffffu, !(v >> 62))) {
                prefix = 0;
                for (uint64_t i = lane; i < tile * kScanTile; i += 32) prefix += hist[i];
#pragma unroll
                for (int o = 16; o; o >>= 1) prefix += __shfl_xor_sync(0xffffffffu, prefix, o);
                break;
            }
            const unsigned whole = __ballot_sync(0xffffffffu, v >> 63);
            const int last = whole ? __ffs(whole) - 1 : 31;
            unsigned long long x = lane <= last ? v & kValue : 0ull;
#pragma unroll
            for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            prefix += x;
            if (whole) break;
            at -= 32;  // every lane had a tile
        }
        if (lane == 0) {
            if (tile) st[tile] = kPrefix | (prefix + total);
            s_prefix = prefix;
        }
    }
    __syncthreads();
    uint64_t run = s_prefix + before + incl - sum;
    if (wide) {
        const ulonglong2 a = make_ulonglong2(run, run + c[0]);
        const ulonglong2 b = make_ulonglong2(a.y + c[1], a.y + c[1] + c[2]);
        reinterpret_cast<ulonglong2*>(starts + i0)[0] = a;
        reinterpret_cast<ulonglong2*>(starts + i0)[1] = b;
        reinterpret_cast<ulonglong2*>(cursor + i0)[0] = a;
        reinterpret_cast<ulonglong2*>(cursor + i0)[1] = b;
        run += sum;
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (i0 + j < n) {
                starts[i0 + j] = run;
                cursor[i0 + j] = run;
            }
            run += c[j];
        }
    }
    if (i0 < n && i0 + 4 >= n) starts[n] = run;  // the thread holding the last counter
}

// Ranks of a bucket's n <= 64 distinct keys, two a lane (k0: element lane, k1:
// element 32 + lane; in0, in1: whether there is one; two: n > 32), by one warp.
// The keys of a bucket lie nearly evenly between its smallest and its largest,
// so 64 equal ranges of them (by the keys' top 32 bits) hold about one key
// each: a count per range, a scan over the counts, and each key is compared
// with the few of its own range only.  240 instructions a bucket of 26 keys where a
// bitonic network over packed words took 350 (15 or 21 steps of two shuffles, a
// 64-bit compare and two selects, 80 % of the ALU pipe).  The counts are zero
// before and after.  A range's first place and end share a word: two words cost
// the warp three more shared-memory wavefronts.
struct WarpRankTile {
    uint64_t key[64];
    uint32_t count[64];
    uint32_t place[64];  // a range's first place, and its end in the upper half
};
__device__ __forceinline__ uint32_t rank_in_range(const WarpRankTile& t, uint64_t k, uint32_t place) {
    uint32_t r = place & 0xffffu;
    const uint64_t *p = t.key + r, *const e = t.key + (place >> 16);
#pragma unroll 1
    for (; p < e; ++p) r += *p < k ? 1u : 0u;
    return r;
}
__device__ __forceinline__ void warp_rank64(WarpRankTile& t, uint64_t k0, uint64_t k1, bool in0, bool in1, bool two,
                                            int key_bits, int lane, uint32_t& r0, uint32_t& r1) {
    const int top = key_bits > 32 ? key_bits - 32 : 0;
    const uint32_t x0 = (uint32_t)(k0 >> top), x1 = (uint32_t)(k1 >> top);
    uint32_t lo = in0 ? x0 : 0xffffffffu, hi = in0 ? x0 : 0u;
    if (in1) {
        lo = min(lo, x1);
        hi = max(hi, x1);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    const int shift = max(0, 26 - __clz((int)(hi - lo)));  // (hi - lo) >> shift < 64
    const uint32_t b0 = (x0 - lo) >> shift, b1 = (x1 - lo) >> shift;
    uint32_t o0 = 0, o1 = 0;
    if (in0) o0 = atomicAdd(&t.count[b0], 1u);
    if (two && in1) o1 = atomicAdd(&t.count[b1], 1u);
    __syncwarp();
    const uint2 c = *reinterpret_cast<const uint2*>(&t.count[2 * lane]);
    *reinterpret_cast<uint2*>(&t.count[2 * lane]) = make_uint2(0u, 0u);
    uint32_t incl = c.x + c.y;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
        // the shuffle's own predicate: whether the lane has a source
        asm volatile(
            "{ .reg .b32 y; .reg .pred p; shfl.sync.up.b32 y|p, %0, %1, 0, 0xffffffff; @p add.u32 %0, %0, y; }"
            : "+r"(incl)
            : "r"(o));
    const uint32_t mid = incl - c.y;
    *reinterpret_cast<uint2*>(&t.place[2 * lane]) = make_uint2((mid - c.x) | mid << 16, mid | incl << 16);
    __syncwarp();
    uint32_t p0 = 0, p1 = 0;
    if (in0) {
        p0 = t.place[b0];
        t.key[(p0 & 0xffffu) + o0] = k0;
    }
    if (two && in1) {
        p1 = t.place[b1];
        t.key[(p1 & 0xffffu) + o1] = k1;
    }
    __syncwarp();
    r0 = rank_in_range(t, k0, p0);
    if (two) r1 = rank_in_range(t, k1, p1);
}

constexpr int kProbeLimit = 64;  // shared-memory table probes (taken in pairs) before a partition splits or falls back

// Filter pattern with the number of bits chosen at run time.
__device__ __forceinline__ uint64_t bloom_pattern_rt(uint64_t g, int n_hashes) {
    uint32_t lo = 0, hi = 0;
    for (int i = 0; i < n_hashes; ++i, g >>= 6) {
        const uint32_t bit = (uint32_t)g & 63u;
        lo |= shl_clamped(1u, bit);
        hi |= shl_clamped(1u, bit ^ 32u);
    }
    return ((uint64_t)hi << 32) | lo;
}

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

}  // namespace kc
