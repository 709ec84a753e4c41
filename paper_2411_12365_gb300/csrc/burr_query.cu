// burr_query.cu -- the layered query (Sec. 2: AND the key's coefficients with
// the table window, parity per value bit; a key below its bucket's threshold
// was bumped and is looked up in the next layer; the threshold is a 2-bit
// level code or, with 1+-bit thresholds, 0 unless the bucket's flag is set)
// and the standalone hash stage.
#include <type_traits>

#include "burr_internal.cuh"

namespace burr {

namespace {

constexpr int kQThreads = 256;

// Parity of a 64-bit word.
__device__ __forceinline__ uint32_t parity64q(uint64_t x) {
    return (uint32_t)__popc((uint32_t)x ^ (uint32_t)(x >> 32)) & 1u;
}

// Bit k of the value is the parity of c AND the 64 table bits of plane k from
// slot s on.  Those bits are bits o.. of block word w0 and bits ..o-1 of the
// next block's word w1 (o = s mod 64), so the parity is that of
// (w0 & (c << o)) ^ (w1 & (c >> (64 - o))): the row is shifted once per key
// instead of the window once per plane.
__device__ __forceinline__ void row_masks(uint64_t c, uint32_t o, uint64_t &cA, uint64_t &cB) {
    cA = c << o;
    cB = o ? c >> (64 - o) : 0ull;
}

// r-bit value of the window [s, s+63] selected by coefficient row c.
__device__ __forceinline__ uint32_t eval_window(const uint64_t *__restrict__ z, uint32_t r, uint32_t s,
                                                uint64_t c) {
    const uint64_t blk = s >> 6;
    const uint32_t o = s & 63u;
    const uint64_t *w0 = z + blk * r;
    uint64_t cA, cB;
    row_masks(c, o, cA, cB);
    uint32_t v = 0;
    if (o == 0) {
        for (uint32_t k = 0; k < r; ++k) v |= parity64q(__ldg(w0 + k) & cA) << k;
    } else {
        const uint64_t *w1 = w0 + r;
        for (uint32_t k = 0; k < r; ++k) v |= parity64q((__ldg(w0 + k) & cA) ^ (__ldg(w1 + k) & cB)) << k;
    }
    return v;
}

// 32-byte read-only global load (four table words).  kKeep: the line stays in
// L1.  A random window of a large table is not met again there, and allocated it
// drives the thresholds out (192 KB of 2-bit codes per 10^8 keys), which are:
// without, 10^8 keys of r = 8 took 1.81 -> 1.64 ms, 5*10^6 of r = 16 (10^7 stored)
// 230 -> 184 us; a table that mostly fits L1 is faster kept (10^6 stored keys, r =
// 3, 10^7 queried: 110 against 120 us).
template <bool kKeep>
__device__ __forceinline__ void ldg_v4(const uint64_t *p, uint64_t &a, uint64_t &b, uint64_t &c, uint64_t &d) {
    if (kKeep) asm("ld.global.nc.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(a), "=l"(b), "=l"(c), "=l"(d) : "l"(p));
    else asm("ld.global.nc.L1::no_allocate.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(a), "=l"(b), "=l"(c), "=l"(d) : "l"(p));
}

// The 2R table words around slot s (blocks s/64 and s/64 + 1), loaded before
// the threshold is known so that both reads are in flight together; R is the
// value width fixed at compile time.  The words are contiguous, so they are read
// in aligned 32-byte loads whatever R is (every table starts on 32 bytes and is
// allocated to a multiple of 32, see the launcher) and moved down by the place
// of the first word: narrow reads cost one L1 request per word and lane, and
// those bound the kernel (10^8 keys, r = 4: 1.76 ms with 8-byte loads).  The
// second block is needed only when the window is not block-aligned, and a window
// that starts at the last block (s = m - 64) has no second block inside the
// table: nothing past the needed words' last load is read.
template <int R>
struct Window {
    static constexpr int kMaxShift = R % 4 == 0 ? 0 : (R % 2 == 0 ? 2 : 3);
    static constexpr int kLoads = (2 * R + kMaxShift + 3) / 4;
    uint64_t w[4 * kLoads];
};

template <int R, bool kKeep>
__device__ __forceinline__ void load_window(const uint64_t *__restrict__ z, uint32_t s, Window<R> &w) {
    const uint64_t at = (uint64_t)(s >> 6) * R;
    const uint32_t shift = (uint32_t)at & 3u & (uint32_t)Window<R>::kMaxShift;
    const uint32_t need = shift + ((s & 63u) ? 2u * R : (uint32_t)R);
    const uint64_t *p = z + (at & ~3ull);
#pragma unroll
    for (int k = 0; k < Window<R>::kLoads; ++k) {
        if (4 * k < R || 4u * k < need) ldg_v4<kKeep>(p + 4 * k, w.w[4 * k], w.w[4 * k + 1], w.w[4 * k + 2], w.w[4 * k + 3]);
        else w.w[4 * k] = w.w[4 * k + 1] = w.w[4 * k + 2] = w.w[4 * k + 3] = 0;
    }
    if (Window<R>::kMaxShift & 1) {
#pragma unroll
        for (int k = 0; k + 1 < 4 * Window<R>::kLoads; ++k) w.w[k] = (shift & 1u) ? w.w[k + 1] : w.w[k];
    }
    if (Window<R>::kMaxShift & 2) {
#pragma unroll
        for (int k = 0; k + 2 < 4 * Window<R>::kLoads; ++k) w.w[k] = (shift & 2u) ? w.w[k + 2] : w.w[k];
    }
}

// The same words by loads of 16 bytes (kPairs, R even) or 8, which need not be moved.
template <int R, bool kPairs>
__device__ __forceinline__ void load_narrow(const uint64_t *__restrict__ z, uint32_t s, Window<R> &w) {
    const uint64_t *p = z + (uint64_t)(s >> 6) * R;
    const bool two = (s & 63u) != 0u;
    if (kPairs) {
        const ulonglong2 *q = reinterpret_cast<const ulonglong2 *>(p);
#pragma unroll
        for (int k = 0; k < R; k += 2) {
            const ulonglong2 x = __ldg(q + k / 2), y = two ? __ldg(q + (R + k) / 2) : ulonglong2{0ull, 0ull};
            w.w[k] = x.x;
            w.w[k + 1] = x.y;
            w.w[R + k] = y.x;
            w.w[R + k + 1] = y.y;
        }
    } else {
#pragma unroll
        for (int k = 0; k < R; ++k) {
            w.w[k] = __ldg(p + k);
            w.w[R + k] = two ? __ldg(p + R + k) : 0ull;
        }
    }
}

template <int R>
__device__ __forceinline__ uint32_t eval_loaded(const Window<R> &w, uint32_t s, uint64_t c) {
    uint64_t cA, cB;
    row_masks(c, s & 63u, cA, cB);   // cB is zero when the window is block-aligned
    uint32_t v = 0;
#pragma unroll
    for (int k = 0; k < R; ++k) v |= parity64q((w.w[k] & cA) ^ (w.w[R + k] & cB)) << k;
    return v;
}

// Values of more than 16 bits, a multiple of 4: the window of eight (four)
// planes at a time.
template <int R, bool kKeep>
__device__ __forceinline__ uint32_t eval_planes(const uint64_t *__restrict__ z, uint32_t s, uint64_t c) {
    const uint64_t *p = z + (uint64_t)(s >> 6) * R;
    uint64_t cA, cB;
    row_masks(c, s & 63u, cA, cB);
    const bool two = (s & 63u) != 0u;
    uint32_t v = 0;
#pragma unroll
    for (int k = 0; k < R; k += 4) {
        uint64_t a[4], b[4] = {0, 0, 0, 0};
        ldg_v4<kKeep>(p + k, a[0], a[1], a[2], a[3]);
        if (two) ldg_v4<kKeep>(p + R + k, b[0], b[1], b[2], b[3]);
#pragma unroll
        for (int j = 0; j < 4; ++j) v |= parity64q((a[j] & cA) ^ (b[j] & cB)) << (k + j);
    }
    return v;
}

// Threshold t of bucket b of bumping layer l: keys with offset < t are bumped.
// The mode is fixed at compile time: the other mode's registers cost occupancy.
template <bool kExact>
__device__ __forceinline__ uint32_t threshold_of(const QueryDesc &Q, uint32_t l, uint32_t b) {
    if (kExact) {
        // flag bit; a flagged bucket's threshold sits at its rank
        const uint64_t *fl = Q.flags[l];
        const uint64_t w = __ldg(fl + (b >> 6));
        if (!((w >> (b & 63u)) & 1ull)) return 0;
        uint32_t rank = __ldg(Q.dir[l] + (b >> 9));
        const uint32_t before = (b >> 6) & 7u;   // the block's flag words before this one
        fl += (b >> 9) << 3;
        // all loads first (a loop to `before` waited for each word)
        uint64_t x[7];
#pragma unroll
        for (uint32_t k = 0; k < 7; ++k) x[k] = k < before ? __ldg(fl + k) : 0ull;
#pragma unroll
        for (uint32_t k = 0; k < 7; ++k) rank += (uint32_t)__popcll(x[k]);
        rank += (uint32_t)__popcll(w & ((1ull << (b & 63u)) - 1ull));
        return __ldg(Q.tbytes[l] + rank);
    }
    return Q.levels[(uint32_t)(__ldg(Q.thresh[l] + (b >> 5)) >> (2 * (b & 31))) & 3u];
}

// The same in either mode, the flag words of a block one by one: less work where
// there is one flag word, or for keys that go through several layers.
__device__ __forceinline__ uint32_t threshold_any(const QueryDesc &Q, uint32_t l, uint32_t b) {
    if (Q.mode != BURR_THRESH_1PLUS) return threshold_of<false>(Q, l, b);
    const uint64_t *fl = Q.flags[l];
    const uint64_t w = __ldg(fl + (b >> 6));
    if (!((w >> (b & 63u)) & 1ull)) return 0;
    uint32_t rank = __ldg(Q.dir[l] + (b >> 9));
    for (uint32_t k = (b >> 9) << 3; k < (b >> 6); ++k) rank += (uint32_t)__popcll(__ldg(fl + k));
    rank += (uint32_t)__popcll(w & ((1ull << (b & 63u)) - 1ull));
    return __ldg(Q.tbytes[l] + rank);
}

// How a kernel finds thresholds.
enum { kCodes = 0, kFlags = 1, kEither = 2 };   // of 2-bit codes, of flags, threshold_any
template <int kHow>
__device__ __forceinline__ uint32_t threshold(const QueryDesc &Q, uint32_t l, uint32_t b) {
    return kHow == kEither ? threshold_any(Q, l, b) : threshold_of<kHow == kFlags>(Q, l, b);
}

// Query kernel for a value width R known at compile time: the table window
// of a layer is loaded together with its threshold (values of up to 16 bits),
// and the thread's next key is read while this key's table reads are in flight.
// Two keys per thread (their layer-0 reads in flight together, 98 registers)
// gave 70.7 ms against 72.5 at 10^9 keys (r = 8) but 4.69 against 4.20 and 0.89
// against 0.79 at 10^8 (r = 16, r = 1).
//
// kLoad: how the window is read (see query_r): by 32-byte loads, kept in L1 or not,
// by loads of 16 or 8 bytes after the threshold, or by 8-byte ones before it.
enum { kWide = 0, kWideKeep = 1, kNarrow = 2, kWords = 3 };
template <typename V, int R, int kLoad, int kHow>
__global__ void __launch_bounds__(kQThreads)
k_query_r(QueryDesc Q, const uint64_t *__restrict__ keys, V *__restrict__ out, uint64_t n) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const uint32_t log2B = 31 - __clz(Q.B);
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    uint64_t key_next = i < n ? keys[i] : 0ull;
    for (; i < n; i += stride) {
        const uint64_t key = key_next;
        if (i + stride < n) key_next = keys[i + stride];
        uint32_t v = 0;
        for (uint32_t l = 0; l <= Q.layers; ++l) {               // [layers] = base case
            const uint64_t m = Q.m[l];
            if (m == 0) break;
            const uint64_t h = mix64(key ^ Q.sigma[l]);
            const uint32_t s = (uint32_t)__umul64hi(h, m - kW + 1);
            if constexpr (R <= 16) {
                Window<R> w;
                if (kLoad == kWords) load_narrow<R, false>(Q.z[l], s, w);
                else if (kLoad != kNarrow) load_window<R, kLoad == kWideKeep>(Q.z[l], s, w);
                if (l < Q.layers && (s & (Q.B - 1)) < threshold<kHow>(Q, l, s >> log2B)) continue;   // bumped: next layer
                // (read before the threshold is known they are slower: r = 7 in 100 KB 77 against 71 us, r = 15 167 / 144)
                if (kLoad == kNarrow) load_narrow<R, R % 2 == 0>(Q.z[l], s, w);
                v = eval_loaded<R>(w, s, mix64(h + Q.sigma[l]) | 1ull);
            } else {
                if (l < Q.layers && (s & (Q.B - 1)) < threshold<kHow>(Q, l, s >> log2B)) continue;
                v = eval_planes<R, kLoad == kWideKeep>(Q.z[l], s, mix64(h + Q.sigma[l]) | 1ull);
            }
            break;
        }
        out[i] = (V)v;
    }
}

// Widths of 8, 16 and 32 bits: a block of R words is R / 4 32-byte sectors, which
// G = R / 4 neighbouring lanes read together, for the keys of the group in turn;
// each lane evaluates four planes of all G keys, and the group exchanges the
// results.  A load is then one request per key and block instead of one per
// sector: those requests of an SM to L2 bound the kernel of one lane per key.
// Now they are at 58% of their peak, the sectors returned at 26%, L1's data pipe at 76% and the ALU
// at 75% (1.6*10^7 keys of a 30 MB table, r = 8).  The bumped keys (2 in 100)
// go on lane by lane in the deeper layers.  Measured against one lane per key:
// r = 8, 10^8 keys of a 100 MB table 1.71 -> 1.58 ms, 2*10^7 of a 1 MB table 445 ->
// 290 us (1+-bit); r = 16, 5*10^6 of 20 MB 182 -> 118 us, 1+-bit 261 -> 130; r = 32,
// 2*10^7 of 40 MB 1070 -> 717 us.
template <typename V, int R, bool kKeep, bool kExact>
__global__ void __launch_bounds__(kQThreads)
k_query_group(QueryDesc Q, const uint64_t *__restrict__ keys, V *__restrict__ out, uint64_t n) {
    constexpr int G = R / 4, kAtOnce = G < 4 ? G : 4;   // keys of the group whose reads are in flight together
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const uint32_t log2B = 31 - __clz(Q.B);
    const int lane = threadIdx.x & 31, q = lane & (G - 1), first = lane & ~(G - 1);
    const uint64_t m0 = Q.m[0], sigma0 = Q.sigma[0];
    const uint64_t *__restrict__ z0 = Q.z[0] + 4 * q;
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    uint64_t key_next = i < n ? keys[i] : 0ull;
    // a whole warp at a time: lanes past the end take part with key 0
    for (; i - (uint64_t)lane < n; i += stride) {
        const uint64_t key = key_next;
        if (i + stride < n) key_next = keys[i + stride];
        const uint64_t h = mix64(key ^ sigma0);
        const uint32_t s = (uint32_t)__umul64hi(h, m0 - kW + 1);
        const bool bumped = (s & (Q.B - 1)) < threshold_of<kExact>(Q, 0, s >> log2B);
        const uint64_t c = mix64(h + sigma0) | 1ull;
        uint32_t part = 0;   // planes 4q .. 4q + 3 of the group's keys, key t at bits 4t
#pragma unroll
        for (int t0 = 0; t0 < G; t0 += kAtOnce) {
            uint64_t a[kAtOnce][4], b[kAtOnce][4];
            uint32_t st[kAtOnce];
#pragma unroll
            for (int t = 0; t < kAtOnce; ++t) {
                st[t] = __shfl_sync(0xffffffffu, s, first + t0 + t);
                const uint64_t *p = z0 + (uint64_t)(st[t] >> 6) * R;
                ldg_v4<kKeep>(p, a[t][0], a[t][1], a[t][2], a[t][3]);
                b[t][0] = b[t][1] = b[t][2] = b[t][3] = 0;
                if (st[t] & 63u) ldg_v4<kKeep>(p + R, b[t][0], b[t][1], b[t][2], b[t][3]);
            }
#pragma unroll
            for (int t = 0; t < kAtOnce; ++t) {
                const uint64_t ct = (uint64_t)__shfl_sync(0xffffffffu, (uint32_t)(c >> 32), first + t0 + t) << 32 |
                                    __shfl_sync(0xffffffffu, (uint32_t)c, first + t0 + t);
                uint64_t cA, cB;
                row_masks(ct, st[t] & 63u, cA, cB);
#pragma unroll
                for (int k = 0; k < 4; ++k) part |= parity64q((a[t][k] & cA) ^ (b[t][k] & cB)) << (4 * (t0 + t) + k);
            }
        }
        uint32_t v = ((part >> (4 * q)) & 15u) << (4 * q);
#pragma unroll
        for (int d = 1; d < G; ++d) {
            const uint32_t x = __shfl_xor_sync(0xffffffffu, part, d);
            v |= ((x >> (4 * q)) & 15u) << (4 * (q ^ d));
        }
        if (bumped) {
            v = 0;
            for (uint32_t l = 1; l <= Q.layers; ++l) {           // [layers] = base case
                const uint64_t m = Q.m[l];
                if (m == 0) break;
                const uint64_t hl = mix64(key ^ Q.sigma[l]);
                const uint32_t sl = (uint32_t)__umul64hi(hl, m - kW + 1);
                if (l < Q.layers && (sl & (Q.B - 1)) < threshold_of<kExact>(Q, l, sl >> log2B)) continue;
                v = eval_planes<R, false>(Q.z[l], sl, mix64(hl + Q.sigma[l]) | 1ull);
                break;
            }
        }
        if (i < n) out[i] = (V)v;
    }
}

// Any width, plane by plane.  (kFlags with the mode fixed is slower: r = 3, 4*10^6
// queries of 7 KB 70 us against 54.)
template <typename V, int kHow>
__global__ void __launch_bounds__(kQThreads)
k_query(QueryDesc Q, const uint64_t *__restrict__ keys, V *__restrict__ out, uint64_t n) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const uint32_t log2B = 31 - __clz(Q.B);
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint64_t key = keys[i];
        uint32_t v = 0;
        uint32_t l = 0;
        for (; l < Q.layers; ++l) {
            const uint64_t m = Q.m[l];
            if (m == 0) break;
            const uint64_t h = mix64(key ^ Q.sigma[l]);
            const uint32_t s = (uint32_t)__umul64hi(h, m - kW + 1);
            const uint32_t b = s >> log2B;
            const uint32_t off = s & (Q.B - 1);
            const uint32_t t = kHow == kFlags && Q.mode != BURR_THRESH_1PLUS ? threshold<kCodes>(Q, l, b) : threshold<kHow>(Q, l, b);
            if (off < t) continue;                             // bumped: next layer
            v = eval_window(Q.z[l], Q.r, s, mix64(h + Q.sigma[l]) | 1ull);
            break;
        }
        if (l == Q.layers && Q.m[l] != 0) {                    // base case
            const uint64_t h = mix64(key ^ Q.sigma[l]);
            const uint32_t s = (uint32_t)__umul64hi(h, Q.m[l] - kW + 1);
            v = eval_window(Q.z[l], Q.r, s, mix64(h + Q.sigma[l]) | 1ull);
        }
        out[i] = (V)v;
    }
}

__global__ void k_hash(const uint64_t *__restrict__ keys, uint64_t n, uint64_t sigma, uint64_t range,
                       uint32_t *__restrict__ start, uint64_t *__restrict__ coeff) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        uint32_t s;
        uint64_t c;
        equation(keys[i], sigma, range, s, c);
        start[i] = s;
        coeff[i] = c;
    }
}

}  // namespace

namespace {

// The kernel of width Q.r, if there is one for the case; false: any width's kernel
// (launch_query), which reads plane by plane.  Times in us for 4*10^6 queries, 2-bit
// thresholds, unless said.
//
// Groups of lanes (r = 8 from 8 KB on, 16, 32; both sides at k_query_group; r = 8 in 2 KB 62, one lane per
// key 56) exchange results, which few keys don't pay for: r = 8 in 50 KB / 1 MB, 10,007 keys 3.4 / 4.1, one
// lane per key 3.2 / 3.6; 10^5 keys 4.4 / 4.8 and 5.0 / 5.3; r = 16, 20 keys 2.5 / 3.3 and 2.1 / 2.7.
//
// Kept in L1, where a table mostly fits it: groups up to 128 KB (kept / not: r = 8, 2 KB 62 / 393,
// 20 KB 55 / 104; r = 16, 200 KB 91 / 95, 800 KB 100 / 95), single keys up to 1 MB.
//
// Widths that are no multiple of 4 pay for moving a window read by wide loads (odd ones most).
// Wide loads / narrow ones:
//   r = 2    20 KB..5 MB  39..40 / 34..36;   1+-bit 60..65 / 52..56
//   r = 3    7 KB 48 / 36;  375 KB 52 / 50 (any width's 48);  1.5 MB 52 / 53;  7 MB 52 / 54
//   r = 5    60 KB 64 / 52;  250 KB 66 (any width's 60);  625 KB 68 / 76 (any width's 70)
//   r = 6    75 KB 57 / 46;  750 KB 64 / 64;  3 MB 64 / 67
//   r = 10, 14   125, 175 KB 85, 109 / 60, 82;  1.3, 1.8 MB 97, 127 / 99, 141
//   r = 13, 15   160, 190 KB 134, 157 / 126, 144;  1.6, 1.9 MB 152, 177 / 167, 199
// and with 1+-bit thresholds, whose loads take the registers, even widths are best narrow (r = 6, 10, 14 in
// 12 to 35 MB: 101, 175, 195 / 83, 124, 162), odd ones up to 11 in any width's kernel (r = 5 in 625 KB: 99 / 98 / 81),
// 13 and 15 narrow (1.6, 1.9 MB: 204, 220 / 196, 226).  With one flag word (a few thousand keys) r = 1 and 8 look
// the words up one by one (r = 8, 10^6 queries of 3,000 keys 19.8 / 21.8).
//
// These lines hold near the default load of 1.015.  Far from it other keys are met in other layers (at 1.3 a
// quarter are bumped and the wide loads of their windows are wasted: r = 15 in 560 KB takes 1.46 times as long as
// plane by plane; at 0.8 hardly a bucket is flagged).  There, and for tables off 32-byte boundaries (of a
// caller's allocator), the widths that lost keep to kernels of either mode.  Over 1,824 combinations of width,
// mode and sizes at each of the loads 0.8, 0.97, 1.04, 1.05, 1.1, 1.3, by the lines alone 80, 27, 28, 30, 87, 223
// are more than 4% slower than plane by plane (r = 1, 8, 16: than one lane per key), with the exception at
// 0.8, 0.97, 1.05, 1.1, 1.3 8, 12, 7, 12, 7; at 1.0, 1.015, 1.03, by the lines, 6, 6, 8 are.
inline bool usual_load(const QueryDesc &Q) { return Q.load >= 0.995f && Q.load <= 1.03f; }
constexpr uint64_t kGroupKeys = 1 << 15, kGroupKeys16 = 256;
template <int R>
bool query_r(const QueryDesc &Q, const uint64_t *keys, void *out, uint64_t n, unsigned grid, bool aligned, cudaStream_t st) {
    using V = std::conditional_t<(R <= 8), uint8_t, std::conditional_t<(R <= 16), uint16_t, uint32_t>>;
    const uint64_t kb = (Q.m[0] / 64) * R * 8 >> 10;   // layer 0 holds nearly all of the table
    const bool exact = Q.mode == BURR_THRESH_1PLUS, other = !usual_load(Q);
    const bool one_word = exact && Q.m[0] <= 64ull * Q.B;   // of flags
    auto go = [&](auto *kernel) {
        kernel<<<grid, kQThreads, 0, st>>>(Q, keys, (V *)out, n);
        return true;
    };
    // without bumping layers there is no layer 0 with thresholds, in either mode
    const bool layers = Q.layers > 0 && Q.m[0] != 0;
    if constexpr (R == 1) {   // two words: narrow reads of the same sector are cheaper than the move
        if (one_word || other) return go(k_query_r<V, 1, kWords, kEither>);
        return exact ? go(k_query_r<V, 1, kWords, kFlags>) : go(k_query_r<V, 1, kWords, kCodes>);
    } else if constexpr (R == 8 || R == 16 || R == 32) {
        auto group = [&]() {
            if (kb < 128) return exact ? go(k_query_group<V, R, true, true>) : go(k_query_group<V, R, true, false>);
            return exact ? go(k_query_group<V, R, false, true>) : go(k_query_group<V, R, false, false>);
        };
        if (!aligned) {
            // (4*10^6 keys: r = 8 151 us, plane by plane 147; r = 16 452, 427; 1,000 keys: 3.1 / 4.4, 4.3 / 7.3)
            if constexpr (R != 32) {
                if (n < kGroupKeys) return go(k_query_r<V, R, kWords, kEither>);
            }
            return false;
        }
        if (!layers) return kb < 1024 ? go(k_query_r<V, R, kWideKeep, kCodes>) : go(k_query_r<V, R, kWide, kCodes>);
        if constexpr (R == 8) {
            if (kb >= 8 && (exact || n >= kGroupKeys)) return group();
            if (one_word || other) return go(k_query_r<V, R, kWideKeep, kEither>);
            return exact ? go(k_query_r<V, R, kWideKeep, kFlags>) : go(k_query_r<V, R, kWideKeep, kCodes>);
        } else {
            if constexpr (R == 16) {
                if (n < kGroupKeys16 || (other && kb < 16)) return go(k_query_r<V, R, kWideKeep, kEither>);
            }
            return group();
        }
    } else if constexpr (R % 4 != 0) {
        if (!aligned || (other && R % 2 != 0)) return false;
        if (exact) {
            if constexpr (R % 2 == 0 || R >= 13) return go(k_query_r<V, R, kNarrow, kFlags>);
            return false;
        }
        if constexpr (R == 2) {
            return go(k_query_r<V, R, kNarrow, kCodes>);
        } else {
            constexpr uint64_t kNarrowKb = R % 2 == 0 ? 512 : R >= 7 ? 256 : 64;
            constexpr uint64_t kGeneralKb = R == 3 ? 1536 : R == 5 ? 512 : kNarrowKb;
            if (kb < kNarrowKb) return go(k_query_r<V, R, kNarrow, kCodes>);
            if (kb < kGeneralKb || other) return false;
            if constexpr (kGeneralKb < 1024) {
                if (kb < 1024) return go(k_query_r<V, R, kWideKeep, kCodes>);
            }
            return go(k_query_r<V, R, kWide, kCodes>);
        }
    } else {
        if (!aligned || (other && exact && R <= 12)) return false;
        if (kb < 1024) return exact ? go(k_query_r<V, R, kWideKeep, kFlags>) : go(k_query_r<V, R, kWideKeep, kCodes>);
        return exact ? go(k_query_r<V, R, kWide, kFlags>) : go(k_query_r<V, R, kWide, kCodes>);
    }
}

bool launch_query_r(const QueryDesc &Q, const uint64_t *keys, void *out, uint64_t n, unsigned grid, bool aligned,
                    cudaStream_t st) {
    switch (Q.r) {
#define BURR_QUERY_R(R) \
    case R: return query_r<R>(Q, keys, out, n, grid, aligned, st);
        BURR_QUERY_R(1) BURR_QUERY_R(2) BURR_QUERY_R(3) BURR_QUERY_R(4) BURR_QUERY_R(5) BURR_QUERY_R(6)
        BURR_QUERY_R(7) BURR_QUERY_R(8) BURR_QUERY_R(9) BURR_QUERY_R(10) BURR_QUERY_R(11) BURR_QUERY_R(12)
        BURR_QUERY_R(13) BURR_QUERY_R(14) BURR_QUERY_R(15) BURR_QUERY_R(16) BURR_QUERY_R(20) BURR_QUERY_R(24)
        BURR_QUERY_R(28) BURR_QUERY_R(32)
#undef BURR_QUERY_R
    default: return false;
    }
}

}  // namespace

cudaError_t launch_query(const QueryDesc &Q, uint32_t vbytes, const uint64_t *keys, void *out, uint64_t n,
                         cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    const unsigned grid = grid_for(n, kQThreads, 152u * 64u);
    // 32-byte reads when every table of the structure starts on 32 bytes (a caller's allocator may
    // give others); the library allocates every table to a multiple of 32 bytes
    bool aligned = true;
    for (uint32_t l = 0; l <= Q.layers; ++l)
        if (Q.m[l] != 0 && ((uintptr_t)Q.z[l] & 31u) != 0) aligned = false;
    if (launch_query_r(Q, keys, out, n, grid, aligned, st)) return cudaGetLastError();
    // any width, plane by plane.  Fixed to a mode: r = 3, 4*10^6 keys of 1 MB 71 / 82 us, r = 9 with 1+-bit
    // thresholds 109 / 124; but r = 5 of 1.9 MB 5.2 / 4.5 us for 10,007 keys, r = 31 15.2 / 10.8, r = 9 with
    // 1+-bit thresholds 9.6 / 9.0 for 10^5 keys of 5.6 MB
    const bool exact = Q.mode == BURR_THRESH_1PLUS;
    const bool few = n < kGroupKeys && Q.m[0] <= 64ull * Q.B;   // keys, and flag words
    const bool either = (!aligned && Q.r != 8 && Q.r != 16) || Q.r > 16 || !usual_load(Q) ||
                        (exact ? few || (Q.m[0] / 64) * Q.r * 8 >= 1 << 20 : Q.r == 5);
    auto go = [&](auto *codes, auto *flags, auto *any, auto *v) {
        (either ? any : exact ? flags : codes)<<<grid, kQThreads, 0, st>>>(Q, keys, v, n);
    };
    switch (vbytes) {
    case 1: go(k_query<uint8_t, kCodes>, k_query<uint8_t, kFlags>, k_query<uint8_t, kEither>, (uint8_t *)out); break;
    case 2: go(k_query<uint16_t, kCodes>, k_query<uint16_t, kFlags>, k_query<uint16_t, kEither>, (uint16_t *)out); break;
    default: k_query<uint32_t, kEither><<<grid, kQThreads, 0, st>>>(Q, keys, (uint32_t *)out, n); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_hash(const uint64_t *keys, uint64_t n, uint64_t sigma, uint64_t range, uint32_t *start,
                        uint64_t *coeff, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    k_hash<<<grid_for(n, 256, 152u * 32u), 256, 0, st>>>(keys, n, sigma, range, start, coeff);
    return cudaGetLastError();
}

}  // namespace burr
