// burr_band.cu -- insertion with bumping ("Insertion" of Fig. 7; Sec. 2
// "Bumping" and Sec. 3 "Bumping at thread boundaries").
//
// One warp per partition.  The paper gives one partition to one CPU thread,
// which eliminates the rows one by one against a stored band.  Here the warp
// sweeps the slots of its partition from left to right instead and settles one
// slot per step:
//
//   * A row is live from its start slot until it becomes the pivot row of a
//     slot.  At slot j every live row has its support in [j, j + 63], so at
//     most 64 of them are independent, and they fit in registers: two rows per
//     lane, as 64 coefficient bits (bit of slot s at position s mod 64, so
//     that nothing is shifted from slot to slot), the right-hand side and a
//     key.
//   * A step picks, among the live rows with bit j, the one of the highest
//     priority (one warp maximum over keys), stores it as slot j's row and
//     XORs it into the others.  No row meets more than one stored row per step
//     and none waits for another lane's chain of eliminations.
//   * Priority is the paper's insertion order: rows of earlier buckets first,
//     then descending offset.  A row is then only ever changed by rows that are
//     inserted before it, so a row that becomes zero is dependent on them, as
//     in the row-by-row elimination in descending offset order; with offset o
//     its bucket's threshold is the least one above o.  The rows at offsets
//     >= t and the slots they hold are untouched by the rows below t, so
//     bumping is just dropping the rows below t and emptying their slots:
//     nothing is rolled back or inserted again, in either threshold mode.
//   * Rows of bucket b may turn out dependent up to 63 slots into bucket b + 1,
//     whose rows they have changed by then.  The live rows at the bucket
//     boundary are therefore kept in shared memory, and bucket b + 1 starts
//     again from them without the dropped rows (a few percent of the buckets).
//   * More live rows than registers means more than 64 rows in 64 slots, so a
//     dependency: the lowest-offset row of the bucket cannot be kept, and the
//     threshold above it is taken at once.
//
// What bounds it: with every CTA slot taken, the ALU pipe (integer logic, selects
// and compares at half rate): 77% of its peak and 66% of the issue slots (3*10^7 keys
// in 3,608 partitions), 43 warp instructions and about 61 cycles of an SM quarter per
// slot (10^9 keys).  A step is 37 of these cycles; the rest is the bookkeeping
// between blocks of slots, staging, writing out, and waits at the pair's barrier.
// With few partitions, the chain of a warp alone: about 6.6 us per bucket, 107
// cycles per slot, of which the step (bit test, warp maximum, shuffle, XOR) is about
// 75.  Layer-0 band, ms (r = 8 unless said), against the streaming insertion
// that it replaces (32 lanes eliminating one row each against a band in shared
// memory, a 128-bit compare-and-swap per step, every bucket as long as its longest
// chain, a dependent bucket inserted again; sparse layers still take it, see
// burr_band_stream.cuh):
//   5*10^4 keys, r = 3 (1 partition)              4.59 -> 2.9 (in segments 0.71)
//   10^6 keys (16 partitions)                     6.57 -> 3.9 (in segments 1.24)
//   10^7 keys, r = 16, 1+-bit, searched cuts      13.7 -> 6.1
//   10^8 keys (1504 partitions)                   8.33 -> 6.2;  1+-bit 16.3 -> 9.0
//   10^9 keys (15034 partitions)                  63.7 -> 47.5
//   10^8 keys, r = 17..32                         8.4 -> 6.9;  1+-bit 16.2 -> 9.6
//   10^8 keys at load 1.3                         13.7 -> 6.9;  1+-bit 50.2 -> 22.3
#include <algorithm>
#include <cmath>

#include "burr_internal.cuh"

namespace burr {

namespace {

constexpr int kRing = 256;              // stored rows kept on chip: a bucket and the one before it
constexpr uint32_t kRingMask = kRing - 1;
constexpr int kStage = 192;             // rows of a bucket staged at once (see stage_rows)
constexpr int kStagePerLane = kStage / 32;
constexpr unsigned kFull = 0xffffffffu;
// Slots per round of the sweep's loop.  The whole sweep has to stay small: with
// 16 slots unrolled and the sweep inlined for both halves of a bucket, the
// warps of an SM, each at its own place in the code, waited on instruction
// fetches (layer-0 band of 10^9 keys 104.7 ms against 60.9 with 4 slots and
// one copy).  Now 4 / 8 / 16 slots: 47.4 / 47.5 / 50.4 ms, 10^6 keys 1.27 / 1.31 / 1.65.
constexpr uint32_t kUnrollSlots = 4;
// CTAs (partitions) per SM that the registers allow: 16 (64 registers a thread, 92
// bytes of spill loads with one-byte values, 48 with wider ones) where partitions
// outnumber what fits, else 14 (72, 56 and 20).  Builds, ms, 16 / 14: 10^9 keys 68.6 / 70.4; 3*10^8
// r = 8 22.9 / 22.9, r = 16 25.2 / 25.5, 1+-bit 30.8 / 31.8, r = 32 30.5 / 29.6, 1+-bit 35.7 / 35.5.  Layer-0 band with all
// partitions resident: 10^8 keys 6.37 / 6.33, 1+-bit 9.41 / 9.33, 10^6 1.31 / 1.27.
constexpr int kManyCtas = 16, kFewCtas = 14;
constexpr uint64_t kFewParts = 152 * kFewCtas;

// Key of a live row: bit 30 = row of an earlier bucket, bits 22..29 = offset + 1,
// bit 21 = which of the lane's two rows, bits 0..4 = lane (so that a key is a
// shuffle's source lane as it is); 0 = no row.  Bits 5..20 hold the right-hand
// side when it has at most 16 bits: the maximum over keys that finds the pivot
// then brings its right-hand side along.
constexpr uint32_t kOldKey = 1u << 30;
constexpr uint32_t kOffsetBit = 22, kRowBit = 21, kValueBit = 5;
constexpr uint32_t kValueMask = 0xffffu << kValueBit;
__device__ __forceinline__ uint32_t key_offset(uint32_t key) { return ((key >> kOffsetBit) & 0xffu) - 1u; }

// A live row: w1:w0 are its 64 coefficient bits relative to the block of slots
// being swept (rotated right by the block's length after it), so that the
// block's slots are the low bits of w0.  A row that starts inside the block
// ignores the slots before its start (whose positions hold its last bits).
struct Row {
    uint32_t w0, w1, key, y, gate;   // y: right-hand sides of more than 16 bits
};

// A stored row of the ring, as it was live at its slot: rotated by the slot's
// place in its block, which is kept in y (in the key's value bits where y is
// taken).  key 0 = empty slot.
struct alignas(16) Pivot {
    uint32_t w0, w1, key, y;
};

// A staged equation: one 16-byte read hands it to a lane.
struct alignas(16) StagedRow {
    uint32_t lo, hi;        // coefficient row (bit 0 = start slot)
    uint32_t y;             // right-hand side
    uint32_t o;             // offset of the start slot in its bucket
};

// What one warp works on: a partition of one structure's layer, and where that
// structure's data sits in the layer-wide arrays (all bases 0 for a single
// structure).  It sits in shared memory: it is read once per bucket or less, and
// held in registers it took 60 of them.
struct Ctx {
    LayerDesc L;
    uint32_t part;
    uint64_t bucket_base, slot_base, tw_base, out_base;
    uint64_t own_hi;         // one past the partition's slots
    uint32_t b0, b1;         // its buckets
    uint32_t pend;           // end of its equations
    unsigned long long *bcount;
    uint32_t *fail;          // base case, batched: per-structure flag
};

struct BandSmem {
    Pivot ring[kRing];             // stored rows of slots [bucket start - B, bucket start + B)
    StagedRow rows[2][kStage];     // staged equations of two buckets, ascending offset
    uint32_t first[2][132];        // first staged index of each offset (+ [128] = count)
    uint32_t tstage[2];            // threshold the bucket starts from
    uint32_t tdone;                // final threshold of the bucket before the one being swept
    // why both warps leave at the barrier of the first or second half of a bucket (kRunError or
    // kRunCoupled; one word per half, or a warp could see the other's next half's reason)
    uint32_t stop[2];
    uint32_t at;                   // bucket where the last run ended
    uint32_t sweeper;              // the warp that sweeps
    uint32_t failed;               // the build has failed already
    Pivot snap[2][32];             // live rows at the bucket's start
    alignas(4) uint8_t stored[64]; // rows (lane, and 32 + lane) that a block of slots stored
    Ctx x;
};

template <typename V>
struct BandArgs {
    LayerDesc L;
    const uint64_t *keys;    // bucket-sorted records h = mix64(key ^ sigma) of the layer's keys (or packed)
    const V *vals;
    const uint32_t *bstart;
    uint64_t *Cg;
    V *Yg;
    uint64_t *thresh;        // 2-bit codes (2-bit mode)
    uint8_t *texact;         // exact threshold of every bucket (1+-bit mode)
    uint64_t *bkeys;
    V *bvals;
    unsigned long long *bcount;
    uint32_t *err;
    BatchView bv;            // sd == nullptr: a single layer described by L
    // segmented launches (see k_band_seg)
    uint32_t seg;            // buckets per segment
    uint32_t nseg;           // segments of the longest partition
    uint64_t *omask;         // per bucket: slots of its first 64 held by rows of the bucket before
    struct Pivot *state[2];  // per segment: live rows at its end, as the last even and odd pass left them
    uint32_t *moved[2];      // per segment: the last odd (even) pass left other rows than the passes before
};

enum { kRunDone = 0, kRunError = 1, kRunCoupled = 2 };

// Least threshold of the layer's mode at or above o (o <= B).
__device__ __forceinline__ uint32_t threshold_from(const LayerDesc &L, uint32_t o) {
    if (L.mode == BURR_THRESH_1PLUS) return o;
    if (o == 0) return 0;
    return o <= L.levels[1] ? L.levels[1] : (o <= L.levels[2] ? L.levels[2] : L.levels[3]);
}

// 2-bit code of threshold t.
__device__ __forceinline__ uint32_t code_of(const LayerDesc &L, uint32_t t) {
    return t == 0 ? 0u : (t <= L.levels[1] ? 1u : (t <= L.levels[2] ? 2u : 3u));
}

// Exclusive scan of first[0..128) in place, first[128] = total.
__device__ __forceinline__ void scan_first(uint32_t *first, int lane) {
    uint32_t v[4], loc = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        v[k] = first[4 * lane + k];
        loc += v[k];
    }
    uint32_t incl = loc;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t t = __shfl_up_sync(kFull, incl, d);
        if (lane >= d) incl += t;
    }
    __syncwarp();
    uint32_t run = incl - loc;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        first[4 * lane + k] = run;
        run += v[k];
    }
    if (lane == 31) first[128] = incl;
    __syncwarp();
}

// Record h and value of equation i (base: the bucket's entry of L.hbase if packed).
template <typename V>
__device__ __forceinline__ uint64_t record(const uint64_t *keys, const V *vals, uint32_t i, bool packed, uint64_t base,
                                           uint32_t &v) {
    const uint64_t k = keys[i];
    if (sizeof(V) == 1 && packed) {
        v = packed_value(k);
        return packed_h(k, base);
    }
    v = (uint32_t)vals[i];
    return k;
}

// Stage the rows of bucket [rs, re) (start slot bB) at offsets >= the returned
// threshold, in ascending offset order; first[o] = first index with offset
// >= o.  The rows at offsets >= o span 63 + B - o slots, so where there are
// more of them the threshold is above o; the rows left after that (at most
// 63 + B) always fit the stage.  Otherwise returns `forced` and stages every
// row (the sweep skips those below the threshold).  A call, not inline code:
// its registers would stay live across the sweep.
template <typename V>
__device__ __noinline__ uint32_t stage_rows(StagedRow *rows, uint32_t *first, const BandArgs<V> &a, const LayerDesc &L,
                                            uint32_t rs, uint32_t re, uint32_t bB, uint32_t forced,
                                            bool packed, uint64_t base, int lane) {
    const uint32_t cnt = re - rs;
    for (int i = lane; i < 132; i += 32) first[i] = 0;
    __syncwarp();
    if (cnt <= (uint32_t)kStage) {
        uint64_t c[kStagePerLane];
        uint32_t y[kStagePerLane], at[kStagePerLane];   // at: offset, and rank among its rows from bit 8
#pragma unroll
        for (int j = 0; j < kStagePerLane; ++j) {
            const uint32_t i = (uint32_t)lane + 32u * j;
            if (i < cnt) {
                const uint64_t h = record(a.keys, a.vals, rs + i, packed, base, y[j]);
                c[j] = coeff_of_h(h, L.sigma);
                const uint32_t o = start_of_h(h, L.range) - bB;
                y[j] &= L.vmask;
                at[j] = o | atomicAdd(&first[o], 1u) << 8;
            }
        }
        __syncwarp();
        scan_first(first, lane);
#pragma unroll
        for (int j = 0; j < kStagePerLane; ++j) {
            const uint32_t i = (uint32_t)lane + 32u * j;
            if (i < cnt) {
                const uint32_t o = at[j] & 0xffu;
                rows[first[o] + (at[j] >> 8)] = StagedRow{(uint32_t)c[j], (uint32_t)(c[j] >> 32), y[j], o};
            }
        }
        __syncwarp();
        return forced;
    }
    // more rows than can be kept: count, find the threshold, stage the rows above it
    uint32_t v = 0;
    for (uint32_t i = rs + lane; i < re; i += 32)
        atomicAdd(&first[start_of_h(record(a.keys, a.vals, i, packed, base, v), L.range) - bB], 1u);
    __syncwarp();
    scan_first(first, lane);
    uint32_t over = 0;   // one above the largest offset o with more than 63 + B - o rows at offsets >= o
    for (uint32_t o = lane; o < L.B; o += 32)
        if (cnt - first[o] > 63u + L.B - o) over = o + 1;
    over = __reduce_max_sync(kFull, over);
    const uint32_t t = max(forced, threshold_from(L, over));
    __syncwarp();
    for (int i = lane; i < 132; i += 32) first[i] = 0;
    __syncwarp();
    for (uint32_t i = rs + lane; i < re; i += 32) {
        const uint32_t o = start_of_h(record(a.keys, a.vals, i, packed, base, v), L.range) - bB;
        if (o >= t) atomicAdd(&first[o], 1u);
    }
    __syncwarp();
    scan_first(first, lane);
    // place the rows: the cursor of offset o is first[o] itself, which then ends where offset
    // o + 1 starts
    for (uint32_t i = rs + lane; i < re; i += 32) {
        const uint64_t h = record(a.keys, a.vals, i, packed, base, v);
        const uint32_t o = start_of_h(h, L.range) - bB;
        if (o >= t) {
            const uint64_t c = coeff_of_h(h, L.sigma);
            const uint32_t p = atomicAdd(&first[o], 1u);
            rows[p] = StagedRow{(uint32_t)c, (uint32_t)(c >> 32), v & L.vmask, o};
        }
    }
    __syncwarp();
    uint32_t f[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) f[k] = first[4 * lane + k];
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 4; ++k) first[4 * lane + k + 1] = f[k];
    if (lane == 0) first[0] = 0;
    __syncwarp();
    return t;
}

// Rows of the bucket below threshold t leave for the next layer (as keys: the
// next layer hashes them with its own seed).
template <typename V>
__device__ __noinline__ void emit_bumped(const BandArgs<V> &a, const Ctx &x, uint32_t rs, uint32_t re, uint32_t bB,
                                         uint32_t t, int lane) {
    const bool packed = sizeof(V) == 1 && x.L.hbase;
    const uint64_t hb = packed ? x.L.hbase[(bB / x.L.B) >> x.L.hshift] : 0ull;
    for (uint32_t base = rs; base < re; base += 32) {
        const uint32_t idx = base + lane;
        bool bump = false;
        uint64_t key = 0;
        uint32_t val = 0;
        if (idx < re) {
            const uint64_t h = record(a.keys, a.vals, idx, packed, hb, val);
            bump = (start_of_h(h, x.L.range) - bB) < t;
            if (bump) {
                key = key_of_h(h, x.L.sigma);
            }
        }
        const uint32_t mask = __ballot_sync(kFull, bump);
        if (!mask) continue;
        unsigned long long ob = 0;
        if (lane == 0) ob = atomicAdd(x.bcount, (unsigned long long)__popc(mask));
        ob = __shfl_sync(kFull, ob, 0);
        if (bump) {
            const unsigned long long o = x.out_base + ob + __popc(mask & ((1u << lane) - 1u));
            a.bkeys[o] = key;
            a.bvals[o] = (V)val;
        }
    }
}

// Write the ring's slots [from, to) to the global band.
template <typename V>
__device__ __forceinline__ void flush(BandSmem &S, const BandArgs<V> &a, const Ctx &x, uint64_t from,
                                      uint64_t to, int lane) {
    __syncwarp();
    for (uint64_t s = from + lane; s < to; s += 32) {
        const Pivot e = S.ring[(uint32_t)s & kRingMask];
        const uint32_t v = (e.key & kValueMask) >> kValueBit;
        const uint32_t q = sizeof(V) <= 2 ? e.y : v;
        const uint32_t lo = __funnelshift_r(e.w0, e.w1, q), hi = __funnelshift_r(e.w1, e.w0, q);
        a.Cg[x.slot_base + s] = e.key ? ((uint64_t)hi << 32) | lo : 0ull;
        a.Yg[x.slot_base + s] = e.key ? (V)(sizeof(V) <= 2 ? v : e.y) : (V)0;
    }
    __syncwarp();
}

// The live row of staged row r, relative to the block that starts at offset o.
template <bool kPacked>
__device__ __forceinline__ void load_row(Row &R, const StagedRow &r, uint32_t o, uint32_t id) {
    const uint32_t q = r.o - o;              // < 32
    R.w0 = __funnelshift_l(r.hi, r.lo, q);   // the row rotated left by its start's position
    R.w1 = __funnelshift_l(r.lo, r.hi, q);
    R.y = kPacked ? 0u : r.y;
    R.gate = kFull << q;
    R.key = ((r.o + 1u) << kOffsetBit) | id | (kPacked ? r.y << kValueBit : 0u);
}

// The slots from the w-th on become the low bits of w0 (w <= 32).
__device__ __forceinline__ void rotate_row(Row &R, uint32_t w) {
    const uint32_t w0 = R.w0;
    R.w0 = __funnelshift_rc(w0, R.w1, w);
    R.w1 = __funnelshift_rc(R.w1, w0, w);
}

// Drop a live row of this bucket (old: of the one before) below threshold t.
__device__ __forceinline__ void drop_row(Row &R, bool old, uint32_t t) {
    if (R.key && (R.key >= kOldKey) == old && key_offset(R.key) < t) R.w0 = R.w1 = R.key = 0;
}

// Empty the ring's slots [from, from + n) held by rows of their own bucket below t.
__device__ __forceinline__ void drop_slots(BandSmem &S, uint32_t from, uint32_t n, uint32_t t, int lane) {
    __syncwarp();
    for (uint32_t i = lane; i < n; i += 32) {
        Pivot &e = S.ring[(from + i) & kRingMask];
        if (e.key && e.key < kOldKey && key_offset(e.key) < t) e.key = 0;
    }
    __syncwarp();
}


// If in is not 0: (w0, w1, y) ^= (p0, p1, py).  Predicated by hand: written as
// conditionals each XOR became a select besides.
__device__ __forceinline__ void xor_row(uint32_t in, uint32_t &w0, uint32_t &w1, uint32_t &y, uint32_t p0, uint32_t p1,
                                        uint32_t py) {
    asm("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t@p xor.b32 %0, %0, %4;\n\t@p xor.b32 %1, %1, %5;\n\t"
        "@p xor.b32 %2, %2, %6;\n\t}"
        : "+r"(w0), "+r"(w1), "+r"(y)
        : "r"(in), "r"(p0), "r"(p1), "r"(py));
}

// One slot: the live row of the highest key with bit `mask` is stored at `e`
// (place c of the block) and XORed into every other such row.  Without such a
// row every lane writes key 0 (an empty slot) and nothing changes.
//
// What a step costs (measured on the GB300, cycles of an SM quarter per warp
// instruction): LOP3, SEL, ISETP 2 each, max 1, warp maximum 2, shuffle 4,
// ballot 4, popc and find-first-bit 8, a 16-byte exchange through shared memory
// about 20.  So the pivot's lane comes out of the maximum itself (its low
// bits) instead of a ballot and a find-first, and the pivot travels by two
// shuffles (three with values of more than 16 bits); the whole step takes 36.5,
// 38.7 with the pivot stored by its own lane.
template <bool kPacked>
__device__ __forceinline__ void sweep_slot(Row &A, Row &B, uint32_t mask, unsigned slot, uint32_t c) {
    const uint32_t xa = A.w0 & A.gate & mask, xb = B.w0 & B.gate & mask;
    const uint32_t ka = xa ? A.key : 0u, kb = xb ? B.key : 0u;
    const bool second = kb > ka;
    const uint32_t s0 = second ? B.w0 : A.w0, s1 = second ? B.w1 : A.w1, sk = max(ka, kb),
                   sy = kPacked ? 0u : (second ? B.y : A.y);
    const uint32_t K = __reduce_max_sync(kFull, sk);
    const uint32_t p0 = __shfl_sync(kFull, s0, (int)K), p1 = __shfl_sync(kFull, s1, (int)K);
    const uint32_t py = kPacked ? K & kValueMask : __shfl_sync(kFull, sy, (int)K);
    // every lane has the pivot now and writes the same 16 bytes: cheaper than a store by its lane
    const uint32_t ek = kPacked || K == 0u ? K : K | c << kValueBit;
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(slot), "r"(p0), "r"(p1), "r"(ek), "r"(kPacked ? c : py));
    uint32_t &ya = kPacked ? A.key : A.y, &yb = kPacked ? B.key : B.y;
    xor_row(xa, A.w0, A.w1, ya, p0, p1, py);
    xor_row(xb, B.w0, B.w1, yb, p0, p1, py);
}

// The two warps of a partition meet.
__device__ __forceinline__ void pair_sync() { asm volatile("bar.sync 0, 64;" ::: "memory"); }

// The sweeping warp's state over its partition.
struct Sweep {
    Row A{0, 0, 0, 0, kFull}, B{0, 0, 0, 0, kFull};
    uint32_t o = 0;        // next offset of the bucket
    uint32_t t = 0;        // its threshold so far
    uint32_t it = 0;       // staged index of its first row at or above t
    uint32_t tprev = 0;    // the previous bucket's threshold
    uint32_t fa = kFull, fb = kFull;   // lanes whose row A, B is free
    __device__ __forceinline__ uint32_t nfree() const { return (uint32_t)(__popc(fa) + __popc(fb)); }
    __device__ __forceinline__ void find_free() {
        fa = __ballot_sync(kFull, A.key == 0);
        fb = __ballot_sync(kFull, B.key == 0);
    }
};

// Sweep offsets [W.o, lim) of the bucket at slot bB.  Returns false if the
// build has to end (the error is recorded).
template <typename V>
__device__ __forceinline__ bool sweep_to(BandSmem &S, const BandArgs<V> &a, Sweep &W, uint32_t lim, uint32_t bB,
                                         const StagedRow *rows, const uint32_t *first, uint32_t tstart, int lane) {
    constexpr bool kPacked = sizeof(V) <= 2;
    const LayerDesc &L = S.x.L;
    const uint32_t lt = (1u << lane) - 1u;
    Row &A = W.A, &B = W.B;
    auto unsolvable = [&]() {
        if (lane == 0) atomicOr(S.x.fail ? S.x.fail : a.err, kErrUnsolvable);
        return false;
    };
    const bool test_window = L.window != 0;
    uint32_t nfree = W.nfree(), i0, up;
    // first staged index of slot W.o, and (per lane) of the slot after W.o + lane.  The bookkeeping
    // between blocks (about ten per bucket) is kept short: i0 advances by the rows taken, and a row's
    // place among them tells whether it is taken (10^7 keys, 1+-bit: 6.46 -> 6.05 ms; 10^8 6.36 -> 6.22)
    auto look_ahead = [&](uint32_t o) { up = max(first[min(o + 1u + (uint32_t)lane, lim)], W.it); };
    auto look = [&](uint32_t o) {
        i0 = max(first[o], W.it);
        look_ahead(o);
    };
    look(W.o);
    while (W.o < lim) {
        const uint32_t o = W.o;
        // the rows that the lanes' free registers would take, read before the block's length is known
        const uint32_t ra = i0 + (uint32_t)__popc(W.fa & lt), rb = i0 + (uint32_t)(__popc(W.fa) + __popc(W.fb & lt));
        const StagedRow sa = rows[min(ra, (uint32_t)kStage - 1u)], sb = rows[min(rb, (uint32_t)kStage - 1u)];
        // the longest block of slots (up to 32) whose new rows fit the free registers, and their number
        const uint32_t w = (uint32_t)__popc(__ballot_sync(kFull, up - i0 <= nfree && o + (uint32_t)lane < lim));
        const uint32_t cnt = w ? __shfl_sync(kFull, up - i0, (int)w - 1) : 0u;
        // (one maximum over both, and the empty slots from the least key stored instead of the block's
        // keys: 6.46 -> 6.18 as well alone, but 10^8 keys 6.36 -> 6.47 and 10^9 47.7 -> 48.9 ms)
        if (w == 0) {
            // more than 64 rows in 64 slots: the lowest-offset row of the bucket goes
            if (L.fallback) return unsolvable();
            uint32_t low = o;
            if (A.key && A.key < kOldKey) low = min(low, key_offset(A.key));
            if (B.key && B.key < kOldKey) low = min(low, key_offset(B.key));
            W.t = threshold_from(L, __reduce_min_sync(kFull, low) + 1u);
            W.it = first[W.t];
            drop_row(A, false, W.t);
            drop_row(B, false, W.t);
            drop_slots(S, bB, o, W.t, lane);
            W.find_free();
            nfree = W.nfree();
            look(o);
            continue;
        }
        if (test_window && o < 64 && o + L.B >= L.window && __any_sync(kFull, max(A.key, B.key) >= kOldKey)) {
            // testing only: a row would be stored past the window that the test asked for
            if (lane == 0) atomicOr(a.err, kErrRingOverflow);
            return false;
        }
        if (cnt == 0 && nfree == 64) {   // no live row: empty slots
            if ((uint32_t)lane < w) S.ring[(bB + o + (uint32_t)lane) & kRingMask].key = 0;
            __syncwarp();   // the caller's lanes read other lanes' slots
            W.o += w;
            look_ahead(W.o);
            continue;
        }
        A.gate = B.gate = kFull;
        if (A.key == 0 && ra - i0 < cnt) load_row<kPacked>(A, sa, o, (uint32_t)lane);
        if (B.key == 0 && rb - i0 < cnt) load_row<kPacked>(B, sb, o, 1u << kRowBit | (uint32_t)lane);
        W.o += w;
        i0 += cnt;
        look_ahead(W.o);   // for the next block, during this one's sweep
        const Pivot *e = &S.ring[(bB + o) & kRingMask];
        const unsigned slot = (unsigned)__cvta_generic_to_shared(e);
        uint32_t c = 0;
#pragma unroll 1
        for (; c + kUnrollSlots <= w; c += kUnrollSlots) {
            const uint32_t mask = 1u << c;
#pragma unroll
            for (uint32_t k = 0; k < kUnrollSlots; ++k)
                sweep_slot<kPacked>(A, B, mask << k, slot + (c + k) * (unsigned)sizeof(Pivot), c + k);
        }
#pragma unroll 1
        for (; c < w; ++c) sweep_slot<kPacked>(A, B, 1u << c, slot + c * (unsigned)sizeof(Pivot), c);
        rotate_row(A, w);
        rotate_row(B, w);
        asm volatile("" ::: "memory");   // the slots' stores
        __syncwarp();
        // free registers: a live row that is zero was stored in this block, or it is dependent
        const bool za = (A.w0 | A.w1) == 0u, zb = (B.w0 | B.w1) == 0u;
        W.fa = __ballot_sync(kFull, za);
        W.fb = __ballot_sync(kFull, zb);
        const uint32_t np = (uint32_t)__popc(__ballot_sync(kFull, (uint32_t)lane < w && e[lane].key != 0));
        const uint32_t expect = nfree - cnt + np;
        nfree = W.nfree();
        if (nfree == expect) {
            if (za) A.key = 0;
            if (zb) B.key = 0;
            continue;
        }
        // the rows that were stored are free, which the block's keys tell the lanes (a shuffle per
        // slot instead took 1,000 cycles)
        const uint32_t K = (uint32_t)lane < w ? e[lane].key : 0u;
        if (lane < 16) reinterpret_cast<uint32_t *>(S.stored)[lane] = 0;
        __syncwarp();
        if (K) S.stored[(K & 31u) | (K >> kRowBit & 1u) << 5] = 1;
        __syncwarp();
        if (S.stored[lane]) A.key = 0;
        if (S.stored[32 + lane]) B.key = 0;
        const uint32_t D = __reduce_max_sync(kFull, max(za ? A.key : 0u, zb ? B.key : 0u));
        if (L.fallback) return unsolvable();
        if (D == 0 || (D >= kOldKey && o >= 64)) {   // not expected
            if (lane == 0) atomicOr(a.err, kErrRingOverflow);
            return false;
        }
        if (D < kOldKey) {
            W.t = threshold_from(L, key_offset(D) + 1u);
            drop_row(A, false, W.t);
            drop_row(B, false, W.t);
            drop_slots(S, bB, o + w, W.t, lane);
        } else {
            // the bucket before: bump its rows below the threshold above this row, and start this
            // bucket again without them
            W.tprev = threshold_from(L, key_offset(D) + 1u);
            Pivot s = S.snap[0][lane];
            A = Row{s.w0, s.w1, s.key, s.y, kFull};
            s = S.snap[1][lane];
            B = Row{s.w0, s.w1, s.key, s.y, kFull};
            drop_row(A, true, W.tprev);
            drop_row(B, true, W.tprev);
            S.snap[0][lane] = Pivot{A.w0, A.w1, A.key, A.y};
            S.snap[1][lane] = Pivot{B.w0, B.w1, B.key, B.y};
            drop_slots(S, bB - L.B, L.B, W.tprev, lane);
            W.t = tstart;
            W.o = 0;
        }
        W.it = first[W.t];
        W.find_free();
        nfree = W.nfree();
        look(W.o);
    }
    return true;
}

// What one warp pair works on: buckets [b0, b1) of its partition.
struct Run {
    uint32_t b0, b1;
    const Pivot *in = nullptr;   // live rows at b0 (64 of them); none: no live rows
    Pivot *out = nullptr;        // live rows at b1 go here
    bool compare = false;        // stop where the stored run over these buckets is met
};

// The partition (or segment's partition) of launch index gp; false if there is none.
template <typename V>
__device__ __forceinline__ bool load_ctx(BandSmem &S, const BandArgs<V> &a, uint64_t gp) {
    Ctx &x = S.x;
    if (a.bv.sd) {
        if (gp >= a.bv.nparts) return false;
        if (a.bv.part_order) gp = a.bv.part_order[gp];   // longest partitions first
        if (threadIdx.x == 0) {
            const uint32_t si = a.bv.part_struct[gp];
            const StructDesc &D = a.bv.sd[si];
            x.L = D.L;
            x.part = (uint32_t)(gp - D.part_base);
            x.bucket_base = D.bucket_base;
            x.slot_base = D.slot_base;
            x.tw_base = D.tw_base;
            x.out_base = D.out_base;
            x.bcount = a.bcount + si;
            x.fail = a.bv.fail ? a.bv.fail + si : nullptr;
        }
    } else {
        gp += a.L.part_lo;
        if (gp >= part_end(a.L)) return false;
        if (threadIdx.x == 0) {
            x.L = a.L;
            x.part = (uint32_t)gp;
            x.bucket_base = x.slot_base = x.tw_base = x.out_base = 0;
            x.bcount = a.bcount;
            x.fail = nullptr;
        }
    }
    if (threadIdx.x == 0) {
        x.b0 = (uint32_t)part_bucket(x.L, x.part);
        x.b1 = (uint32_t)part_bucket(x.L, x.part + 1);
        x.own_hi = part_own_hi(x.L, x.part);
        x.pend = a.bstart[x.bucket_base + x.b1];
        uint32_t slot;
        asm volatile("mov.u32 %0, %%warpid;" : "=r"(slot));
        S.sweeper = (slot >> 2) & 1u;
        // read once for the CTA: other CTAs may be setting it
        S.failed = (*a.err & (kErrRingOverflow | kErrUnsolvable)) || (x.fail && *x.fail);
    }
    __syncthreads();
    return true;
}

// Whether the rows that buckets before bucket b left live at its start (slot
// bB) span the same space, right-hand sides included, as those of the stored
// run.  Each run's pivots of these rows, which lie in the bucket's first 64
// slots, are an echelon basis of its space; `mine` and `theirs` are their slots.
template <typename V>
__device__ __forceinline__ bool same_space(BandSmem &S, const BandArgs<V> &a, uint64_t slot, uint32_t bB, uint64_t mine,
                                           uint64_t theirs, int lane) {
    if (mine != theirs) return false;
    uint64_t *c = reinterpret_cast<uint64_t *>(&S.snap[0][0]);        // the snapshot is not needed any more
    uint32_t *y = reinterpret_cast<uint32_t *>(c + 64);
    __syncwarp();
    for (int i = lane; i < 64; i += 32) {   // (the partition's slots reach at least 64 past its last bucket's start)
        const bool has = (theirs >> i) & 1ull;
        c[i] = has ? a.Cg[slot + i] << i : 0ull;
        y[i] = has ? (uint32_t)a.Yg[slot + i] : 0u;
    }
    __syncwarp();
    bool same = true;
    for (int i = lane; i < 64; i += 32) {
        if (!((mine >> i) & 1ull)) continue;
        const Pivot e = S.ring[(bB + (uint32_t)i) & kRingMask];
        const uint32_t v = (e.key & kValueMask) >> kValueBit, q = sizeof(V) <= 2 ? e.y : v;
        uint64_t w = ((uint64_t)__funnelshift_r(e.w1, e.w0, q) << 32 | __funnelshift_r(e.w0, e.w1, q)) << i;
        uint32_t z = sizeof(V) <= 2 ? v : e.y;
        for (int n = 0; w && n < 64; ++n) {   // each step clears the lowest bit, or there is no row for it
            const int p = __ffsll((long long)w) - 1;
            if (!c[p]) break;
            w ^= c[p];
            z ^= y[p];
        }
        same &= w == 0 && z == 0;
    }
    same = __all_sync(kFull, same);
    __syncwarp();
    return same;
}

// Band the buckets of a run.  One warp of the pair sweeps.  The other stages
// the next bucket's rows during the first 64 slots of a bucket, and during the
// rest writes out the bucket before, whose threshold and slots are final by
// then: done by the sweeping warp itself these were a quarter of its time per
// bucket.  Which warp sweeps alternates with the hardware warp slot: slots are
// dealt to the four SM quarters in turn, and with warp 0 sweeping everywhere
// the sweeps of an SM shared two of its quarters (layer-0 band of 10^8 keys
// 16.4 ms).
//
// kSeg: thresholds go to texact in either mode and no row is emitted
// (k_band_finish does both), and what a later run needs to meet this one is kept.
template <typename V, bool kSeg>
__device__ __forceinline__ uint32_t run_buckets(BandSmem &S, const BandArgs<V> &a, const Run &R, int lane) {
    const Ctx &x = S.x;
    const LayerDesc &L = x.L;
    const uint32_t b0 = R.b0, b1 = R.b1, Bs = L.B;
    if (kSeg) pair_sync();               // the run before is done with the ring
    if (threadIdx.x == 0) S.stop[0] = S.stop[1] = 0;
    pair_sync();

    if ((threadIdx.x >> 5) == S.sweeper) {
        Sweep W;
        if (kSeg && R.in) {
            Pivot s = R.in[lane];
            W.A = Row{s.w0, s.w1, s.key, s.y, kFull};
            s = R.in[32 + lane];
            W.B = Row{s.w0, s.w1, s.key, s.y, kFull};
            W.find_free();
        }
        pair_sync();   // the first bucket is staged
        // the last round, past the run's buckets, only finishes the rows of the last one
        for (uint32_t b = b0; b <= b1; ++b) {
            const uint32_t q = b & 1u, bB = b * Bs;   // (low 32 bits of the start slot)
            const uint32_t tstart = S.tstage[q];
            if (W.A.key) W.A.key |= kOldKey;
            if (W.B.key) W.B.key |= kOldKey;
            S.snap[0][lane] = Pivot{W.A.w0, W.A.w1, W.A.key, W.A.y};
            S.snap[1][lane] = Pivot{W.B.w0, W.B.w1, W.B.key, W.B.y};
            W.tprev = W.t;
            W.t = tstart;
            W.it = S.first[q][tstart];
            W.o = 0;
#pragma unroll 1
            for (uint32_t half = 0; half < 2; ++half) {
                const uint32_t lim = half == 0 ? 64u : (b < b1 ? Bs : 64u);
                uint32_t why = sweep_to(S, a, W, lim, bB, S.rows[q], S.first[q], tstart, lane) ? kRunDone : kRunError;
                if (kSeg && half == 0 && why == kRunDone) {
                    if (b < b1) {
                        const uint32_t k0 = S.ring[(bB + lane) & kRingMask].key, k1 = S.ring[(bB + 32 + lane) & kRingMask].key;
                        const uint64_t mine = (uint64_t)__ballot_sync(kFull, k1 >= kOldKey) << 32 |
                                              __ballot_sync(kFull, k0 >= kOldKey);
                        // one lane reads the stored mask and replaces it, so the store follows the
                        // read (other lanes' reads would have to be ordered before it)
                        uint64_t *om = a.omask + x.bucket_base + b;
                        if (R.compare) {
                            uint64_t theirs = 0;
                            if (lane == 0) theirs = *om;
                            theirs = __shfl_sync(kFull, theirs, 0);
                            if (same_space(S, a, x.slot_base + (uint64_t)b * Bs, bB, mine, theirs, lane)) why = kRunCoupled;
                        }
                        if (lane == 0 && why == kRunDone) *om = mine;
                    } else if (R.out) {
                        R.out[lane] = S.snap[0][lane];
                        R.out[32 + lane] = S.snap[1][lane];
                    }
                }
                if (lane == 0) {
                    if (half == 0) {   // (final then; the other warp reads it during the second half)
                        S.tdone = W.tprev;
                        S.at = b;
                    }
                    if (why) S.stop[half] = why;
                }
                pair_sync();
                if (S.stop[half]) return S.stop[half];
            }
        }
        return kRunDone;
    }

    uint64_t flushed = b0 == x.b0 ? part_own_lo(L, x.part) : (uint64_t)b0 * Bs;
    const uint64_t own_hi = b1 == x.b1 ? x.own_hi : (uint64_t)b1 * Bs;
    uint64_t tword = 0;
    uint32_t rs = a.bstart[x.bucket_base + b0];   // first equation of the next bucket to stage
    // packed records: the entry of hbase holds for 2^hshift buckets
    const bool packed = sizeof(V) == 1 && L.hbase;
    uint32_t bin = ~0u;
    uint64_t base = 0;
    auto stage = [&](uint32_t b) {
        if (packed && b >> L.hshift != bin) {
            bin = b >> L.hshift;
            base = L.hbase[bin];
        }
        const uint32_t q = b & 1u, re = a.bstart[x.bucket_base + b + 1];
        uint32_t t = 0;
        if (x.part > 0 && b == x.b0 && !L.fallback)
            t = L.mode == BURR_THRESH_1PLUS ? kW : L.levels[L.forced_code & 3];   // after a cut
        // the next bucket's equations are prefetched into L2
        if (lane < 16) {
            const uint32_t k = re + (uint32_t)lane * (128u / sizeof(uint64_t));
            if (k < x.pend) prefetch_l2(a.keys + k);
        } else if (lane < 24 && !packed) {
            const uint32_t k = re + (uint32_t)(lane - 16) * (128u / sizeof(V));
            if (k < x.pend) prefetch_l2(a.vals + k);
        }
        const uint32_t ts = stage_rows(S.rows[q], S.first[q], a, L, rs, re, b * Bs, t, packed, base, lane);
        if (lane == 0) S.tstage[q] = ts;
        rs = re;
        if (ts > t && L.fallback) {
            if (lane == 0) {
                atomicOr(x.fail ? x.fail : a.err, kErrUnsolvable);
                S.stop[0] = kRunError;
            }
        }
    };
    stage(b0);
    pair_sync();
    for (uint32_t b = b0; b <= b1; ++b) {
        if (b + 1 < b1) {
            stage(b + 1);
        } else {                       // nothing more: no rows
            for (int i = lane; i < 132; i += 32) S.first[(b + 1) & 1u][i] = 0;
            if (lane == 0) S.tstage[(b + 1) & 1u] = 0;
        }
        pair_sync();
        const uint32_t why = S.stop[0];
        if (why == kRunError) return why;
        if (b > b0) {
            const uint32_t bp = b - 1, t = S.tdone;
            const uint64_t end = min((uint64_t)b * Bs, own_hi);
            if (end > flushed) {
                flush(S, a, x, flushed, end, lane);
                flushed = end;
            }
            if (!L.fallback) {
                if (!kSeg && t > 0) emit_bumped(a, x, a.bstart[x.bucket_base + bp], a.bstart[x.bucket_base + b], bp * Bs, t, lane);
                if (kSeg || L.mode == BURR_THRESH_1PLUS) {
                    if (lane == 0) a.texact[x.bucket_base + bp] = (uint8_t)t;
                } else {
                    tword |= (uint64_t)code_of(L, t) << (2 * (bp & 31));
                    if ((b & 31u) == 0 || b == b1) {
                        if (lane == 0 && tword)
                            atomicOr((unsigned long long *)&a.thresh[x.tw_base + (bp >> 5)], (unsigned long long)tword);
                        tword = 0;
                    }
                }
            }
        }
        if (why) return why;           // the stored run goes on from here
        pair_sync();
        if (S.stop[1]) return S.stop[1];
    }
    if (own_hi > flushed) flush(S, a, x, flushed, own_hi, lane);
    return kRunDone;
}

// One partition per CTA, from its first bucket to its last.
template <typename V, int kCtas>
__global__ void __launch_bounds__(64, kCtas)
k_band(BandArgs<V> a) {
    __shared__ BandSmem S;
    if (!load_ctx(S, a, blockIdx.x)) return;
    Run R{S.x.b0, S.x.b1};
    run_buckets<V, false>(S, a, R, (int)(threadIdx.x & 31));
}

#include "burr_band_stream.cuh"

// Few partitions: each is banded in segments of a.seg buckets at the same time.
//
// A bucket's result depends on the buckets before it only through the rows
// they leave live at its start, as a space (of equations, right-hand sides
// included): thresholds are a property of sets, and any basis gives the same
// solution.  Runs that start from different live rows soon leave the same
// space (here: two runs from no live rows and from the true ones, over random
// start buckets of a layer at load 1.015, 2-bit thresholds: after 15 buckets in
// the median, 23 on average, 53 / 115 / 179 in 90 / 99 / 100% of 409 starts;
// 1+-bit thresholds 34 / 58 on average).  So
//   pass 0: every segment is banded from no live rows, and its live rows at the
//           end are kept;
//   pass 1: every segment but a partition's first is banded again from the rows
//           that pass 0 left before it, up to the bucket where it meets its own
//           stored run; a segment that never does leaves other rows than before;
//   pass 2..: the same for the segments behind those;
//   last:   one CTA per partition goes on behind what is left of them, in
//           order, each time until the stored run is met (rare, but then as
//           long as it takes).
// In the end every bucket's stored threshold and slots follow from true live
// rows, so the result does not depend on the segments.  k_band_finish then
// emits the bumped rows.
template <typename V>
__global__ void __launch_bounds__(64, kFewCtas)
k_band_seg(BandArgs<V> a, uint32_t nparts, uint32_t pass, bool last) {
    __shared__ BandSmem S;
    // the partition, its first segment, and the place of this one in it
    const bool table = a.bv.seg_first != nullptr;
    const uint32_t gp = last ? blockIdx.x : (table ? a.bv.seg_part[blockIdx.x] : blockIdx.x % nparts);
    const uint64_t base = table ? (uint64_t)a.bv.seg_first[gp] : (uint64_t)gp * a.nseg;
    const uint32_t i = last ? 0 : (table ? blockIdx.x - (uint32_t)base : blockIdx.x / nparts);
    const uint64_t g = base + i;
    const uint32_t now = pass & 1u, then = now ^ 1u;
    // (a partition's first segment starts from true rows; what a segment behind a partition's end
    // finds here does not matter)
    if (!last && pass > 0 && (i == 0 || (pass > 1 && (i == 1 || !a.moved[then][g - 1])))) {
        if (threadIdx.x == 0) a.moved[now][g] = 0;
        return;
    }
    if (!load_ctx(S, a, gp) || (pass > 0 && S.failed)) return;   // after a failure the stored runs are incomplete
    const int lane = (int)(threadIdx.x & 31);
    const uint32_t b0 = S.x.b0, b1 = S.x.b1, n = (b1 - b0 + a.seg - 1) / a.seg;
    if (!last) {
        if (i >= n) return;
        Run R{b0 + i * a.seg, min(b0 + (i + 1) * a.seg, b1)};
        if (i + 1 < n) R.out = a.state[now] + g * 64;
        if (pass > 0) {
            R.in = a.state[then] + (g - 1) * 64;
            R.compare = true;
        }
        const uint32_t why = run_buckets<V, true>(S, a, R, lane);
        if (threadIdx.x == 0) a.moved[now][g] = why == kRunDone;
        return;
    }
    for (uint32_t j = 2; j < n;) {
        if (!a.moved[then][base + j - 1]) {
            ++j;
            continue;
        }
        Run R{b0 + j * a.seg, b1};
        R.in = a.state[then] + (base + j - 1) * 64;
        R.compare = true;
        if (run_buckets<V, true>(S, a, R, lane) != kRunCoupled) return;
        j = (S.at - b0) / a.seg + 1;
    }
}

// After a segmented launch: emit the bumped rows of every bucket and pack the
// 2-bit codes.  One CTA per 32 buckets of a partition (aligned to the code words).
template <typename V>
__global__ void __launch_bounds__(128) k_band_finish(BandArgs<V> a, uint32_t nparts) {
    __shared__ BandSmem S;
    uint32_t gp = blockIdx.x % nparts, i = blockIdx.x / nparts;   // the partition and a word of its
    if (a.bv.seg_first) {   // those of its segments, and one more: its buckets may start inside a word
        const uint32_t per = a.seg / 32, words = a.bv.nsegs * per;
        gp = blockIdx.x < words ? a.bv.seg_part[blockIdx.x / per] : blockIdx.x - words;
        i = blockIdx.x < words ? blockIdx.x - a.bv.seg_first[gp] * per : (a.bv.seg_first[gp + 1] - a.bv.seg_first[gp]) * per;
    }
    if (!load_ctx(S, a, gp) || S.failed) return;
    const Ctx &x = S.x;
    const int lane = (int)(threadIdx.x & 31);
    const uint32_t warp = threadIdx.x >> 5;
    const uint32_t w = (x.b0 >> 5) + i, b = w * 32u + (uint32_t)lane;
    if (w * 32u >= x.b1) return;
    const uint32_t t = b >= x.b0 && b < x.b1 ? a.texact[x.bucket_base + b] : 0u;
    if (warp == 0 && x.L.mode != BURR_THRESH_1PLUS) {
        const uint64_t c = (uint64_t)code_of(x.L, t) << (2 * lane);
        const uint32_t lo = __reduce_or_sync(kFull, (uint32_t)c), hi = __reduce_or_sync(kFull, (uint32_t)(c >> 32));
        if (lane == 0 && (lo | hi))
            atomicOr((unsigned long long *)&a.thresh[x.tw_base + w], (unsigned long long)((uint64_t)hi << 32 | lo));
    }
    uint32_t left = __ballot_sync(kFull, t > 0);
    for (uint32_t k = 0; left; ++k, left &= left - 1) {   // the bumping buckets, dealt to the warps in turn
        if ((k & 3u) != warp) continue;
        const int j = __ffs((int)left) - 1;
        const uint32_t bj = w * 32u + (uint32_t)j, tj = __shfl_sync(kFull, t, j);
        emit_bumped(a, x, a.bstart[x.bucket_base + bj], a.bstart[x.bucket_base + bj + 1], bj * x.L.B, tj, lane);
    }
}

// Segments of a launch: buckets per segment (0: whole partitions) and segments
// of the longest partition.  A launch of few partitions is bound by their chains
// (512 buckets in a default partition) while most of the chip idles.  Segments of 32
// buckets are passed 2 to 6 times until the last one has met its stored run.  Layer-0
// band, ms, whole partitions / segments: 5*10^4 keys (1 partition) 3.2 / 0.71, 10^6 (16) 3.9 / 1.24,
// 10^7 (151, segments of 64) 4.2 / 1.88, 3*10^7 (451, segments of 128) 4.3 / 3.15.
// The passes bring about 23 buckets' work per segment, so a launch that fills the
// chip as it is keeps whole partitions: the segment length grows until segments and
// partitions together are at most kSegCap (2,128 CTAs are resident; caps of 1,216 / 2,128 / 2,432 / 3,648: 10^7 keys
// 1.85 / 1.88 / 1.88 / 2.39, 3*10^7 3.95 / 3.55 / 3.15 / 3.15).  With exact thresholds the right-hand
// sides of different bumped rows survive for 58 buckets on average, so segments pay
// with fewer of them: 5*10^4 keys 4.0 / 1.5, 10^6 6.2 / 4.0, 6*10^6 (91 partitions, segments of 128) 6.3 /
// 5.4, but 10^7 6.4 / 7.1.
constexpr uint64_t kSegCap = 2432, kSegMin = 32, kSegCapExact = 460, kSegMaxExact = 128;
// Passes before the last one: enough for runs that meet after 190 buckets.
inline uint32_t seg_passes(uint32_t seg) { return 1 + (190 + seg - 1) / seg; }
// A layer's partitions have nearly the same length, and each has as many segments
// in the launch's arrays as the longest.  Those of a batch may be one long and many
// short ones, so a batched launch has a table of segments: their number is at most
// partitions + buckets / segment length then, which kSegCap bounds (a product with
// the longest partition's took 2 GB for one structure of 4*10^6 keys among 1,000 of 100).
struct BandPlan {
    uint32_t seg = 0, nseg = 0;
    uint64_t parts = 0, buckets = 0, nsegs = 0;   // nsegs: of the launch
    bool sparse = false, stream = false;          // the stream beats the sweep of whole partitions, and segments too
};

// Which launches of sparse layers are streamed (burr_band_stream.cuh): estimates of
// a launch in us from the chain over its longest partition and the chip's
// throughput, in buckets of 128 slots.  Measured, r = 2, 2-bit thresholds, at loads
// 0.25 / 0.5 / 0.7 / 0.85 / 0.9 / 0.95:
//   stream   one warp alone 2.5 / 3.5 / 4.7 / 6.1 / 7.1 / 8.8 us per bucket, the chip full 1.4 / 1.9 / 2.6 / 3.8 / 4.4 / 5.7 ns
//   sweep    6.6 us, 5.5 to 5.9 ns; in segments 8.5 us per bucket of one segment, at any of these loads
// so the line lies at 0.87 (few partitions) to 0.95 (many).  Layer-0 band, ms, sweep / stream:
//   6*10^7 keys, partitions of 4,096 slots   - , 5.15 / 1.80, 3.76 / 1.74, 3.16 / 2.10, 3.01 / 2.29, 2.90 / 2.80
//   6*10^7 keys, default (964 to 1,832)      - , 7.24 / 2.17, 5.54 / 2.64, 4.32 / 3.37, 4.32 / 3.91, 4.38 / 4.93
//   2*10^7 keys, default, from 0.5 on in segments   5.43 / 1.38, 2.82 / 1.79, 1.51 / 2.24, 1.48 / 3.05, 1.52 / 3.55, 1.62 / 4.53
// Above kStreamLoad nothing is streamed: there many buckets are dependent.
constexpr double kStreamLoad = 1.0;
inline double band_us(double bucket_us, double longest, double bucket_ns, double buckets) {
    return std::hypot(bucket_us * longest, bucket_ns * 1e-3 * buckets);
}
inline double stream_us(double longest, double buckets, double load) {
    const double x = 1.0 / (1.1 - load);
    return band_us(1.1 + 1.27 * x, longest, 0.44 + 0.81 * x, buckets);
}

BandPlan band_plan(const LayerDesc &L, const BatchView *bv) {
    BandPlan p;
    uint64_t total, longest, moved = 0;   // moved: buckets by which searched cuts may lengthen a partition
    if (bv) {
        p.parts = bv->nparts;
        total = bv->nbuckets;
        longest = bv->max_len;
        p.buckets = bv->nbuckets;
    } else {
        p.parts = part_end(L) - L.part_lo;
        // partitions of P slots, the last one with the remainder; searched cuts move by less than P
        moved = L.K > 1 && L.cuts ? L.P / L.B : 0;
        longest = L.K <= 1 ? L.nb : std::max<uint64_t>(L.P / L.B, L.nb - (L.K - 1) * (L.P / L.B)) + moved;
        total = std::min<uint64_t>(L.nb, p.parts * longest);
        p.buckets = L.nb;
    }
    const uint32_t mode = bv ? bv->mode : L.mode;
    const bool fallback = bv ? bv->fallback : L.fallback != 0;
    const bool exact = mode == BURR_THRESH_1PLUS && !fallback;
    const uint64_t cap = exact ? kSegCapExact : kSegCap;
    uint64_t seg = kSegMin;
    while (p.parts + total / seg > cap && seg * 2 <= longest) seg *= 2;
    if (p.parts + total / seg > cap || seg * 2 > longest || (exact && seg > kSegMaxExact)) seg = 0;
    const double load = bv ? bv->load : L.load;
    if (load <= kStreamLoad) {
        const double len = (bv ? (double)bv->max_slots : (double)(longest - moved) * L.B) / 128.0;
        const double all = bv ? (double)total : (double)total * L.B / 128.0;
        const double us = stream_us(len, all, load);
        p.sparse = us < band_us(6.6, len, 5.7, all + 0.5 * (double)p.parts);   // (64 slots past each end)
        p.stream = seg ? us < band_us(8.5, (double)seg, 6.6, all) : p.sparse;
    }
    if (seg == 0 || p.stream) return p;
    p.seg = (uint32_t)seg;
    p.nseg = (uint32_t)((longest + seg - 1) / seg);
    p.nsegs = bv ? bv->nsegs : p.parts * p.nseg;
    return p;
}
inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

template <typename V>
cudaError_t band_impl(const LayerDesc &L, const uint64_t *keys, const V *vals, const uint32_t *bstart,
                      uint64_t *Cg, V *Yg, uint64_t *thresh, uint8_t *texact, uint64_t *bkeys, V *bvals,
                      unsigned long long *bcount, uint32_t *err, cudaStream_t st, const BatchView *bv, void *scratch) {
    BandArgs<V> a;
    if (bv) a.bv = *bv;
    a.L = L;
    a.keys = keys;
    a.vals = vals;
    a.bstart = bstart;
    a.Cg = Cg;
    a.Yg = Yg;
    a.thresh = thresh;
    a.texact = texact;
    a.bkeys = bkeys;
    a.bvals = bvals;
    a.bcount = bcount;
    a.err = err;
    const BandPlan p = band_plan(L, bv);
    if (p.stream || (p.sparse && !scratch)) {
        const bool exact = (bv ? bv->mode : L.mode) == BURR_THRESH_1PLUS;
        auto go = [&](auto *kernel) -> cudaError_t {
            const cudaError_t e = prefer_shared(kernel);
            if (e != cudaSuccess) return e;
            kernel<<<(unsigned)((p.parts + kStreamWarps - 1) / kStreamWarps), 32 * kStreamWarps, 0, st>>>(a);
            return cudaGetLastError();
        };
        return exact ? go(k_band_stream<V, true>) : go(k_band_stream<V, false>);
    }
    if (!scratch || !p.seg) {
        auto go = [&](auto *kernel) -> cudaError_t {
            const cudaError_t e = prefer_shared(kernel);
            if (e != cudaSuccess) return e;
            kernel<<<(unsigned)p.parts, 64, 0, st>>>(a);
            return cudaGetLastError();
        };
        // (a part of a split layer runs beside the rest, at its registers; a shard's range does as well)
        const bool whole = bv ? bv->slots != 0 : L.part_lo == 0 && L.part_hi == 0;
        return whole && p.parts <= kFewParts ? go(k_band<V, kFewCtas>) : go(k_band<V, kManyCtas>);
    }
    char *q = (char *)(((uintptr_t)scratch + 255) & ~(uintptr_t)255);   // (a caller's allocator gives the block)
    a.seg = p.seg;
    a.nseg = p.nseg;
    a.omask = (uint64_t *)q;
    q += align256(p.buckets * 8);
    for (int i = 0; i < 2; ++i) {
        a.state[i] = (Pivot *)q;
        q += align256(p.nsegs * 64 * sizeof(Pivot));
    }
    for (int i = 0; i < 2; ++i) {
        a.moved[i] = (uint32_t *)q;
        q += align256(p.nsegs * 4);
    }
    if (!a.texact) a.texact = (uint8_t *)q;
    const uint32_t parts = (uint32_t)p.parts;
    const bool fallback = bv ? bv->fallback : L.fallback != 0;
    cudaError_t e;
    if ((e = prefer_shared(k_band_seg<V>)) != cudaSuccess || (e = prefer_shared(k_band_finish<V>)) != cudaSuccess) return e;
    const uint32_t passes = seg_passes(p.seg), segs = (uint32_t)p.nsegs;
    for (uint32_t pass = 0; pass < passes; ++pass) k_band_seg<V><<<segs, 64, 0, st>>>(a, parts, pass, false);
    k_band_seg<V><<<parts, 64, 0, st>>>(a, parts, passes, true);
    // (a partition's buckets may start inside a code word)
    if (!fallback) k_band_finish<V><<<segs * (p.seg / 32) + parts * (bv ? 1u : 2u), 128, 0, st>>>(a, parts);
    return cudaGetLastError();
}

}  // namespace

uint32_t band_segment(const BatchView &bv) { return bv.nparts ? band_plan(LayerDesc(), &bv).seg : 0u; }

size_t band_scratch_bytes(const LayerDesc &L, const BatchView *bv) {
    if (bv ? bv->nparts == 0 : part_end(L) <= L.part_lo) return 0;
    const BandPlan p = band_plan(L, bv);
    if (!p.seg) return 0;
    return 256 + align256(p.buckets * 8) + align256(p.buckets) + 2 * align256(p.nsegs * 64 * sizeof(Pivot)) +
           2 * align256(p.nsegs * 4);
}

uint32_t band_kernel_count(const LayerDesc &L, const BatchView *bv) {
    if (band_scratch_bytes(L, bv) == 0) return 1u;
    return seg_passes(band_plan(L, bv).seg) + ((bv ? bv->fallback : L.fallback != 0) ? 1u : 2u);
}

cudaError_t launch_band(const LayerDesc &L, uint32_t vbytes, const uint64_t *keys, const void *vals,
                        const uint32_t *bucket_start, uint64_t *Cg, void *Yg, uint64_t *thresh, uint8_t *texact,
                        uint64_t *bumped_keys, void *bumped_vals, unsigned long long *bumped_count,
                        uint32_t *err, cudaStream_t st, const BatchView *bv, void *scratch) {
    if (bv ? bv->nparts == 0 : part_end(L) <= L.part_lo) return cudaSuccess;
    switch (vbytes) {
    case 1:
        return band_impl<uint8_t>(L, keys, (const uint8_t *)vals, bucket_start, Cg, (uint8_t *)Yg, thresh, texact,
                                  bumped_keys, (uint8_t *)bumped_vals, bumped_count, err, st, bv, scratch);
    case 2:
        return band_impl<uint16_t>(L, keys, (const uint16_t *)vals, bucket_start, Cg, (uint16_t *)Yg, thresh, texact,
                                   bumped_keys, (uint16_t *)bumped_vals, bumped_count, err, st, bv, scratch);
    default:
        return band_impl<uint32_t>(L, keys, (const uint32_t *)vals, bucket_start, Cg, (uint32_t *)Yg, thresh, texact,
                                   bumped_keys, (uint32_t *)bumped_vals, bumped_count, err, st, bv, scratch);
    }
}

}  // namespace burr
