// burr_band_stream.cuh -- the band of sparse layers (included by burr_band.cu):
// a warp inserts a bucket's rows as a stream, 32 at a time.
//
// The sweep pays for every slot, whether it gets a row or not, so its time per
// bucket hardly falls with the load (6.6 us for a warp alone, 5.5 to 6 ns with the
// chip full).  Here 32 lanes eliminate one row each and take their steps in
// lockstep, which pays for steps of elimination: at low loads most rows find
// their slot at once.  2*10^7 keys at load 0.25, partitions of 4,096 slots: layer-0
// band 0.90 ms, swept 3.46.  Both sides at other loads stand at the rule (band_plan).
//
//   * A set of rows is inserted together; its result does not depend on their
//     order (the kept rows are a property of the set, and so is the table).  The
//     whole bucket is one set, which mostly inserts.  If it is dependent it is
//     taken back and the rows at offsets >= the next threshold are tried, in 2-bit
//     mode level by level, in 1+-bit mode by bisection (a set is independent
//     whenever a larger one is).
//   * A step is one 128-bit compare-and-swap on the ring slot of the row's leading
//     bit: it claims the slot if that is empty, or returns the stored row to XOR
//     with.  The next kLook slots are read beside it, and elimination goes on
//     through those that hold stored rows.  Lanes whose row was stored take the
//     next rows of the set.
//   * The rows of a bucket have their pivots at most 190 slots past its start, so
//     a ring of 256 slots holds what is live; slots left behind are final.
// What bounds it: the chains of steps (barrier, reads, swap, elimination) of the 16
// warps that an SM holds at up to 128 registers a thread.

constexpr int kStreamWarps = 2;   // partitions (warps) per CTA
constexpr int kLook = 3;          // slots read ahead of the swap in a step (2: 3 to 5% slower where the chain bounds)

struct alignas(16) RingSlot {
    unsigned long long c;   // stored coefficient row (bit 0 = pivot), 0 = empty
    unsigned long long y;   // kStored | right-hand side; 0 = empty
};
constexpr unsigned long long kStored = 1ull << 32;

struct StreamSmem {
    RingSlot ring[kRing + kLook];   // live slots, and a pad for the reads ahead: zero, never written
    StagedRow rows[kStage];         // staged equations, ascending offset
    uint32_t first[132];            // first staged index of each offset (+ [128] = count)
    uint8_t list[kRing];            // ring slots stored by the current set
    uint32_t nlist;
    Ctx x;
};
static_assert(kRing <= 256, "the list holds ring slots in a byte");

enum { kSetIn = 0, kSetDependent = 1, kSetOverflow = 2 };

// If the slot is empty it becomes (c, y); its previous contents are returned.
__device__ __forceinline__ void slot_cas(unsigned addr, unsigned long long c, unsigned long long y, unsigned long long &oc,
                                         unsigned long long &oy) {
    asm volatile("{\n\t.reg .b128 d, b, v;\n\tmov.b128 b, {%2, %2};\n\tmov.b128 v, {%3, %4};\n\t"
                 "atom.shared.cas.b128 d, [%5], b, v;\n\tmov.b128 {%0, %1}, d;\n\t}"
                 : "=l"(oc), "=l"(oy)
                 : "l"(0ull), "l"(c), "l"(y), "r"(addr)
                 : "memory");
}

// Insert staged rows [lo, hi) into the band.  The slots stored are listed; nothing is taken back here.
__device__ int stream_set(StreamSmem &S, uint32_t lo, uint32_t hi, uint32_t bB, uint32_t wlim, int lane) {
    if (lane == 0) S.nlist = 0;
    if (hi <= lo) {
        __syncwarp();
        return kSetIn;
    }
    const unsigned lt = (1u << lane) - 1u;
    const unsigned ring0 = (unsigned)__cvta_generic_to_shared(&S.ring[0]);
    uint32_t nc = 0;                       // rows stored; as many more than 32 have been handed out
    bool has = lo + (uint32_t)lane < hi;
    // a lane without a row swaps (0, 0) in, which leaves every slot as it was
    unsigned long long cur = 0, y = 0;
    uint32_t pos = bB;
    if (has) {
        const StagedRow r = S.rows[lo + (uint32_t)lane];
        cur = (unsigned long long)r.hi << 32 | r.lo;
        y = kStored | r.y;
        pos = bB + r.o;
    }
    int result = kSetIn;
    for (;;) {
        const uint32_t ri = pos & kRingMask;
        const unsigned addr = ring0 + ri * (unsigned)sizeof(RingSlot);
        // The reads ahead come after the last step's swaps and before this one's, so a slot reads
        // as empty or as a stored row that stays.  The pivot lies below bB + wlim, so they stay
        // inside the window; past the ring's end they read the pad as empty.
        __syncwarp();
        uint32_t lcl[kLook], lch[kLook], ly[kLook];
#pragma unroll
        for (int j = 0; j < kLook; ++j)
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, _}, [%3];"
                         : "=r"(lcl[j]), "=r"(lch[j]), "=r"(ly[j])
                         : "r"(addr + (unsigned)((j + 1) * sizeof(RingSlot)))
                         : "memory");
        __syncwarp();
        unsigned long long oc, oy;
        slot_cas(addr, cur, y, oc, oy);
        // an empty slot is all zero and a stored row has its pivot bit set
        const bool stored = has && ((uint32_t)oc & 1u) == 0u;
        // the next rows are handed out first: their shared reads are in flight during the elimination
        const unsigned sm = __ballot_sync(kFull, stored);
        const uint32_t ci = nc + (uint32_t)__popc(sm & lt), nidx = lo + 32u + ci;
        const bool nhas = stored && nidx < hi;
        StagedRow nr = StagedRow{0u, 0u, 0u, 0u};
        if (nhas) nr = S.rows[nidx];
        if (stored) S.list[ci] = (uint8_t)ri;
        nc += (uint32_t)__popc(sm);
        // Elimination against the returned row, then through the slots read ahead.  The row is
        // (over : hi32 : lo32), bit j = slot pos + j; bit 0 is clear now.  Which rows are used
        // depends on the low word only; the other words are XORed afterwards, all at once.
        const bool act = has && !stored;
        uint32_t lo32 = (uint32_t)cur ^ (uint32_t)oc, hi32 = (uint32_t)(cur >> 32) ^ (uint32_t)(oc >> 32), over = 0;
        uint32_t y2 = (uint32_t)y ^ (uint32_t)oy;
        uint32_t go = 1u, um[kLook];   // go: bits 0 .. j - 1 are clear; um: all ones if the row of slot pos + j is used
#pragma unroll
        for (int j = 1; j <= kLook; ++j) {
            const uint32_t occ = lcl[j - 1] & 1u, bit = (lo32 >> j) & 1u;
            um[j - 1] = 0u - (go & bit & occ);
            lo32 ^= (lcl[j - 1] << j) & um[j - 1];
            go &= (bit ^ 1u) | occ;
        }
#pragma unroll
        for (int j = 1; j <= kLook; ++j) {
            hi32 ^= __funnelshift_l(lcl[j - 1], lch[j - 1], (unsigned)j) & um[j - 1];
            over ^= (lch[j - 1] >> (32 - j)) & um[j - 1];
            y2 ^= ly[j - 1] & um[j - 1];
        }
        // the leading bit (past bit 0) moves down to bit 0; it is almost always in the low word
        int tz = __ffs((int)lo32) - 1;
        uint32_t n0 = __funnelshift_r(lo32, hi32, (unsigned)tz), n1 = __funnelshift_r(hi32, over, (unsigned)tz);
        bool zero = false;
        if (act && lo32 == 0u) {
            zero = (hi32 | over) == 0u;
            if (hi32) {
                tz = 31 + __ffs((int)hi32);
                n0 = __funnelshift_r(hi32, over, (unsigned)(tz - 32));
                n1 = over >> (tz - 32);
            } else {
                tz = 63 + __ffs((int)over);
                n0 = over >> ((tz - 64) & 31);
                n1 = 0;
            }
        }
        const uint32_t npos = pos + (uint32_t)tz;
        const bool dep = act && zero, ovf = act && !zero && npos - bB >= wlim;
        if (act) {
            cur = (unsigned long long)n1 << 32 | n0;
            y = kStored | y2;
            pos = npos;
        }
        if (stored) {
            has = nhas;
            cur = (unsigned long long)nr.hi << 32 | nr.lo;
            y = nhas ? kStored | nr.y : 0ull;
            if (nhas) pos = bB + nr.o;
        }
        if (__ballot_sync(kFull, dep || ovf)) {
            result = __ballot_sync(kFull, ovf) ? kSetOverflow : kSetDependent;
            break;
        }
        if (!__ballot_sync(kFull, has)) break;
    }
    if (lane == 0) S.nlist = nc;
    __syncwarp();
    return result;
}

// Insert the staged rows of offsets [olo, ohi) as one set; a set that does not go in is taken back.
template <typename V>
__device__ int insert_set(StreamSmem &S, const BandArgs<V> &a, uint32_t olo, uint32_t ohi, uint32_t bB, int lane) {
    const uint32_t wlim = S.x.L.window ? min(S.x.L.window, (uint32_t)(kRing - kLook)) : (uint32_t)(kRing - kLook);
    const int rc = stream_set(S, S.first[olo], S.first[ohi], bB, wlim, lane);
    if (rc == kSetIn) return rc;
    const uint32_t n = S.nlist;
    for (uint32_t i = lane; i < n; i += 32) S.ring[S.list[i]] = RingSlot{0ull, 0ull};
    __syncwarp();
    if (rc == kSetOverflow && lane == 0) atomicOr(a.err, kErrRingOverflow);
    return rc;
}

// Write the ring's slots [from, to) to the global band and clear them.
template <typename V>
__device__ __forceinline__ void flush_stream(StreamSmem &S, const BandArgs<V> &a, const Ctx &x, uint64_t from, uint64_t to,
                                             int lane) {
    __syncwarp();
    for (uint64_t s = from + lane; s < to; s += 32) {
        RingSlot &e = S.ring[(uint32_t)s & kRingMask];
        a.Cg[x.slot_base + s] = e.c;
        a.Yg[x.slot_base + s] = (V)(uint32_t)e.y;
        e = RingSlot{0ull, 0ull};
    }
    __syncwarp();
}

// The partition of launch index gp, filled in by one lane; false if there is none.
// (load_ctx does the same for a CTA; shared, the sweep's kernels came out 1 to 2% slower.)
template <typename V>
__device__ __forceinline__ bool load_part(Ctx &x, const BandArgs<V> &a, uint64_t gp, bool leader) {
    uint32_t si = 0;
    if (a.bv.sd) {
        if (gp >= a.bv.nparts) return false;
        if (a.bv.part_order) gp = a.bv.part_order[gp];   // longest partitions first
        si = a.bv.part_struct[gp];
        gp -= a.bv.sd[si].part_base;
    } else {
        gp += a.L.part_lo;
        if (gp >= part_end(a.L)) return false;
    }
    if (!leader) return true;
    x.L = a.L;
    x.bucket_base = x.slot_base = x.tw_base = x.out_base = 0;
    x.fail = nullptr;
    if (a.bv.sd) {
        const StructDesc &D = a.bv.sd[si];
        x.L = D.L;
        x.bucket_base = D.bucket_base;
        x.slot_base = D.slot_base;
        x.tw_base = D.tw_base;
        x.out_base = D.out_base;
        if (a.bv.fail) x.fail = a.bv.fail + si;
    }
    x.bcount = a.bcount + si;
    x.part = (uint32_t)gp;
    x.b0 = (uint32_t)part_bucket(x.L, gp);
    x.b1 = (uint32_t)part_bucket(x.L, gp + 1);
    x.own_hi = part_own_hi(x.L, gp);
    x.pend = a.bstart[x.bucket_base + x.b1];
    return true;
}

// One partition per warp.  kExact: 1+-bit thresholds.
template <typename V, bool kExact>
__global__ void __launch_bounds__(32 * kStreamWarps, 8)
k_band_stream(BandArgs<V> a) {
    __shared__ StreamSmem smem[kStreamWarps];
    StreamSmem &S = smem[threadIdx.x >> 5];
    const int lane = (int)(threadIdx.x & 31);
    if (!load_part(S.x, a, (uint64_t)blockIdx.x * kStreamWarps + (threadIdx.x >> 5), lane == 0)) return;
    for (int i = lane; i < kRing + kLook; i += 32) S.ring[i] = RingSlot{0ull, 0ull};
    __syncwarp();
    const Ctx &x = S.x;
    const LayerDesc &L = x.L;
    const uint32_t b0 = x.b0, b1 = x.b1, Bs = L.B;
    const bool packed = sizeof(V) == 1 && L.hbase;
    const uint32_t *bst = a.bstart + x.bucket_base;
    uint64_t flushed = part_own_lo(L, x.part), tword = 0, base = 0;
    uint32_t rs = bst[b0], bin = ~0u;
    for (uint32_t b = b0; b < b1; ++b) {
        const uint32_t bB = b * Bs, re = bst[b + 1];   // (low 32 bits of the start slot)
        // the next bucket's equations are prefetched into L2
        if (lane < 16) {
            const uint32_t k = re + (uint32_t)lane * (128u / sizeof(uint64_t));
            if (k < x.pend) prefetch_l2(a.keys + k);
        } else if (lane < 24 && !packed) {
            const uint32_t k = re + (uint32_t)(lane - 16) * (128u / sizeof(V));
            if (k < x.pend) prefetch_l2(a.vals + k);
        }
        if (packed && b >> L.hshift != bin) {
            bin = b >> L.hshift;
            base = L.hbase[bin];
        }
        if ((uint64_t)b * Bs > flushed) {
            flush_stream(S, a, x, flushed, (uint64_t)b * Bs, lane);
            flushed = (uint64_t)b * Bs;
        }
        uint32_t forced = 0;
        if (x.part > 0 && b == b0 && !L.fallback) forced = kExact ? kW : L.levels[L.forced_code & 3];   // after a cut
        uint32_t t = forced;
        if (re > rs) {
            t = stage_rows(S.rows, S.first, a, L, rs, re, bB, forced, packed, base, lane);
            const int rc = L.fallback && t > forced ? kSetDependent : insert_set(S, a, t, Bs, bB, lane);
            if (rc == kSetOverflow) return;
            if (rc == kSetDependent) {
                if (L.fallback) {
                    if (lane == 0) atomicOr(x.fail ? x.fail : a.err, kErrUnsolvable);
                    return;
                }
                uint32_t fails = t, goes = Bs;   // the rows at offsets >= fails are dependent, those >= goes are in
                for (uint32_t k = 1; kExact ? goes - fails > 1 : k <= 2 && goes == Bs; ++k) {
                    // exact thresholds are mostly small: all but the lowest 16 offsets first, then halves
                    const uint32_t mid = !kExact ? L.levels[k] : (k == 1 && fails + 16 < goes ? fails + 16 : (fails + goes) >> 1);
                    if (!kExact && mid <= fails) continue;
                    const int rc2 = insert_set(S, a, mid, goes, bB, lane);
                    if (rc2 == kSetOverflow) return;
                    (rc2 == kSetIn ? goes : fails) = mid;
                }
                t = goes;
            }
            if (!L.fallback && t > 0) emit_bumped(a, x, rs, re, bB, t, lane);
        }
        rs = re;
        if (L.fallback) continue;
        if (kExact) {
            if (lane == 0) a.texact[x.bucket_base + b] = (uint8_t)t;
        } else {
            tword |= (uint64_t)code_of(L, t) << (2 * (b & 31));
            if ((b & 31u) == 31u || b + 1 == b1) {
                if (lane == 0 && tword) atomicOr((unsigned long long *)&a.thresh[x.tw_base + (b >> 5)], (unsigned long long)tword);
                tword = 0;
            }
        }
    }
    if (x.own_hi > flushed) flush_stream(S, a, x, flushed, x.own_hi, lane);
}
