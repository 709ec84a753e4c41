// burr_backsub.cu -- back-substitution ("Back Substitution" of Fig. 7): the
// table Z from the band.
#include <algorithm>

#include "burr_internal.cuh"

namespace burr {

namespace {

// Back-substitution, right to left over the partition's owned slots, one
// window per value bit: Z[i] = Y[i] ^ parity((C[i] >> 1) & Z[i+1 .. i+63]),
// Z[i] = 0 on empty slots (C = Y = 0 there).  The 64-bit register T holds Z of
// the 64 slots right of the current group (bit j = slot i+1+j); after a block
// of 64 slots it is exactly that block's table word for this bit plane.
//
// Four slots are solved per step so that the dependent chain is short: with
// c'_s = C[s] >> 1, the four parities against T are independent,
//   A_d = Y[i-d] ^ parity((c'_{i-d} >> d) & T),  d = 0..3,
// and the slots of the group then correct each other through the low bits of
// their own rows:
//   z_i = A_0,  z_{i-1} = A_1 ^ c'_{i-1}[0] z_i,
//   z_{i-2} = A_2 ^ c'_{i-2}[0] z_{i-1} ^ c'_{i-2}[1] z_i,
//   z_{i-3} = A_3 ^ c'_{i-3}[0] z_{i-2} ^ c'_{i-3}[1] z_{i-1} ^ c'_{i-3}[2] z_i,
//   T <- (T << 4) | z_i z_{i-1} z_{i-2} z_{i-3}.
constexpr int kBsWarps = 4;

__device__ __forceinline__ uint32_t parity64(uint64_t x) {
    return (uint32_t)__popc((uint32_t)x ^ (uint32_t)(x >> 32)) & 1u;
}

// Back-substitution with several partitions per warp: a partition needs only
// R lanes (R = r for one-byte values, one bit plane per lane; r / 2 or r / 4
// rounded up with 2 or 4 planes per lane for wider values), so a warp solves
// G = min(32 / R, kBsGroups) partitions side by side, lanes [q*R, q*R + R) on
// partition q.  For a batch, whose structures may differ in r, R comes from
// the widest value type (8 lanes); lanes past a structure's r sit out.  Each group runs the four-slot steps above; sharing each instruction
// among G partitions cuts the issue load G-fold, which matters because the
// solve runs beside the next layer's sort and band.  Partitions of one warp may
// differ in length: each walks its own blocks from the right, and a finished
// group idles until the longest one is done.
constexpr int kBsGroups = 8;

//
// kG (1, 2, 4 or 8) bounds G at compile time, so that the per-group registers
// of a launch with few groups (G = 4 at r = 8) are not those of eight.  A warp
// job is one set of G partitions; the grid may hold fewer warps than jobs
// (a cap on the CTAs per SM leaves room beside it for the next layer's
// kernels), and then every warp walks the jobs with the grid's stride.
//
// kPL bit planes per lane (1, 2 or 4; for r up to 8, 16, 32): lane k of a
// group solves planes k*kPL .. k*kPL + kPL - 1, each with its own window T, and
// the rows' reads, shifts and low bits serve all of them.  At r = 16 a group
// then needs 8 lanes instead of 16, so a warp takes 4 partitions instead of 2.
template <typename V, int kG, int kPL>
__global__ void __launch_bounds__(32 * kBsWarps, kG >= 8 ? 4 : 1)
k_backsub_multi(LayerDesc L0, const uint64_t *__restrict__ Cg, const V *__restrict__ Yg, uint64_t *__restrict__ Z0,
                BatchView bv, uint32_t R, uint32_t G, uint64_t njobs) {
    __shared__ __align__(16) uint64_t sc[kBsWarps][kG][64];
    __shared__ __align__(16) uint32_t sy[kBsWarps][kG][64];
    __shared__ uint64_t sbase[kBsWarps][kG];  // first slot of the group's structure in the layer arrays
    __shared__ uint64_t shi[kBsWarps][kG];    // one past the last block of the group's partition
    __shared__ uint32_t slen[kBsWarps][kG];   // its number of blocks
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t q = (uint32_t)lane / R, k = (uint32_t)lane % R;
    for (uint64_t job = (uint64_t)blockIdx.x * kBsWarps + warp; job < njobs;
         job += (uint64_t)gridDim.x * kBsWarps) {
    uint64_t gp = job * G + q + (bv.sd ? 0 : L0.part_lo);
    const uint64_t nparts = bv.sd ? bv.nparts : part_end(L0);
    uint64_t bhi = 0, base = 0;
    uint32_t len = 0, r = 0;
    uint64_t *Z = Z0;
    if (q < G && gp < nparts) {
        LayerDesc L;
        uint64_t part;
        if (bv.sd) {
            if (bv.part_order) gp = bv.part_order[gp];   // partitions of similar length share a warp
            const StructDesc &D = bv.sd[bv.part_struct[gp]];
            L = D.L;
            part = gp - D.part_base;
            base = D.slot_base;
            Z += D.z_base;
        } else {
            L = L0;
            part = gp;
        }
        const uint64_t lo = part_own_lo(L, part) >> 6, hi = part_own_hi(L, part) >> 6;
        if (hi > lo) {
            bhi = hi;
            len = (uint32_t)(hi - lo);
        }
        r = L.r;
    }
    if (q < G && k == 0) {
        sbase[warp][q] = base;
        shi[warp][q] = bhi;
        slen[warp][q] = len;
    }
    const uint32_t maxlen = __reduce_max_sync(0xffffffffu, len);
    __syncwarp();
    if (maxlen == 0) continue;
    uint64_t gh[kG], gb[kG];
    uint32_t gl[kG];
#pragma unroll
    for (int g = 0; g < kG; ++g) {
        gh[g] = (uint32_t)g < G ? shi[warp][g] : 0;
        gb[g] = (uint32_t)g < G ? sbase[warp][g] : 0;
        gl[g] = (uint32_t)g < G ? slen[warp][g] : 0;
    }
    // software pipeline: registers hold every group's next block while this one is solved
    uint64_t nc0[kG], nc1[kG];
    uint32_t ny0[kG], ny1[kG];
#pragma unroll
    for (int g = 0; g < kG; ++g) {
        nc0[g] = nc1[g] = 0;
        ny0[g] = ny1[g] = 0;
        if (gl[g] > 0) {
            const uint64_t s0 = gb[g] + ((gh[g] - 1) << 6);
            nc0[g] = Cg[s0 + lane];
            nc1[g] = Cg[s0 + lane + 32];
            ny0[g] = Yg[s0 + lane];
            ny1[g] = Yg[s0 + lane + 32];
        }
    }
    const bool solve = k * kPL < r;
    uint64_t T[kPL];
#pragma unroll
    for (int pl = 0; pl < kPL; ++pl) T[pl] = 0;
    for (uint32_t t = 0; t < maxlen; ++t) {
        __syncwarp();
#pragma unroll
        for (int g = 0; g < kG; ++g) {
            if (t < gl[g]) {
                sc[warp][g][lane] = nc0[g] >> 1;
                sc[warp][g][lane + 32] = nc1[g] >> 1;
                sy[warp][g][lane] = ny0[g];
                sy[warp][g][lane + 32] = ny1[g];
            }
        }
        __syncwarp();
#pragma unroll
        for (int g = 0; g < kG; ++g) {
            if (t + 1 < gl[g]) {
                const uint64_t s0 = gb[g] + ((gh[g] - 2 - t) << 6);
                nc0[g] = Cg[s0 + lane];
                nc1[g] = Cg[s0 + lane + 32];
                ny0[g] = Yg[s0 + lane];
                ny1[g] = Yg[s0 + lane + 32];
            }
        }
        if (solve && t < len) {
            const uint64_t *c = sc[warp][q];
            const uint32_t *yv = sy[warp][q];
#pragma unroll 4
            for (int g = 15; g >= 0; --g) {
                // slots 4g .. 4g+3 in three 16-byte shared reads
                const ulonglong2 clo = *reinterpret_cast<const ulonglong2 *>(c + 4 * g);
                const ulonglong2 chi = *reinterpret_cast<const ulonglong2 *>(c + 4 * g + 2);
                const uint4 yq = *reinterpret_cast<const uint4 *>(yv + 4 * g);
                const uint64_t c0 = chi.y, c1 = chi.x >> 1, c2 = clo.y >> 2, c3 = clo.x >> 3;
                const uint32_t l1 = (uint32_t)chi.x, l2 = (uint32_t)clo.y, l3 = (uint32_t)clo.x;
#pragma unroll
                for (int pl = 0; pl < kPL; ++pl) {
                    const uint32_t b = k * kPL + (uint32_t)pl;   // this plane's value bit
                    const uint32_t a0 = ((yq.w >> b) & 1u) ^ parity64(c0 & T[pl]);
                    const uint32_t a1 = ((yq.z >> b) & 1u) ^ parity64(c1 & T[pl]);
                    const uint32_t a2 = ((yq.y >> b) & 1u) ^ parity64(c2 & T[pl]);
                    const uint32_t a3 = ((yq.x >> b) & 1u) ^ parity64(c3 & T[pl]);
                    const uint32_t z0 = a0;
                    const uint32_t z1 = a1 ^ (l1 & z0);
                    const uint32_t z2 = a2 ^ ((l2 >> 1) & z0) ^ (l2 & z1);
                    const uint32_t z3 = a3 ^ ((l3 >> 2) & z0) ^ ((l3 >> 1) & z1) ^ (l3 & z2);
                    T[pl] = (T[pl] << 4) | (uint64_t)(((z0 << 3) | (z1 << 2) | (z2 << 1) | z3) & 15u);
                }
            }
#pragma unroll
            for (int pl = 0; pl < kPL; ++pl)
                if (k * kPL + (uint32_t)pl < r) Z[(bhi - 1 - t) * r + k * kPL + pl] = T[pl];
        }
    }
    __syncwarp();   // the warp's shared arrays are reused by its next job
    }
}

// ---------------------------------------------------------------------------
// Few partitions: the chain of a partition (1,024 blocks of 64 slots at about
// 2,950 cycles each in k_backsub_multi) sets the time.  Most of a block's work
// does not depend on the blocks to its right, so it is done first for all blocks
// at once: k_bs_reduce eliminates the block's own slots from its rows (row k
// into every row above it that has bit k, k from 63 down), after which
//   z_i = y'_i ^ parity(c'_i & Z_next)
// with the 64 slots of the next block only.  k_bs_chain then walks the blocks
// with one 64-bit parity per row and bit plane, all rows of a block at once
// (two per lane, a ballot per 32 rows is the new table word).
//
// The reduction costs 192 shuffles per block, so a launch of many partitions,
// which hides the chains behind each other, is faster without it.
// ---------------------------------------------------------------------------
constexpr int kRdWarps = 8;

// If bit `bit` (a one-bit mask) of `in` is set: (lo, hi, y) ^= (plo, phi, py).
__device__ __forceinline__ void take_row(uint32_t in, uint32_t bit, uint32_t &lo, uint32_t &hi, uint32_t &y, uint32_t plo,
                                         uint32_t phi, uint32_t py) {
    asm("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t@p xor.b32 %0, %0, %4;\n\t@p xor.b32 %1, %1, %5;\n\t"
        "@p xor.b32 %2, %2, %6;\n\t}"
        : "+r"(lo), "+r"(hi), "+r"(y)
        : "r"(in & bit), "r"(plo), "r"(phi), "r"(py));
}

template <typename V>
__global__ void __launch_bounds__(32 * kRdWarps) k_bs_reduce(uint64_t *__restrict__ Cg, V *__restrict__ Yg, uint64_t nblocks) {
    const int lane = threadIdx.x & 31;
    const uint64_t blk = (uint64_t)blockIdx.x * kRdWarps + (threadIdx.x >> 5);
    if (blk >= nblocks) return;
    uint64_t *c = Cg + blk * 64;
    V *y = Yg + blk * 64;
    const uint64_t ca = c[lane], cb = c[lane + 32];
    uint32_t ya = y[lane], yb = y[lane + 32];
    // the rows' bits inside the block (their own pivot bit left out) and right of it
    const uint64_t ia = (ca & ~1ull) << lane;
    const uint32_t a0 = (uint32_t)ia, a1 = (uint32_t)(ia >> 32), b1 = (uint32_t)((cb & ~1ull) << lane);
    const uint64_t ra = lane ? ca >> (64 - lane) : 0ull, rb = cb >> (32 - lane);
    uint32_t al = (uint32_t)ra, ah = (uint32_t)(ra >> 32), bl = (uint32_t)rb, bh = (uint32_t)(rb >> 32);
#pragma unroll 8
    for (int k = 31; k >= 0; --k) {       // row 32 + k
        const uint32_t pl = __shfl_sync(0xffffffffu, bl, k), ph = __shfl_sync(0xffffffffu, bh, k),
                       py = __shfl_sync(0xffffffffu, yb, k), bit = 1u << k;
        take_row(a1, bit, al, ah, ya, pl, ph, py);
        take_row(b1, bit, bl, bh, yb, pl, ph, py);
    }
#pragma unroll 8
    for (int k = 31; k > 0; --k) {        // row k
        const uint32_t pl = __shfl_sync(0xffffffffu, al, k), ph = __shfl_sync(0xffffffffu, ah, k),
                       py = __shfl_sync(0xffffffffu, ya, k);
        take_row(a0, 1u << k, al, ah, ya, pl, ph, py);
    }
    c[lane] = (uint64_t)ah << 32 | al;
    c[lane + 32] = (uint64_t)bh << 32 | bl;
    y[lane] = (V)ya;
    y[lane + 32] = (V)yb;
}

// One warp per partition and kChainPlanes bit planes.  kChainAhead blocks are
// on their way to shared memory (loads into registers were waited for together:
// 370 us for the 1,024 blocks of a default partition with 4 or 8 of them ahead).
// 1, 2, 4 and 8 planes per warp: 157, 196, 196, 259 us there, but 5.37, 5.30, 5.27, 5.24 ms per build
// at 3*10^7 keys, where it runs beside the next layer; 16 blocks ahead are no faster than 8.
constexpr int kChainPlanes = 4, kChainAhead = 8, kChainWarps = 4;

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(gmem) : "memory");
}

template <typename V>
struct alignas(16) ChainBlock {
    uint64_t c[64];
    V y[64];
};

template <typename V>
__global__ void __launch_bounds__(32 * kChainWarps)
k_bs_chain(LayerDesc L0, const uint64_t *__restrict__ Cg, const V *__restrict__ Yg, uint64_t *__restrict__ Z0,
           BatchView bv, uint32_t groups, uint64_t njobs) {
    __shared__ ChainBlock<V> ring[kChainWarps][kChainAhead];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t job = (uint64_t)blockIdx.x * kChainWarps + warp;
    if (job >= njobs) return;
    uint64_t gp = job / groups;
    const uint32_t k0 = (uint32_t)(job % groups) * kChainPlanes;
    uint64_t lo, hi, base = 0;
    uint32_t r;
    uint64_t *Z = Z0;
    if (bv.sd) {
        if (bv.part_order) gp = bv.part_order[gp];
        const StructDesc &D = bv.sd[bv.part_struct[gp]];
        const uint64_t part = gp - D.part_base;
        lo = part_own_lo(D.L, part) >> 6;
        hi = part_own_hi(D.L, part) >> 6;
        base = D.slot_base;
        Z += D.z_base;
        r = D.L.r;
    } else {
        gp += L0.part_lo;
        lo = part_own_lo(L0, gp) >> 6;
        hi = part_own_hi(L0, gp) >> 6;
        r = L0.r;
    }
    if (k0 >= r || hi <= lo) return;
    const uint64_t len = hi - lo;
    // a block in 16-byte copies: two rows per lane, and the right-hand sides by the first lanes
    const uint64_t *c = Cg + base + (hi - 1) * 64 + 2 * (uint64_t)lane;   // the rightmost block
    const char *y = (const char *)(Yg + base + (hi - 1) * 64) + 16 * lane;
    uint64_t *z = Z + (hi - 1) * r + k0 + lane;
    uint64_t next = 0;
    auto fetch = [&]() {
        if (next < len) {
            ChainBlock<V> &q = ring[warp][next % kChainAhead];
            cp_async16(&q.c[2 * lane], c);
            if (lane < (int)(4 * sizeof(V))) cp_async16((char *)q.y + 16 * lane, y);
            c -= 64;
            y -= 64 * sizeof(V);
        }
        ++next;
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll 1
    for (int u = 0; u < kChainAhead - 1; ++u) fetch();
    uint32_t wl[kChainPlanes], wh[kChainPlanes];
#pragma unroll
    for (int k = 0; k < kChainPlanes; ++k) wl[k] = wh[k] = 0;
    const bool writes = lane < kChainPlanes && k0 + (uint32_t)lane < r;
    for (uint64_t t = 0; t < len; ++t) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kChainAhead - 2) : "memory");
        __syncwarp();   // block t is here for every lane, and every lane is done with block t - 1
        const ChainBlock<V> &q = ring[warp][t % kChainAhead];
        const uint64_t ca = q.c[lane], cb = q.c[lane + 32];
        const uint32_t ya = (uint32_t)q.y[lane] >> k0, yb = (uint32_t)q.y[lane + 32] >> k0;
        fetch();        // into the place of block t - 1
        uint32_t ml = 0, mh = 0;
#pragma unroll
        for (int k = 0; k < kChainPlanes; ++k) {
            const uint32_t a = ((uint32_t)ca & wl[k]) ^ ((uint32_t)(ca >> 32) & wh[k]);
            const uint32_t b = ((uint32_t)cb & wl[k]) ^ ((uint32_t)(cb >> 32) & wh[k]);
            wl[k] = __ballot_sync(0xffffffffu, (__popc(a) ^ (ya >> k)) & 1u);
            wh[k] = __ballot_sync(0xffffffffu, (__popc(b) ^ (yb >> k)) & 1u);
            if (lane == k) {
                ml = wl[k];
                mh = wh[k];
            }
        }
        if (writes) *z = (uint64_t)mh << 32 | ml;
        z -= r;
    }
}

template <typename V>
cudaError_t backsub_blocks(const LayerDesc &L, uint64_t *Cg, V *Yg, uint64_t *Z, cudaStream_t st, const BatchView &v,
                           uint32_t rmax, uint64_t parts, uint64_t first_slot, uint64_t slots) {
    cudaError_t e;
    if ((e = prefer_shared(k_bs_reduce<V>)) != cudaSuccess || (e = prefer_shared(k_bs_chain<V>)) != cudaSuccess) return e;
    const uint64_t nblocks = slots / 64;
    k_bs_reduce<V><<<(unsigned)((nblocks + kRdWarps - 1) / kRdWarps), 32 * kRdWarps, 0, st>>>(Cg + first_slot, Yg + first_slot,
                                                                                            nblocks);
    const uint32_t groups = (rmax + kChainPlanes - 1) / kChainPlanes;
    const uint64_t jobs = parts * groups;
    k_bs_chain<V><<<(unsigned)((jobs + kChainWarps - 1) / kChainWarps), 32 * kChainWarps, 0, st>>>(L, Cg, Yg, Z, v, groups,
                                                                                                  jobs);
    return cudaGetLastError();
}

// Slots of a launch, and whether it reduces its blocks first (see k_bs_reduce).
// Without the reduction a launch takes about 1.1 us per block of its longest
// partition while the chip has room; with it 0.19 us and about 10 us per 10^6
// slots.  Layer-0 back-substitution with / without, in us: 5*10^4 keys (1
// partition) 138 / 928, 10^6 (16) 196 / 1103, 10^7 (151) 323 / 1105, 3*10^7 (451)
// 702 / 1194 (build 5.27 / 5.63 ms); at 10^8 keys (1504) the reduction took 1.96 ms
// beside layer 1 against 1.16 (build 11.0 / 10.25 ms).  The line lies between the
// last two for default partitions (1,024 blocks), and in proportion for others.
constexpr uint64_t kReduceSlotsPerBlock = 50000;
struct BsPlan {
    uint64_t parts, first, slots;
    bool blocks;
};
BsPlan bs_plan(const LayerDesc &L, const BatchView *bv) {
    BsPlan p{0, 0, 0, false};
    uint64_t longest;   // in blocks
    if (bv) {
        p.parts = bv->nparts;
        p.slots = bv->slots;                // 0: only some of the layer's partitions
        longest = bv->max_slots / 64;
    } else {
        if (part_end(L) <= L.part_lo) return p;
        p.parts = part_end(L) - L.part_lo;
        p.first = L.part_lo == 0 ? 0 : part_own_lo(L, L.part_lo);
        p.slots = (part_end(L) == L.K ? L.m : part_own_hi(L, part_end(L) - 1)) - p.first;
        longest = (L.K <= 1 ? L.m : L.P) / 64;
    }
    p.blocks = p.slots != 0 && p.slots <= longest * kReduceSlotsPerBlock;
    return p;
}

template <typename V, int kG, int kPL>
cudaError_t backsub_launch(const LayerDesc &L, const uint64_t *Cg, const V *Yg, uint64_t *Z, cudaStream_t st,
                           const BatchView &v, uint32_t R, uint32_t G, uint64_t njobs, unsigned grid) {
    const cudaError_t e = prefer_shared(k_backsub_multi<V, kG, kPL>);
    if (e != cudaSuccess) return e;
    k_backsub_multi<V, kG, kPL><<<grid, 32 * kBsWarps, 0, st>>>(L, Cg, Yg, Z, v, R, G, njobs);
    return cudaGetLastError();
}

// Planes per lane: one for values of a byte (r <= 8 lanes already fit four
// groups in a warp), else as many as the value's bytes.
template <typename V>
constexpr int planes_per_lane() {
    return sizeof(V) == 1 ? 1 : (int)sizeof(V);
}

template <typename V>
cudaError_t backsub_impl(const LayerDesc &L, const uint64_t *Cg, const V *Yg, uint64_t *Z, cudaStream_t st,
                         const BatchView &v, uint32_t R, uint32_t G, uint64_t njobs, unsigned grid) {
    constexpr int PL = planes_per_lane<V>();
    if (G <= 1) return backsub_launch<V, 1, PL>(L, Cg, Yg, Z, st, v, R, G, njobs, grid);
    if (G <= 2) return backsub_launch<V, 2, PL>(L, Cg, Yg, Z, st, v, R, G, njobs, grid);
    if (G <= 4) return backsub_launch<V, 4, PL>(L, Cg, Yg, Z, st, v, R, G, njobs, grid);
    return backsub_launch<V, kBsGroups, PL>(L, Cg, Yg, Z, st, v, R, G, njobs, grid);
}

}  // namespace

cudaError_t launch_backsub(const LayerDesc &L, uint32_t vbytes, uint64_t *Cg, void *Yg,
                           uint64_t *Z, cudaStream_t st, const BatchView *bv, uint32_t max_ctas_per_sm) {
    const BsPlan p = bs_plan(L, bv);
    const uint64_t parts = p.parts;
    if (parts == 0) return cudaSuccess;
    const BatchView v = bv ? *bv : BatchView();
    // (16-byte copies of the band: a caller's allocator may give less aligned blocks)
    if (p.blocks && (((uintptr_t)Cg | (uintptr_t)Yg) & 15u) == 0) {
        const uint32_t rmax = bv ? 8u * vbytes : L.r;
        switch (vbytes) {
        case 1: return backsub_blocks<uint8_t>(L, Cg, (uint8_t *)Yg, Z, st, v, rmax, parts, p.first, p.slots);
        case 2: return backsub_blocks<uint16_t>(L, Cg, (uint16_t *)Yg, Z, st, v, rmax, parts, p.first, p.slots);
        default: return backsub_blocks<uint32_t>(L, Cg, (uint32_t *)Yg, Z, st, v, rmax, parts, p.first, p.slots);
        }
    }
    const uint32_t pl = vbytes == 1 ? 1u : vbytes;
    const uint32_t R = bv ? 8u * vbytes / pl : (L.r + pl - 1) / pl;
    const uint32_t G = std::min<uint32_t>(32u / R, (uint32_t)kBsGroups);
    const uint64_t njobs = (parts + G - 1) / G;
    uint64_t grid = (njobs + kBsWarps - 1) / kBsWarps;
    if (max_ctas_per_sm) {
        int dev = 0, sms = 152;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        grid = std::min<uint64_t>(grid, (uint64_t)sms * max_ctas_per_sm);
    }
    switch (vbytes) {
    case 1: return backsub_impl<uint8_t>(L, Cg, (const uint8_t *)Yg, Z, st, v, R, G, njobs, (unsigned)grid);
    case 2: return backsub_impl<uint16_t>(L, Cg, (const uint16_t *)Yg, Z, st, v, R, G, njobs, (unsigned)grid);
    default: return backsub_impl<uint32_t>(L, Cg, (const uint32_t *)Yg, Z, st, v, R, G, njobs, (unsigned)grid);
    }
}

uint32_t backsub_kernel_count(const LayerDesc &L, const BatchView *bv) {
    return bs_plan(L, bv).blocks ? 2u : 1u;
}

}  // namespace burr
