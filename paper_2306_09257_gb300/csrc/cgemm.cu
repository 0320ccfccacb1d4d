// Complex tensor-core GEMM for sm_103a, C = alpha A B^T + beta C with A, B in
// split form (cgemm.h): tcgen05.mma (kind::f16, bf16 operands, float32
// accumulation in tensor memory), operands staged by TMA, one persistent CTA (or
// CTA pair, cta_group::2) per SM (pair), 1 TMA warp, 1 MMA warp, 8 epilogue warps.
//
// Real and imaginary parts are separate operand planes and separate
// accumulators of one tile, for each retained plane product:
//   one CTA:  [rr | ri] += Ar [Br; Bi],  [ir | ii] += Ai [Br; Bi],  re = rr - ii, im = ri + ir at the end;
//   a pair:   re += Ar Br, im += Ar Bi, re -= Ai Bi (negate bit), im += Ai Br.
// An operand is therefore stored and loaded once, not twice as in the real form
// [Re b, -Im b; Im b, Re b]: half the bytes of the stored slab inverses, and a
// sub-block of a larger matrix is an operand as it lies.  An MMA takes 64 clocks
// or more however narrow it is (the 128 rows of A are read from shared memory
// each time), so the one-CTA form joins Br and Bi, adjacent in shared memory, into
// one wide B: 24 MMAs of N = 128 per k block instead of 48 of N = 64.
//
// The epilogue writes what the next step reads: float32 planes, the split form,
// and both transposed, so no packing or transposing pass runs between the
// products of the recursion; and for a result known to be symmetric (Schur
// complements) it walks only the tiles that touch the lower triangle.
//
// Which form runs depends on K and on the row count the caller names, not on the
// number of problems in the launch, and a tile's width does not change the order
// of its sums: the bits of a result do not depend on what shares its launch.
#include "cgemm.h"
#include "tc_gemm.h"
#include "tc_ptx.cuh"

#include <algorithm>
#include <stdlib.h>
#include <string.h>

namespace {

using namespace tc;

constexpr int EPI_WARPS = 8, THREADS = 64 + 32 * EPI_WARPS;

struct CgParams {
    int M;
    CgOut o, t;
    const float *in_re, *in_im;
    long long ldi;
    int *flags;
};
template <int P>
struct CgArgs {
    CUtensorMap a[P], b[P];
    CgParams p[P];
    int nprob, N, Mt, Nt, ntl, kblocks, nseg, planes, sym, vec, t_block, passes;
    uint32_t seg_pairs;
    float alpha, beta;
};

// A kernel variant.  CG: CTAs per tile (2: a pair); BNC: complex columns of a
// tile; NQ: component tiles (plane, re / im) of each operand per stage, 4 (both
// planes, all three products from one stage) or 2 (one plane product per stage,
// any number of planes); CROSS: the cross products x0 y1 + x1 y0 in accumulators
// of their own, added in the epilogue.
// CROSS is for the field sweeps: the tensor cores truncate what they add to an
// accumulator, so its error grows with the number of additions at full
// magnitude; a third as many of them leaves a third of the error of a K = 4096
// product, and the sweeps (unlike the elimination, where it makes no difference)
// set how far one refinement sweep gets: 4096 x 260, two sweeps, residual 8e-11
// without and 2e-11 with it.  PASSES: for the same reason the pair tile adds up at
// most 16 k blocks in the tensor memory (and half of a product of up to 32), and the
// passes are added in registers; with one plane product per stage the smaller
// products are a pass of their own.  Residual of the first solve and after a sweep,
// time of an evaluation to 1e-10: 4096 x 260 in one pass 3.9e-4, 1.0e-7; passes of 32
// blocks 2.7e-4, 4.0e-8, 55.2 ms; of 16 2.1e-4, 1.7e-8, 55.8 ms; of 8 no better by more
// than a third, 57.1 ms.  8192 x 280: 32 blocks 3.9e-4, 1.1e-7, 274 ms; 16 blocks 3.2e-4,
// 4.6e-8, 278 ms.  Three planes, 4096 x 260: one pass 3.6e-4, 1.0e-7, 96.6 ms; 16 blocks
// 9.9e-5, 8.6e-9, 98.2 ms.
// MERGED: a product with fewer than 128 columns takes the tensor core as long as one
// with 128 (64 clocks per 16 of K), so the 128 x 32 tile multiplies x0 by both planes
// of y at once, which leaves the cross products in accumulators of their own: 4
// instead of 6 such products, 1100 instead of 1536 clocks per 64 of K.  The 128 x 64
// tile gives the same bits (which of the two runs depends on how many products share
// a launch), so one-CTA tiles of two planes always have CROSS.
// Shared memory per stage: 128 rows of A and the CTA's rows of B (all BNC, or half
// of them in a pair), 128 bytes each.  Tensor memory: an accumulator group is
// [rr | ri | ir | ii] (one CTA; MERGED: [rr | ri] and [ir | ii] of both groups side by
// side) or [re | im] (pair), a set one group or, with CROSS, two; two sets where
// they fit, so that the epilogue of a tile overlaps the products of the next, else
// the epilogue reads the whole set before its stores (HELD).
template <int CG, int BNC, int NQ, int CROSS>
struct CgLayout {
    static constexpr int STAGES = NQ == 4 ? 2 : 4;
    static constexpr int A_TILE = BM * BK * 2;
    static constexpr int B_ROWS = BNC / CG;
    static constexpr int B_TILE = B_ROWS * BK * 2;
    static constexpr int STAGE = NQ * (A_TILE + B_TILE);
    static constexpr int OUT = STAGES * STAGE;                // one 32 x 32 float block per epilogue warp
    static constexpr int BAR = OUT + EPI_WARPS * 32 * 32 * 4;
    static constexpr int TOTAL = BAR + (2 * STAGES + 4) * 8 + 16 + 1024;
    static constexpr int GROUP = (CG == 1 ? 4 : 2) * BNC;  // tensor-memory columns
    static constexpr int ACC = (CROSS ? 2 : 1) * GROUP;
    static constexpr int SETS = 2 * ACC <= 512 ? 2 : 1;
    static constexpr bool MERGED = CG == 1 && NQ == 4 && 4 * BNC <= 128;
    static constexpr bool PASSES = CG == 2 && (CROSS || NQ == 2);  // long sums in several passes
    static constexpr int HELD = SETS == 1 || PASSES ? BNC / 32 : 1;  // blocks of a tile read before the first is stored
    // offset of the accumulator of component q's first (x r..) or second (x i..) half in group g
    static constexpr int acc(int g, int i, int r) { return MERGED ? (4 * i + 2 * g + r) * BNC : g * GROUP + (2 * i + r) * BNC; }
    static constexpr int TMEM = SETS * ACC;
    static_assert(B_TILE % 1024 == 0, "B tiles must fill whole 128-byte swizzle atoms");
    static_assert(TMEM == 256 || TMEM == 512, "tensor-memory allocation");
    static_assert(!CROSS || NQ == 4, "cross accumulators need both planes in one stage");
};

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Split planes of (a, b), packed: a in the low half of w[p].
__device__ __forceinline__ void split2(float a, float b, int planes, uint32_t (&w)[3]) {
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        if (p >= planes) break;
        const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
        memcpy(&w[p], &h, 4);
        a -= __uint_as_float(w[p] << 16);
        b -= __uint_as_float(w[p] & 0xffff0000u);
    }
}

__device__ __forceinline__ void store_split(const Mirror &m, int q, int planes, long long r, long long c, float x) {
    uint32_t w[3];
    split2(x, 0.f, planes, w);
    for (int p = 0; p < planes; ++p)
        m.base[(2 * p + q) * m.qpitch + r * m.pitch + c] = __ushort_as_bfloat16((unsigned short)w[p]);
}

// Component q (0 re, 1 im) of a 32 x 32 block whose row `row` this lane holds, to
// the transposed output (t32: its float32 plane or null): neighbouring lanes exchange halves, so that a store covers
// two columns of 32 rows.
__device__ __forceinline__ void store_transposed(const CgOut &t, float *t32, int q, int planes, int row, int c0, int lane,
                                                 float (&v)[32]) {
    const bool odd = lane & 1;
    const long long col = c0 + (odd ? 16 : 0);
    const int r0 = row & ~1;
#pragma unroll
    for (int i = 0; i < 16; ++i) {  // v[i], v[i + 16] <- even and odd row of column col + i
        const float got = __shfl_xor_sync(0xffffffffu, odd ? v[i] : v[i + 16], 1);
        if (odd) v[i] = got;
        else v[i + 16] = got;
    }
    if (float *d = t32) {
        d += col * t.ld + r0;
#pragma unroll
        for (int i = 0; i < 16; ++i, d += t.ld) *reinterpret_cast<float2 *>(d) = make_float2(v[i], v[i + 16]);
    }
    if (t.m.base) {
        __nv_bfloat16 *d = t.m.base + q * t.m.qpitch + col * t.m.pitch + r0;
        const long long plane = 2 * t.m.qpitch;
#pragma unroll
        for (int i = 0; i < 16; ++i, d += t.m.pitch) {
            uint32_t w[3];
            split2(v[i], v[i + 16], planes, w);
#pragma unroll
            for (int p = 0; p < 3; ++p)
                if (p < planes) *reinterpret_cast<uint32_t *>(d + p * plane) = w[p];
        }
    }
}

// The rows of such a block from shared memory to the output, eight lanes per row
// (x[i]: this lane's four columns of row r0 + 4 i; rows at and past M are left out).
__device__ __forceinline__ void store_rows(const CgOut &o, int q, int planes, int r0, int M, int col, const float4 (&x)[8]) {
    if (float *d = q ? o.im : o.re) {
        d += (long long)r0 * o.ld + col;
#pragma unroll
        for (int i = 0; i < 8; ++i, d += 4 * o.ld)
            if (r0 + 4 * i < M) *reinterpret_cast<float4 *>(d) = x[i];
    }
    if (o.m.base) {
        __nv_bfloat16 *d = o.m.base + q * o.m.qpitch + (long long)r0 * o.m.pitch + col;
        const long long plane = 2 * o.m.qpitch;
#pragma unroll
        for (int i = 0; i < 8; ++i, d += 4 * o.m.pitch) {
            uint32_t w0[3], w1[3];
            split2(x[i].x, x[i].y, planes, w0);
            split2(x[i].z, x[i].w, planes, w1);
#pragma unroll
            for (int p = 0; p < 3; ++p)
                if (p < planes && r0 + 4 * i < M) *reinterpret_cast<uint2 *>(d + p * plane) = make_uint2(w0[p], w1[p]);
        }
    }
}

template <int CG, int BNC, int NQ, int CROSS, int P>
__global__ void __launch_bounds__(THREADS, 1) k_cgemm(const __grid_constant__ CgArgs<P> args) {
    using L = CgLayout<CG, BNC, NQ, CROSS>;
    constexpr int STAGES = L::STAGES, SETS = L::SETS;
    extern __shared__ uint8_t smem_raw[];
    // same offset in both CTAs of a pair: the MMA addresses both CTAs' tiles with one descriptor
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *full = (uint64_t *)(smem + L::BAR);
    uint64_t *empty = full + STAGES;
    uint64_t *tfull = empty + STAGES;  // [2]
    uint64_t *tempty = tfull + 2;      // [2]
    uint32_t *tmem_slot = (uint32_t *)(tempty + 2);
    volatile int *abort_flag = (volatile int *)(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = CG == 2 ? cluster_rank() : 0;
    const bool lead = (rank == 0);
    const int ntl = args.ntl, ntiles = ntl * args.nprob;  // tiles of problem pr: [pr ntl, (pr + 1) ntl)
    const int cid = (int)blockIdx.x / CG, ncl = (int)gridDim.x / CG;
    const int total = args.kblocks * (NQ == 4 ? 1 : args.nseg);
    const int passes = L::PASSES ? args.passes : 1;
    // first k step of pass ps: equal parts, but with one plane product per stage all the
    // smaller products together are the first pass
    auto pass_begin = [&](int ps) {
        if (NQ == 4 || !L::PASSES) return total * ps / passes;
        const int small = args.nseg > 1 ? 1 : 0;
        return ps < small ? 0 : total - args.kblocks * (passes - ps) / (passes - small);
    };
    // first row and column of tile tt (pair: of the whole 256-row tile); with
    // sym, row block mi has the column blocks up to its last row
    auto tile_at = [&](int tt, int &m0, int &n0) {
        constexpr int RATIO = CG * BM / BNC;
        int mi, ni;
        if (args.sym) {
            mi = 0;
            while (RATIO * (mi + 1) * (mi + 2) / 2 <= tt) ++mi;
            ni = tt - RATIO * mi * (mi + 1) / 2;
        } else {
            mi = tt % args.Mt;
            ni = tt / args.Mt;
        }
        m0 = mi * CG * BM;
        n0 = ni * BNC;
    };

    if (warp == 0 && lane == 0 && cid < ntiles) {
        prefetch_map(&args.a[cid / ntl]);
        prefetch_map(&args.b[cid / ntl]);
    }
    if (threadIdx.x == 32) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], EPI_WARPS * CG);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        if (CG == 2) {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                         "r"(L::TMEM)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                         "r"(L::TMEM)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
    }
    fence_before();
    if (CG == 2) cluster_sync();
    else __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;
    bool ok = true;
    int issued = 0;

    if (warp == 0) {
        if (lane == 0) {
            int it = 0;
            for (int t = cid; t < ntiles && ok; t += ncl) {
                const int pr = t / ntl;
                int m0, n0;
                tile_at(t - pr * ntl, m0, n0);
                m0 += (int)rank * BM;
                n0 += (int)rank * L::B_ROWS;
                const CUtensorMap *tmA = &args.a[pr], *tmB = &args.b[pr];
                for (int kk = 0; kk < total; ++kk, ++it) {
                    const int s = it % STAGES, r = it / STAGES;
                    if (!mbar_wait(&empty[s], (r & 1) ^ 1, abort_flag)) { ok = false; break; }
                    // one product per stage: the smallest products first (see CROSS)
                    const int sq = NQ == 4 ? 0 : kk / args.kblocks, kb = kk - sq * args.kblocks, seg = args.nseg - 1 - sq;
                    const int qa = NQ == 4 ? 0 : 2 * ((args.seg_pairs >> (4 * seg + 2)) & 3);
                    const int qb = NQ == 4 ? 0 : 2 * ((args.seg_pairs >> (4 * seg)) & 3);
                    uint8_t *sa = smem + s * L::STAGE;
                    uint8_t *sb = sa + NQ * L::A_TILE;
                    if (CG == 2) {
                        const uint32_t fb = lead ? smem_u32(&full[s]) : peer_addr(&full[s], 0);
                        if (lead) mbar_expect_tx(&full[s], 2 * L::STAGE);
                        tma_load_3d_pair(sa, tmA, fb, kb * BK, m0, qa);
                        tma_load_3d_pair(sb, tmB, fb, kb * BK, n0, qb);
                    } else {
                        mbar_expect_tx(&full[s], L::STAGE);
                        tma_load_3d(sa, tmA, &full[s], kb * BK, m0, qa);
                        tma_load_3d(sb, tmB, &full[s], kb * BK, n0, qb);
                    }
                    issued = it + 1;
                }
            }
        }
    } else if (warp == 1) {
        if (lead && lane == 0) {
            constexpr uint32_t base = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)((CG * BM) >> 4) << 24);
            constexpr uint32_t idesc = base | ((uint32_t)(BNC >> 3) << 17);
            constexpr uint32_t idesc_neg = idesc | (1u << 13);  // negate A
            constexpr uint32_t idesc_both = base | ((uint32_t)((2 * BNC) >> 3) << 17);
            int it = 0, tl = 0;
            for (int w = 0; w < passes * ((ntiles - cid + ncl - 1) / ncl) && ok; ++w, ++tl) {  // tiles times passes
                const int b = tl % SETS, u = tl / SETS;
                if (!mbar_wait(&tempty[b], (u & 1) ^ 1, abort_flag)) { ok = false; break; }
                fence_after();
                const uint32_t set = tmem + (uint32_t)(b * L::ACC);
                const int ps = w % passes, k0 = pass_begin(ps), k1 = pass_begin(ps + 1);
                for (int kk = k0; kk < k1; ++kk, ++it) {
                    const int s = it % STAGES, r = it / STAGES;
                    if (!mbar_wait(&full[s], r & 1, abort_flag)) { ok = false; break; }
                    fence_after();
                    const uint32_t sa = smem_u32(smem + s * L::STAGE), sb = sa + NQ * L::A_TILE;
                    if (L::MERGED) {
                        // x0 with both planes of y at once: [rr0 | ri0 | rr1 | ri1], [ir0 | ii0 | ir1 | ii1]
                        constexpr uint32_t idesc_all = base | ((uint32_t)((4 * BNC) >> 3) << 17);
#pragma unroll
                        for (int g = 0; g < 2; ++g) {  // x0 (y0, y1), x1 y0
                            const uint32_t ar = sa + 2 * g * L::A_TILE, ai = ar + L::A_TILE;
#pragma unroll
                            for (int k4 = 0; k4 < BK / 16; ++k4) {
                                const uint64_t dar = sw128_desc(ar + k4 * 32), dai = sw128_desc(ai + k4 * 32), db = sw128_desc(sb + k4 * 32);
                                const uint32_t acc = (kk > k0 || k4 > 0 || g > 0) ? 1u : 0u, to = set + 2 * g * BNC;
                                mma_bf16(to, dar, db, g ? idesc_both : idesc_all, acc);
                                mma_bf16(to + 4 * BNC, dai, db, g ? idesc_both : idesc_all, acc);
                            }
                        }
                    } else {
#pragma unroll
                    for (int g = 0; g < (NQ == 4 ? 3 : 1); ++g) {  // x0 y0, x0 y1, x1 y0
                        const uint32_t ar = sa + (g == 2 ? 2 : 0) * L::A_TILE, ai = ar + L::A_TILE;
                        const uint32_t br = sb + (g == 1 ? 2 : 0) * L::B_TILE, bi = br + L::B_TILE;
                        const uint32_t re = set + (CROSS && g > 0 ? L::GROUP : 0), im = re + BNC;
#pragma unroll
                        for (int k4 = 0; k4 < BK / 16; ++k4) {
                            const uint32_t acc = (kk > k0 || k4 > 0 || g > CROSS) ? 1u : 0u;
                            const uint64_t dar = sw128_desc(ar + k4 * 32), dai = sw128_desc(ai + k4 * 32);
                            const uint64_t dbr = sw128_desc(br + k4 * 32), dbi = sw128_desc(bi + k4 * 32);
                            if (CG == 2) {
                                mma_bf16_pair(re, dar, dbr, idesc, acc);
                                mma_bf16_pair(im, dar, dbi, idesc, acc);
                                mma_bf16_pair(re, dai, dbi, idesc_neg, 1u);
                                mma_bf16_pair(im, dai, dbr, idesc, 1u);
                            } else {
                                mma_bf16(re, dar, dbr, idesc_both, acc);            // [rr | ri]
                                mma_bf16(re + 2 * BNC, dai, dbr, idesc_both, acc);  // [ir | ii]
                            }
                        }
                    }
                    }
                    if (CG == 2) {
                        mma_commit_pair(smem_u32(&empty[s]));
                        mma_commit_pair(peer_addr(&empty[s], 1));
                    } else {
                        mma_commit(&empty[s]);
                    }
                }
                if (!ok) break;
                if (CG == 2) {
                    mma_commit_pair(smem_u32(&tfull[b]));
                    mma_commit_pair(peer_addr(&tfull[b], 1));
                } else {
                    mma_commit(&tfull[b]);
                }
            }
            if (!ok) {
                // let the MMAs already issued drain before the tensor memory is freed
                if (CG == 2) mma_commit_pair(smem_u32(&tfull[0]));
                else mma_commit(&tfull[0]);
                mbar_wait(&tfull[0], 0, abort_flag, true);
            }
        }
    } else {
        // A warp takes one component of its 32 rows, 32 columns at a time.  It holds
        // a row per lane, as the tensor memory hands them out; what goes to or comes
        // from memory along the rows passes through a block of shared memory (16-byte
        // cells, cell c of row r at c ^ (r % 8)), so that eight lanes share a row.
        // One lane per row instead: 10k clocks for a 128 x 32 tile, 20k where it
        // crosses the diagonal (element by element); like this 5.5k either way, which
        // is what 128 KB take at the 32 bytes per clock that the stores of an SM reach.
        const int q4 = warp & 3, q = (warp - 2) >> 2;  // tensor-memory lane quarter, component
        const bool use_beta = args.beta != 0.f, vec = args.vec != 0;
        const int planes = NQ == 4 ? 2 : args.planes;
        float *block = reinterpret_cast<float *>(smem + L::OUT) + (warp - 2) * 1024;
        auto cell = [&](int r, int c) { return reinterpret_cast<float4 *>(block + 32 * r + 4 * (c ^ (r & 7))); };
        const int sr = lane >> 3, sc = lane & 7;  // this lane's row (of four) and cell in the shared layout
        int tl = 0;
        for (int t = cid; t < ntiles; t += ncl, ++tl) {
            int b = 0;  // the set in use
            const int pr = t / ntl;
            const CgParams &p = args.p[pr];
            int m0, n0;
            tile_at(t - pr * ntl, m0, n0);
            const int row0 = m0 + (int)rank * BM + 32 * q4, row = row0 + lane;
            const float *in = q ? p.in_im : p.in_re;
            float *const o32 = q ? p.o.im : p.o.re;
            // the first block's beta input is fetched before the accumulator is waited for
            // (a single set: after it has been read, beside the next tile's products)
            float4 pre[8];
            auto fetch = [&](int c0) {
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int r = row0 + 4 * i + sr, c = c0 + 4 * sc;
                    const float *src = in + (long long)r * p.ldi + c;
                    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (r < p.M && c < args.N) {
                        if (vec) {
                            x = *reinterpret_cast<const float4 *>(src);
                        } else {
                            x.x = src[0];
                            if (c + 1 < args.N) x.y = src[1];
                            if (c + 2 < args.N) x.z = src[2];
                            if (c + 3 < args.N) x.w = src[3];
                        }
                    }
                    pre[i] = x;
                }
            };
            // one component of a block: rr - ii or ri + ir (pair: as accumulated), added to v
            auto read = [&](int c0, float (&v)[32], bool add) {
                const uint32_t ta = tmem + ((uint32_t)(32 * q4) << 16) + (uint32_t)(b * L::ACC + (c0 - n0));
#pragma unroll
                for (int g = 0; g <= CROSS; ++g) {
#pragma unroll
                    for (int hc = 0; hc < 32; hc += 16) {
                        uint32_t x[16], y[16];
                        tmem_ld16(ta + (q ? L::acc(g, 0, 1) : L::acc(g, 0, 0)) + hc, x);
                        if (CG == 1) tmem_ld16(ta + (q ? L::acc(g, 1, 0) : L::acc(g, 1, 1)) + hc, y);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            float z = __uint_as_float(x[i]);
                            if (CG == 1) z += q ? __uint_as_float(y[i]) : -__uint_as_float(y[i]);
                            v[hc + i] = add || g ? v[hc + i] + z : z;
                        }
                    }
                }
            };
            auto skip = [&](int c0) { return c0 >= args.N || row0 >= p.M || (args.sym && c0 > row0); };  // warp-uniform
            auto release = [&] {
                fence_before();
                __syncwarp();
                if (lane == 0) {
                    if (CG == 2) mbar_arrive_cluster(lead ? smem_u32(&tempty[b]) : peer_addr(&tempty[b], 0));
                    else mbar_arrive(&tempty[b]);
                }
            };
            if (L::HELD == 1 && use_beta && !skip(n0)) fetch(n0);
            float held[L::HELD][32];
            for (int ps = 0; ps < passes; ++ps) {
                const int use = tl * passes + ps;
                b = use % SETS;
                if (!mbar_wait(&tfull[b], (use / SETS) & 1, abort_flag)) { ok = false; break; }
                __syncwarp();
                fence_after();
                if (L::HELD > 1) {  // free the set for the next products before the stores
#pragma unroll
                    for (int i = 0; i < L::HELD; ++i)
                        if (!skip(n0 + 32 * i)) read(n0 + 32 * i, held[i], L::PASSES && ps > 0);
                    release();
                }
            }
            if (!ok) break;
            auto finish = [&](int c0, float (&v)[32]) {
#pragma unroll
                for (int i = 0; i < 32; ++i) v[i] *= args.alpha;
                if (use_beta) {
                    if (L::HELD > 1 || c0 > n0) fetch(c0);
#pragma unroll
                    for (int i = 0; i < 8; ++i) *cell(4 * i + sr, sc) = pre[i];
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float4 x = *cell(lane, i);
                        v[4 * i] += args.beta * x.x;
                        v[4 * i + 1] += args.beta * x.y;
                        v[4 * i + 2] += args.beta * x.z;
                        v[4 * i + 3] += args.beta * x.w;
                    }
                    __syncwarp();
                }
                const bool diagonal = args.sym && c0 == row0;
                float *const t32 = !args.t_block || c0 / args.t_block == row0 / args.t_block ? (q ? p.t.im : p.t.re) : nullptr;
                const bool cols = vec && c0 + 31 < args.N, whole = cols && row0 + 31 < p.M;
                if (o32 || p.o.m.base || !whole) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) *cell(lane, i) = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                    __syncwarp();
                    if (diagonal) {  // the block mirrored at its diagonal: no transposed store
#pragma unroll
                        for (int i = 1; i < 32; ++i)
                            if (i > lane) v[i] = block[32 * i + 4 * ((lane >> 2) ^ (i & 7)) + (lane & 3)];
                        __syncwarp();
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            *cell(lane, i) = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                        __syncwarp();
                    }
                    if (cols) {
                        float4 x[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) x[i] = *cell(4 * i + sr, sc);
                        store_rows(p.o, q, planes, row0 + sr, p.M, c0 + 4 * sc, x);
                    }
                    if (!whole && row < p.M && (!cols || t32 || p.t.m.base)) {  // ragged edges
#pragma unroll 1
                        for (int i = 0; i < 32 && c0 + i < args.N; ++i) {
                            const int col = c0 + i;
                            const float x = block[32 * lane + 4 * ((i >> 2) ^ (lane & 7)) + (i & 3)];
                            if (!cols) {
                                if (o32) o32[(long long)row * p.o.ld + col] = x;
                                if (p.o.m.base) store_split(p.o.m, q, planes, row, col, x);
                            }
                            if (diagonal) continue;
                            if (t32) t32[(long long)col * p.t.ld + row] = x;
                            if (p.t.m.base) store_split(p.t.m, q, planes, col, row, x);
                        }
                    }
                }
                if (!diagonal && whole && (t32 || p.t.m.base)) store_transposed(p.t, t32, q, planes, row, c0, lane, v);
                __syncwarp();
            };
            if (L::HELD > 1) {
#pragma unroll
                for (int i = 0; i < L::HELD; ++i)
                    if (!skip(n0 + 32 * i)) finish(n0 + 32 * i, held[i]);
            } else {
#pragma unroll 1
                for (int c0 = n0; c0 < n0 + BNC; c0 += 32) {
                    if (skip(c0)) continue;
                    read(c0, held[0], false);
                    finish(c0, held[0]);
                }
                release();
            }
        }
    }
    if (!ok) {
        *abort_flag = 1;
        for (int pr = 0; pr < args.nprob; ++pr)
            if (args.p[pr].flags) atomicOr(args.p[pr].flags, FLAG_TIMEOUT);
    }
    __syncwarp();
    // after a failure anywhere, wait (bounded) for the copies in flight (a pair's land on the even CTA's barriers)
    if (lead && warp == 0 && lane == 0 && *abort_flag) {
        for (int it = issued > STAGES ? issued - STAGES : 0; it < issued; ++it)
            mbar_wait(&full[it % STAGES], (it / STAGES) & 1, abort_flag, true);
    }
    fence_before();
    if (CG == 2) cluster_sync();
    else __syncthreads();
    if (warp == 1) {
        fence_after();
        if (CG == 2)
            asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(L::TMEM) : "memory");
        else
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(L::TMEM) : "memory");
    }
    if (CG == 2) cluster_sync();
}

// Two-SM tiles (APF_GEMM_PAIR=0: one-CTA tiles only).
bool pair_enabled() {
    static int v = -1;
    if (v < 0) {
        const char *e = getenv("APF_GEMM_PAIR");  // tuning knob; default on
        v = (e && e[0] == '0') ? 0 : 1;
    }
    return v == 1;
}

template <int CG, int BNC, int NQ, int CROSS, int P>
int launch_cg(apf_ctx *c, int nprob, const CgProblem *pb, CgArgs<P> &args, int M, int N, int K, int slots,
              cudaStream_t s) {
    using L = CgLayout<CG, BNC, NQ, CROSS>;
    for (int i = 0; i < nprob; ++i) {
        // K columns, not whole k blocks: what follows a sub-block in memory belongs to
        // its neighbour, and TMA fills the rest of the last k block with zeros
        if (!tc_make_map(&args.a[i], pb[i].A.base, K, pb[i].M, 2 * args.planes, pb[i].A.pitch, pb[i].A.qpitch, BM, NQ) ||
            !tc_make_map(&args.b[i], pb[i].B.base, K, N, 2 * args.planes, pb[i].B.pitch, pb[i].B.qpitch, L::B_ROWS, NQ))
            return set_err(c, APF_ECUDA, "tensor map encode failed (M=%d N=%d K=%d)", pb[i].M, N, K);
    }
    args.Mt = (M + CG * BM - 1) / (CG * BM);
    args.Nt = (N + BNC - 1) / BNC;
    constexpr int RATIO = CG * BM / BNC;
    args.ntl = args.sym ? RATIO * args.Mt * (args.Mt + 1) / 2 : args.Mt * args.Nt;
    const long long tiles = (long long)args.ntl * nprob;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(CG * std::min<long long>(tiles, slots)));
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = L::TOTAL;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = CG == 2 ? 1 : 0;
    cudaError_t e = cudaLaunchKernelEx(&cfg, k_cgemm<CG, BNC, NQ, CROSS, P>, args);
    if (e != cudaSuccess) return check_cuda(c, e, "tensor-core GEMM launch");
    c->launches++;
    return APF_OK;
}

template <int CG, int BNC, int NQ, int CROSS>
void set_attr() {
    constexpr int bytes = CgLayout<CG, BNC, NQ, CROSS>::TOTAL;
    cudaFuncSetAttribute(k_cgemm<CG, BNC, NQ, CROSS, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    cudaFuncSetAttribute(k_cgemm<CG, BNC, NQ, CROSS, CG_MAX_PROB>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

// How many SMs a launch may use, and how many two-CTA clusters can be resident
// at once (the SMs of a pair must share a GPC, so this can be below half).
void sm_slots(int *sms, int *pairs) {
    static int v = 0, p = 0;
    if (!v) {
        int dev = 0, n = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 148;
        // SMs left free for kernels of other streams: none by default, since the
        // library runs one solve at a time per GPU
        const char *e = getenv("APF_GEMM_RESERVED_SMS");  // tuning knob; default 0
        int reserve = e ? atoi(e) : 0;
        if (reserve < 0 || reserve > n / 2 || n <= 64) reserve = 0;
        using L = CgLayout<2, 128, 4, 0>;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(2);
        cfg.blockDim = dim3(THREADS);
        cfg.dynamicSmemBytes = L::TOTAL;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int q = 0;
        if (cudaOccupancyMaxActiveClusters(&q, k_cgemm<2, 128, 4, 0, 2>, &cfg) != cudaSuccess || q <= 0) {
            cudaGetLastError();
            q = n / 2;
        }
        p = std::max(1, std::min(q, (n - reserve) / 2));
        v = n - reserve;
    }
    *sms = v;
    *pairs = p;
}

template <int P>
int dispatch(apf_ctx *c, int nprob, const CgProblem *pb, int planes, int M, int N, int K, float alpha, float beta,
             bool sym, bool cross, int rows, cudaStream_t s) {
    CgArgs<P> args;
    memset(&args, 0, sizeof args);
    args.nprob = nprob;
    args.N = N;
    args.kblocks = (K + BK - 1) / BK;
    args.planes = planes;
    args.seg_pairs = tc_seg_pairs(planes, &args.nseg);
    args.alpha = alpha;
    args.beta = beta;
    args.sym = sym ? 1 : 0;
    args.t_block = pb[0].t_block;
    args.passes = std::max(2, args.kblocks / 16);  // see PASSES
    if (planes != 2 && args.nseg > 1) args.passes++;  // the smaller products
    bool vec = N % 16 == 0;
    for (int i = 0; i < nprob; ++i) {
        const CgProblem &q = pb[i];
        args.p[i] = CgParams{q.M, q.out, q.outT, q.in_re, q.in_im, q.ldi, q.flags};
        for (const CgOut *o : {&q.out, &q.outT}) {
            vec = vec && o->ld % 4 == 0 && o->m.pitch % 8 == 0 && o->m.qpitch % 8 == 0 &&
                  ((((uintptr_t)o->re) | ((uintptr_t)o->im) | ((uintptr_t)o->m.base)) & 15) == 0;
        }
        if (beta != 0.f) vec = vec && q.ldi % 4 == 0 && ((((uintptr_t)q.in_re) | ((uintptr_t)q.in_im)) & 15) == 0;
    }
    args.vec = vec ? 1 : 0;
    int sms, pairs;
    sm_slots(&sms, &pairs);
    if (planes != 2)
        return pair_enabled() && K >= 2048 && rows > BM ? launch_cg<2, 128, 2, 0, P>(c, nprob, pb, args, M, N, K, pairs, s)
                                        : launch_cg<1, 64, 2, 0, P>(c, nprob, pb, args, M, N, K, sms, s);
    // Pair tiles (256 x 128 over two SMs) for the long products of many rows: at
    // full load as fast per SM as the one-CTA 128 x 64 tile or faster, with half
    // its operand traffic (4096^3: 840 against 1043 us; 2048^3: 133 against 148);
    // below K = 2048 a product has too few of them to fill the chip (1024^3 took
    // 40 us with them, 26 with one-CTA tiles).  128 x 32 tiles, where they still go
    // in one round, take both planes of B at once and store sooner (512^3: 13.8 us,
    // 16.1 with 128 x 64 tiles).
    int kind = 1;
    if (pair_enabled() && K >= 2048 && rows > BM) {
        kind = 2;
    } else {
        const long long mt = (M + BM - 1) / BM, nt = (N + 31) / 32;
        if ((sym ? 2 * mt * (mt + 1) : mt * nt) * nprob <= sms) kind = 0;
    }
    if (kind == 0) return launch_cg<1, 32, 4, 1, P>(c, nprob, pb, args, M, N, K, sms, s);
    if (kind == 1) return launch_cg<1, 64, 4, 1, P>(c, nprob, pb, args, M, N, K, sms, s);
    return cross ? launch_cg<2, 128, 4, 1, P>(c, nprob, pb, args, M, N, K, pairs, s)
                 : launch_cg<2, 128, 4, 0, P>(c, nprob, pb, args, M, N, K, pairs, s);
}

}  // namespace

void cgemm_init_attrs() {
    set_attr<2, 128, 4, 0>();
    set_attr<1, 32, 4, 1>();
    set_attr<1, 64, 4, 1>();
    set_attr<2, 128, 4, 1>();
    set_attr<1, 64, 2, 0>();
    set_attr<2, 128, 2, 0>();
}

int cgemm_n(apf_ctx *c, int nprob, const CgProblem *pb, int planes, int M, int N, int K, float alpha, float beta,
            bool sym, bool cross, cudaStream_t s, int rows) {
    if (M <= 0 || N <= 0 || nprob <= 0) return APF_OK;
    if (nprob > CG_MAX_PROB) return set_err(c, APF_EINVAL, "cgemm_n: %d problems > %d", nprob, CG_MAX_PROB);
    int pi = -1;
    if (c->prof_on && 2 * (c->prof_used + 1) <= (int)c->prof_ev.size()) {
        pi = c->prof_used++;
        int nseg = 0;
        tc_seg_pairs(planes, &nseg);
        double rows = 0.0;
        for (int i = 0; i < nprob; ++i) rows += pb[i].M;
        // one complex multiply-add = 8 flops; of a symmetric result only one triangle is needed
        const double alg = 8.0 * rows * (sym ? 0.5 * (N + 1) : (double)N) * K;
        c->prof_alg[pi] = alg;
        c->prof_hw[pi] = alg * nseg;
        record_event(c, c->prof_ev[2 * pi], s);
    }
    const int rc = nprob <= 2 ? dispatch<2>(c, nprob, pb, planes, M, N, K, alpha, beta, sym, cross, rows > 0 ? rows : M, s)
                              : dispatch<CG_MAX_PROB>(c, nprob, pb, planes, M, N, K, alpha, beta, sym, cross, rows > 0 ? rows : M, s);
    if (rc != APF_OK) return rc;
    if (pi >= 0) record_event(c, c->prof_ev[2 * pi + 1], s);
    return APF_OK;
}
