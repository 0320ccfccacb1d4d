// Tensor-core GEMM for sm_103a: tcgen05.mma (kind::f16, bf16 operands, fp32
// accumulation in tensor memory), operands staged by TMA with 128-byte
// swizzle, warp-specialized (1 TMA producer warp, 1 MMA-issuing warp, 4
// epilogue warps).
//
// The GEMM is real: D[m][n] = sum_k A[m][k] B[n][k] with A and B "K-major"
// (rows contiguous in k).  Complex products and extra precision are both
// expressed through the operand layout.  It serves the gradient contraction
// Q_j = Gamma F_j in three planes (the elimination and the field sweeps have
// their own kernel, cgemm.cu):
//   * complex: A-row = [Re a, Im a], B-rows = [Re b, -Im b] (real part of the
//     output) and [Im b, Re b] (imaginary part), so a complex m x k x n product
//     is one real m x 2k x 2n product;
//   * precision: each operand is split into bf16 planes (x = x0 + x1 + x2);
//     the kernel walks "segments", one per retained plane product (x0 y0, x0 y1,
//     x1 y0, x0 y2, x1 y1, x2 y0), all accumulated in the same fp32
//     tensor-memory tile.
// Operand planes live in 3-D tensor maps (k, row, plane), so rows past the
// operand's end are zero-filled by TMA and no padding is needed in m or n.
#include "apf_internal.h"
#include "tc_gemm.h"
#include "tc_ptx.cuh"

#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <stdlib.h>
#include <string.h>

namespace {

using namespace tc;

template <int BN, int STAGES>
struct Layout {
    static constexpr int A_BYTES = BM * BK * 2;
    static constexpr int B_BYTES = BN * BK * 2;
    static constexpr int STAGE = A_BYTES + B_BYTES;
    static constexpr int BAR = STAGES * STAGE;
    static constexpr int TOTAL = BAR + (2 * STAGES + 4) * 8 + 16 + 1024;
};

// Epilogue of one 32-column chunk of one accumulator row.
__device__ __forceinline__ void store_chunk(const TcParams &p, int row, int col0, const uint32_t (&r)[32]) {
    if (row >= p.M) return;
    const bool whole = (col0 + 32 <= p.N) && ((col0 < p.n_cplx) == (col0 + 31 < p.n_cplx));
    float *dst = (col0 < p.n_cplx ? p.out_re + col0 : p.out_im + (col0 - p.n_cplx)) + (long long)row * p.ldo;
    if (whole && (((uintptr_t)dst) & 15) == 0) {
#pragma unroll
        for (int v = 0; v < 8; ++v)
            *reinterpret_cast<float4 *>(dst + 4 * v) = make_float4(__uint_as_float(r[4 * v]), __uint_as_float(r[4 * v + 1]),
                                                                   __uint_as_float(r[4 * v + 2]), __uint_as_float(r[4 * v + 3]));
        return;
    }
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        const int col = col0 + i;
        if (col >= p.N) break;
        (col < p.n_cplx ? p.out_re + col : p.out_im + (col - p.n_cplx))[(long long)row * p.ldo] = __uint_as_float(r[i]);
    }
}

// Persistent: one CTA per SM walks the output tiles (M index fastest, so the
// CTAs working on one B panel run together); two tensor-memory accumulators
// let the epilogue of one tile overlap the MMAs of the next.
template <int BN, int STAGES, int P>
__global__ void __launch_bounds__(192, 1) k_tc_gemm(const __grid_constant__ TcArgs<P> args) {
    using L = Layout<BN, STAGES>;
    const TcParams &p = args.p[0];  // shape and precision: the same for every problem
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *full = (uint64_t *)(smem + L::BAR);
    uint64_t *empty = full + STAGES;
    uint64_t *tfull = empty + STAGES;   // [2]
    uint64_t *tempty = tfull + 2;       // [2]
    uint32_t *tmem_slot = (uint32_t *)(tempty + 2);
    volatile int *abort_flag = (volatile int *)(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int Mt = (p.M + BM - 1) / BM, Nt = (p.N + BN - 1) / BN;
    const int ntl = Mt * Nt, ntiles = ntl * args.nprob;  // tiles of problem pr: [pr ntl, (pr + 1) ntl)
    const int total = p.nseg * p.kblocks;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], 4);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(2 * BN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;
    bool ok = true;
    int issued = 0;

    if (warp == 0) {
        if (lane == 0) {
            int it = 0;
            for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
                const int pr = tile / ntl, tt = tile - pr * ntl;
                const int m0 = (tt % Mt) * BM, n0 = (tt / Mt) * BN;
                const CUtensorMap *tmA = &args.a[pr], *tmB = &args.b[pr];
                for (int kk = 0; kk < total; ++kk, ++it) {
                    const int s = it % STAGES, r = it / STAGES;
                    if (!mbar_wait(&empty[s], (r & 1) ^ 1, abort_flag)) { ok = false; break; }
                    const int seg = kk / p.kblocks, kb = kk - seg * p.kblocks;
                    const int pa = (p.seg_pairs >> (4 * seg + 2)) & 3, pb = (p.seg_pairs >> (4 * seg)) & 3;
                    uint8_t *sa = smem + s * L::STAGE;
                    uint8_t *sb = sa + L::A_BYTES;
                    mbar_expect_tx(&full[s], L::A_BYTES + L::B_BYTES);
                    tma_load_3d(sa, tmA, &full[s], kb * BK, m0, pa);
                    tma_load_3d(sb, tmB, &full[s], kb * BK, n0, pb);
                    issued = it + 1;
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                                   ((uint32_t)(BM >> 4) << 24);
            int it = 0, tl = 0;
            for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x, ++tl) {
                const int b = tl & 1, u = tl >> 1;
                if (!mbar_wait(&tempty[b], (u & 1) ^ 1, abort_flag)) { ok = false; break; }
                fence_after();
                const uint32_t acc = tmem + (uint32_t)(b * BN);
                for (int kk = 0; kk < total; ++kk, ++it) {
                    const int s = it % STAGES, r = it / STAGES;
                    if (!mbar_wait(&full[s], r & 1, abort_flag)) { ok = false; break; }
                    fence_after();
                    const uint32_t sa = smem_u32(smem + s * L::STAGE);
                    const uint32_t sb = sa + L::A_BYTES;
#pragma unroll
                    for (int k4 = 0; k4 < BK / 16; ++k4)
                        mma_bf16(acc, sw128_desc(sa + k4 * 32), sw128_desc(sb + k4 * 32), idesc,
                                 (kk > 0 || k4 > 0) ? 1u : 0u);
                    mma_commit(&empty[s]);
                }
                if (!ok) break;
                mma_commit(&tfull[b]);
            }
            if (!ok) {
                // let the MMAs already issued drain before TMEM is freed
                mma_commit(&tfull[0]);
                mbar_wait(&tfull[0], 0, abort_flag, true);
            }
        }
    } else {
        const int q = warp & 3;  // TMEM lane quarter this warp may access
        int tl = 0;
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++tl) {
            const int b = tl & 1, u = tl >> 1;
            if (!mbar_wait(&tfull[b], u & 1, abort_flag)) { ok = false; break; }
            fence_after();
            const int pr = tile / ntl, tt = tile - pr * ntl;
            const int m0 = (tt % Mt) * BM, n0 = (tt / Mt) * BN;
            const int row = m0 + 32 * q + lane;
#pragma unroll 1
            for (int c = 0; c < BN; c += 32) {
                uint32_t r[32];
                tmem_ld32(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(b * BN + c), r);
                store_chunk(args.p[pr], row, n0 + c, r);
            }
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[b]);
        }
    }
    if (!ok) {
        *abort_flag = 1;
        for (int pr = 0; pr < args.nprob; ++pr)
            if (args.p[pr].flags) atomicOr(args.p[pr].flags, FLAG_TIMEOUT);
    }
    __syncwarp();
    // after a failure anywhere, wait (bounded) for the producer's copies in flight
    if (warp == 0 && lane == 0 && *abort_flag) {
        for (int it = issued > STAGES ? issued - STAGES : 0; it < issued; ++it)
            mbar_wait(&full[it % STAGES], (it / STAGES) & 1, abort_flag, true);
    }
    fence_before();
    __syncthreads();
    if (warp == 1) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * BN) : "memory");
    }
}

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

bool ensure_encode() {
    if (g_encode) return true;
    cudaDriverEntryPointQueryResult q;
    void *fn = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
            cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn) {
        cudaGetLastError();
        return false;
    }
    g_encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
    return true;
}

}  // namespace

// Tensor map of bf16 planes (k, row, plane): cols x rows x planes elements with
// the given row and plane pitches (in elements), box 64 x box_rows x box_planes,
// 128-byte swizzle; what lies outside is read as zero.
bool tc_make_map(CUtensorMap *m, const void *base, long long cols, long long rows, long long planes,
                 long long row_pitch, long long plane_pitch, int box_rows, int box_planes) {
    if (!ensure_encode()) return false;
    cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)planes};
    cuuint64_t strides[2] = {(cuuint64_t)row_pitch * 2, (cuuint64_t)plane_pitch * 2};
    cuuint32_t box[3] = {(cuuint32_t)BK, (cuuint32_t)box_rows, (cuuint32_t)box_planes};
    cuuint32_t es[3] = {1, 1, 1};
    CUresult r = g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, es,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

namespace {

template <int BN, int STAGES>
void set_attr() {
    cudaFuncSetAttribute(k_tc_gemm<BN, STAGES, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         Layout<BN, STAGES>::TOTAL);
    cudaFuncSetAttribute(k_tc_gemm<BN, STAGES, APF_MAX_BATCH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         Layout<BN, STAGES>::TOTAL);
}

}  // namespace

// Segment lists: (a plane, b plane) per retained product of split planes.
uint32_t tc_seg_pairs(int nsplit, int *nseg) {
    if (nsplit == 1) { *nseg = 1; return 0u; }
    if (nsplit == 2) {
        *nseg = 3;  // x0y0, x0y1, x1y0
        return (0u << 0) | ((0u << 2 | 1u) << 4) | ((1u << 2 | 0u) << 8);
    }
    *nseg = 6;  // + x0y2, x1y1, x2y0
    return (0u) | ((0u << 2 | 1u) << 4) | ((1u << 2 | 0u) << 8) | ((0u << 2 | 2u) << 12) | ((1u << 2 | 1u) << 16) |
           ((2u << 2 | 0u) << 20);
}

void tc_init_attrs() {
    set_attr<256, 4>();
    set_attr<128, 6>();
}

int tc_init() { return ensure_encode() ? APF_OK : APF_ECUDA; }

namespace {

template <int P, typename K>
cudaError_t launch_args(apf_ctx *c, K kern, unsigned grid, int smem, cudaStream_t s, const TcArgs<P> &args) {
    kern<<<grid, 192, smem, s>>>(args);
    c->launches++;
    return cudaGetLastError();
}

// Fill the tensor maps and parameters of nprob problems and launch the 128- or
// 256-wide tile kernel.
template <int P>
int launch_variant(apf_ctx *c, bool wide, int nprob, const TcProblem *pb, const TcParams &base, unsigned grid,
                   cudaStream_t s) {
    TcArgs<P> args;
    memset(&args, 0, sizeof args);
    args.nprob = nprob;
    for (int i = 0; i < nprob; ++i) {
        if (!tc_make_map(&args.a[i], pb[i].A.base, pb[i].A.kp, pb[i].A.rows, pb[i].A.planes, pb[i].A.kp,
                         pb[i].A.plane_pitch, BM, 1) ||
            !tc_make_map(&args.b[i], pb[i].B.base, pb[i].B.kp, pb[i].B.rows, pb[i].B.planes, pb[i].B.kp,
                         pb[i].B.plane_pitch, wide ? 256 : 128, 1))
            return set_err(c, APF_ECUDA, "tensor map encode failed (M=%d N=%d kp=%lld)", base.M, base.N, pb[i].A.kp);
        TcParams q = base;
        q.out_re = pb[i].out_re; q.out_im = pb[i].out_im;
        q.flags = pb[i].flags;
        args.p[i] = q;
    }
    cudaError_t e = wide ? launch_args(c, k_tc_gemm<256, 4, P>, grid, Layout<256, 4>::TOTAL, s, args)
                         : launch_args(c, k_tc_gemm<128, 6, P>, grid, Layout<128, 6>::TOTAL, s, args);
    if (e != cudaSuccess) return check_cuda(c, e, "tensor-core GEMM launch");
    return APF_OK;
}

}  // namespace

int tc_gemm_n(apf_ctx *c, int nprob, const TcProblem *pb, int nsplit, int M, int N, int n_cplx, long long ldo,
              cudaStream_t s) {
    if (M <= 0 || N <= 0 || nprob <= 0) return APF_OK;
    if (nprob > APF_MAX_BATCH) return set_err(c, APF_EINVAL, "tc_gemm_n: %d problems > %d", nprob, APF_MAX_BATCH);
    if (!ensure_encode()) return set_err(c, APF_ECUDA, "cuTensorMapEncodeTiled unavailable");
    for (int i = 0; i < nprob; ++i)
        if (pb[i].A.kp != pb[i].B.kp || pb[i].A.kp % BK != 0 || pb[i].A.kp != pb[0].A.kp)
            return set_err(c, APF_EINVAL, "tc_gemm: K mismatch (%lld vs %lld)", pb[i].A.kp, pb[i].B.kp);
    const long long kp = pb[0].A.kp;
    TcParams p{};
    p.M = M; p.N = N; p.n_cplx = n_cplx;
    p.kblocks = (int)(kp / BK);
    p.seg_pairs = tc_seg_pairs(nsplit, &p.nseg);
    p.ldo = ldo;
    // Tile width: score the wave utilisation of 256- and 128-wide tiles.
    static int num_sms = 0;
    if (!num_sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev);
        if (num_sms <= 0) num_sms = 148;
    }
    auto util = [&](int bn) {
        long long t = (long long)nprob * ((N + bn - 1) / bn) * ((M + BM - 1) / BM);
        long long waves = (t + num_sms - 1) / num_sms;
        return (double)t / (double)(waves * num_sms);
    };
    // 128 x 256 tiles need ~25% less L2->SM operand traffic per flop; take them
    // unless they waste much more of the last wave
    bool wide = (N > 128) && util(256) >= 0.7 * util(128);
    int bn = wide ? 256 : 128;
    long long ntiles = (long long)nprob * ((N + bn - 1) / bn) * ((M + BM - 1) / BM);
    // SMs left free for kernels of other streams: none by default, since the
    // library runs one solve at a time per GPU and a stream's kernels follow
    // each other (a caller that overlaps its own kernels may reserve some)
    static int reserve = -1;
    if (reserve < 0) {
        const char *e = getenv("APF_GEMM_RESERVED_SMS");  // tuning knob; default 0
        reserve = e ? atoi(e) : 0;
        if (reserve < 0 || reserve > num_sms / 2) reserve = 0;
        if (num_sms <= 64) reserve = 0;
    }
    unsigned grid = (unsigned)std::min<long long>(ntiles, num_sms - reserve);
    int pi = -1;
    if (c->prof_on && 2 * (c->prof_used + 1) <= (int)c->prof_ev.size()) {
        pi = c->prof_used++;
        // complex m x k x n product: M = m, N = 2n, kp ~ 2k real
        double alg = 2.0 * (double)M * (double)N * (double)kp * nprob;
        c->prof_alg[pi] = alg;
        c->prof_hw[pi] = alg * p.nseg;
        record_event(c, c->prof_ev[2 * pi], s);
    }
    int rc = nprob == 1 ? launch_variant<1>(c, wide, 1, pb, p, grid, s)
                        : launch_variant<APF_MAX_BATCH>(c, wide, nprob, pb, p, grid, s);
    if (rc != APF_OK) return rc;
    if (pi >= 0) record_event(c, c->prof_ev[2 * pi + 1], s);
    return APF_OK;
}
