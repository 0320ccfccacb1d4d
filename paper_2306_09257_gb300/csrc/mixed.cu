// Mixed-precision slab elimination and float64 iterative refinement.
//
// The slab Schur blocks X_j and their inverses G_j are held in float32
// (separate real / imaginary planes).  Every product runs on the tensor cores
// (cgemm.cu) with operands split into bf16 planes: two planes and three
// products ("bf16x3") for the elimination and the field sweeps, three planes
// and six products for the gradient contraction (tc_gemm.cu).  Accuracy is then
// won back by float64 iterative refinement of the slab fields:
//     r = R - K E (float64 5-point stencil + boundary circulants),
//     E <- E + Khat^-1 r,
// where Khat^-1 is the block-LU solve with the stored low-precision G_j.
//
// The slab rows are eliminated from both ends towards the middle row m = h / 2:
// X_j = K_j - G_{j-1} below it, X_j = K_j - G_{j+1} above it, X_m = K_m - G_{m-1} -
// G_{m+1}.  The two chains are independent, so one launch carries a row of each
// (of every design of a batch): half as many dependent steps, which is what a
// single design's time consists of (four CTAs per 128 x 128 diagonal block, a few
// tiles per product of the lower recursion levels).
#include "apf_internal.h"
#include "cgemm.h"
#include "tc_gemm.h"
#include "leaf.cuh"

#include <algorithm>
#include <complex>
#include <stdio.h>
#include <stdlib.h>
#include <vector>

// Work arrays of one of the two chains of a design.
struct SideWork {
    float *Xre = nullptr, *Xim = nullptr;  // n x n working block
    Mirror XP;                             // its split form
    __nv_bfloat16 *TP = nullptr, *TT = nullptr;  // T and T^T of every recursion level, split
    float *O32 = nullptr;                  // field products (re, im), ncol x n each
    Mirror PA;                             // field operand, ncol x n
};

struct MixedWork {
    int nsplit_elim = 2, nsplit_grad = 3, leaf = 128, leaf_variant = 0;
    int nside = 2;                                   // 1 with recomputation
    SideWork sd[2];
    __nv_bfloat16 *GA = nullptr, *GB = nullptr;      // gradient operands
    __nv_bfloat16 *GP = nullptr;                     // split G_j: h of them, or seg_rows when recomputing
    long long gp_stride = 0;
    // Recomputation of the slab Schur blocks (seg_rows > 0).  The rows are taken
    // in the order of the chains (lower chain, upper chain, middle row), cut into
    // segments of seg_rows positions; only the split inverses of one segment are
    // held (GP slot = position mod seg_rows), plus the float32 inverse before
    // every segment start (checkpoint s - 1 for segment s), from which a
    // segment's inverses are recomputed when a sweep needs them, and that of the
    // lower chain's last row (CKB), which the middle row needs again.
    int seg_rows = 0, nseg = 1, seg_loaded = -1;
    float *CK = nullptr, *CKB = nullptr;             // 2 n^2 floats per checkpoint
    // Symmetric random butterfly transform of every slab block before its
    // inversion (bfly = 1): X' = U^T X U, G = U X'^-1 U^T with a depth-2
    // recursive butterfly U; BW holds its 2 n random diagonal entries.
    int bfly = 0;
    float *BW = nullptr;
    double2 *r = nullptr, *delta = nullptr;          // refinement buffers (h*ncol*nx)
    double2 *cb = nullptr, *ct = nullptr;            // circulant products on the boundary rows
    double *rnorm = nullptr;                         // ||R_c||^2, ||r_c||^2
    double *rpart = nullptr;                         // partial sums of ||r_c||^2
    int km = 0;                                      // GMRES(km) refinement (0: plain refinement)
    double2 *KV = nullptr, *KZ = nullptr;            // Krylov basis (km+1 fields) and preconditioned vectors (km)
    double2 *kdot = nullptr, *ky = nullptr;          // Gram-Schmidt coefficients (km+1)*km*ncol, update km*ncol
    double *knrm = nullptr;                          // ||W_c||^2 per Arnoldi step, km*ncol
    std::vector<void *> allocs;
};

namespace {
struct Bat;
}
int recompute_segment_b(const Bat &bt, int seg, cudaStream_t s);

namespace {

// Per-problem pointers of a launch (entry blockIdx.z, or blockIdx.x for the
// one-CTA-per-block leaf kernels); a single problem uses entry 0.
template <typename T>
struct Tab {
    T v[CG_MAX_PROB];
};

__device__ __forceinline__ void split_bf16(float x, int nsplit, __nv_bfloat16 *o) {
    __nv_bfloat16 h0 = __float2bfloat16_rn(x);
    o[0] = h0;
    if (nsplit > 1) {
        float x1 = x - __bfloat162float(h0);
        __nv_bfloat16 h1 = __float2bfloat16_rn(x1);
        o[1] = h1;
        if (nsplit > 2) o[2] = __float2bfloat16_rn(x1 - __bfloat162float(h1));
    }
}

// Split form of R x C float32 planes (trans: of their transpose, R x C): the
// operands of the test hooks and of the leaf variants that only write float32.
__global__ void k_mirror(const float *re, const float *im, long long ld, int R, int C, int trans, Mirror m, int planes) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x, r = blockIdx.y;
    if (c >= C) return;
    const long long g = trans ? (long long)c * ld + r : (long long)r * ld + c;
    __nv_bfloat16 a[3], b[3];
    split_bf16(re[g], planes, a);
    split_bf16(im[g], planes, b);
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        if (p >= planes) break;
        __nv_bfloat16 *o = m.base + 2 * p * m.qpitch + r * m.pitch + c;
        o[0] = a[p];
        o[m.qpitch] = b[p];
    }
}

// A-layout pack of complex float64 rows: row r = [Re v(r,:), Im v(r,:)].
__global__ void k_pack64_A(const __grid_constant__ Tab<const double2 *> srct, long long ld, int R, int K,
                           int nsplit, const __grid_constant__ Tab<__nv_bfloat16 *> outt, long long kp, long long plane_pitch) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    int r = blockIdx.y;
    if (k >= K || r >= R) return;
    __nv_bfloat16 *out = outt.v[blockIdx.z];
    const double2 v = srct.v[blockIdx.z][(long long)r * ld + k];
    __nv_bfloat16 sa[3], sb[3];
    split_bf16((float)v.x, nsplit, sa);
    split_bf16((float)v.y, nsplit, sb);
    #pragma unroll
    for (int p = 0; p < 3; ++p) {
        if (p >= nsplit) break;
        __nv_bfloat16 *o = out + p * plane_pitch + (long long)r * kp;
        o[k] = sa[p];
        o[K + k] = sb[p];
    }
}

// B-layout pack of the transpose of complex float64 rows: logical
// v(r, k) = src[k][r] (r < R, k < K) -> rows r and R + r.
__global__ void k_pack64_BT(const __grid_constant__ Tab<const double2 *> srct, long long ld, int R, int K, int nsplit,
                            const __grid_constant__ Tab<__nv_bfloat16 *> outt, long long kp, long long plane_pitch) {
    __shared__ double2 t[32][33];
    const double2 *__restrict__ src = srct.v[blockIdx.z];
    __nv_bfloat16 *out = outt.v[blockIdx.z];
    int r0 = blockIdx.y * 32, k0 = blockIdx.x * 32;
    int tx = threadIdx.x, ty = threadIdx.y;
    for (int i = ty; i < 32; i += 8) {
        int k = k0 + i, r = r0 + tx;
        double2 v = cmk(0, 0);
        if (r < R && k < K) v = src[(long long)k * ld + r];
        t[tx][i] = v;
    }
    __syncthreads();
    for (int i = ty; i < 32; i += 8) {
        int r = r0 + i, k = k0 + tx;
        if (r >= R || k >= K) continue;
        double2 v = t[i][tx];
        __nv_bfloat16 sa[3], sb[3];
        split_bf16((float)v.x, nsplit, sa);
        split_bf16((float)v.y, nsplit, sb);
        #pragma unroll
        for (int p = 0; p < 3; ++p) {
            if (p >= nsplit) break;
            __nv_bfloat16 *o = out + p * plane_pitch;
            o[(long long)r * kp + k] = sa[p];
            o[(long long)r * kp + K + k] = __hneg(sb[p]);
            o[(long long)(R + r) * kp + k] = sb[p];
            o[(long long)(R + r) * kp + K + k] = sa[p];
        }
    }
}

// ---------------------------------------------------------------------------
// One step of the slab elimination between two inversions, for 4 x 4 groups of
// elements (rows {i, i+n/4, i+n/2, i+3n/4} x the same columns), two column
// groups per thread:
//   * the inverses just computed (transformed, "y space") become G = U Y U^T and
//     are written in split form (for the sweeps) and, at a checkpoint, in float32;
//   * the next block X = K_row - G (- G of the other chain) is assembled and
//     transformed, X' = U^T X U, and written as the recursion reads it: float32 on
//     and below the diagonal blocks, split form below them.
// U = P Q with Q the n-point butterfly (1/sqrt2)[R0 R1; R0 -R1] and P = diag of two
// n/2-point butterflies, R* random diagonals near 1; such a two-sided transform
// spreads every row over rows n/4 apart, so that the leading blocks of the Schur
// recursion (which pivots only inside its 32 x 32 leaves) are not the nearly
// singular sub-blocks of a strongly structured slab (high-contrast ridges) --
// the randomisation that lets symmetric indefinite elimination run without
// pivoting.  w[0 .. n): level-Q diagonals (R0 at i, R1 at n/2 + i); w[n .. 2n):
// level-P, half h (0 / 1) at n + h n/2 (R0 at i, R1 at n/4 + i).
// 24 n^2 bytes against the 72 n^2 of the five passes it replaces (inverse
// transform, packing, assembly, forward transform).  Two 4096 blocks: 179 us, 4.5
// TB/s (0.66 of the copy rate; about 100 instructions per element); 399 us with
// the source and the next block in separate registers and K evaluated for
// every element.
struct RowSrc {
    const float *re, *im;     // n x n block (null: no such source)
    int yspace, use;          // still transformed; subtracted from the next block
    Mirror gp;                // split G goes here (null base: not written)
    float *ck_re, *ck_im;     // float32 G goes here (null: not written)
};
struct RowJob {
    RowSrc s[2];
    const double *eps;        // slab permittivity
    int row, out;             // row of K (-1: none); whether the next block is written
    float sgn;                // X = K + sgn G
    float *Xre, *Xim;
    Mirror XP;                // (null base: float32 only)
};
template <int N>
struct RowJobs {
    RowJob j[N];
};

__device__ __forceinline__ void bf_fwd(float2 &t, float2 &b, float wa, float wb) {
    const float c = 0.70710678118654752f;
    const float2 s = make_float2(t.x + b.x, t.y + b.y), d = make_float2(t.x - b.x, t.y - b.y);
    t = make_float2(c * wa * s.x, c * wa * s.y);
    b = make_float2(c * wb * d.x, c * wb * d.y);
}
// The last product is not contracted into a following subtraction, so that G is
// the same number whether it is used at once or read back from a checkpoint.
__device__ __forceinline__ void bf_inv(float2 &t, float2 &b, float wa, float wb) {
    const float c = 0.70710678118654752f;
    const float2 u = make_float2(wa * t.x, wa * t.y), v = make_float2(wb * b.x, wb * b.y);
    t = make_float2(__fmul_rn(c, u.x + v.x), __fmul_rn(c, u.y + v.y));
    b = make_float2(__fmul_rn(c, u.x - v.x), __fmul_rn(c, u.y - v.y));
}

__device__ __forceinline__ void store_split2(const Mirror &m, int planes, long long r, long long c, float2 a, float2 b) {
    __nv_bfloat16 ar[3], ai[3], br[3], bi[3];
    split_bf16(a.x, planes, ar);
    split_bf16(a.y, planes, ai);
    split_bf16(b.x, planes, br);
    split_bf16(b.y, planes, bi);
    __nv_bfloat16 *o = m.base + r * m.pitch + c;
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        if (p >= planes) break;
        *reinterpret_cast<__nv_bfloat162 *>(o + 2 * p * m.qpitch) = __halves2bfloat162(ar[p], br[p]);
        *reinterpret_cast<__nv_bfloat162 *>(o + (2 * p + 1) * m.qpitch) = __halves2bfloat162(ai[p], bi[p]);
    }
}

// TWO: both sources (the middle row); otherwise only s[0] is looked at, and the
// block is assembled in the registers that held the source.
template <bool BF, bool TWO, int N>
__global__ void __launch_bounds__(128, TWO ? 2 : 4) k_row_step(GridDev g, const __grid_constant__ RowJobs<N> jobs, int n, const double2 *__restrict__ circ,
                                                               const float *__restrict__ w, int planes, int leaf) {
    const RowJob &J = jobs.j[blockIdx.z];
    const int q = n >> 2, half = n >> 3;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= q * half) return;
    const int i = idx / half, j = 2 * (idx - i * half);
    const float *wq = w, *wp0 = w + n, *wp1 = w + n + n / 2;
    float2 x[4][8];  // [row group][2 column group + column]
    // a source into v: load, transform, write out
    auto source = [&](const RowSrc &S, float2 (&v)[4][8]) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const long long o = (long long)(i + r * q) * n + j + c * q;
                const float2 a = *reinterpret_cast<const float2 *>(S.re + o), b = *reinterpret_cast<const float2 *>(S.im + o);
                v[r][2 * c] = make_float2(a.x, b.x);
                v[r][2 * c + 1] = make_float2(a.y, b.y);
            }
        if (BF && S.yspace) {  // G = U Y U^T: rows and columns, Q then P
            auto rows = [&](int a, int b, float wa, float wb) {
#pragma unroll
                for (int c = 0; c < 8; ++c) bf_inv(v[a][c], v[b][c], wa, wb);
            };
            auto cols = [&](int a, int b, const float *wa, const float *wb) {
                const float2 fa = *reinterpret_cast<const float2 *>(wa + j), fb = *reinterpret_cast<const float2 *>(wb + j);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    bf_inv(v[r][2 * a], v[r][2 * b], fa.x, fb.x);
                    bf_inv(v[r][2 * a + 1], v[r][2 * b + 1], fa.y, fb.y);
                }
            };
            rows(0, 2, wq[i], wq[2 * q + i]); rows(1, 3, wq[q + i], wq[3 * q + i]);
            rows(0, 1, wp0[i], wp0[q + i]); rows(2, 3, wp1[i], wp1[q + i]);
            cols(0, 2, wq, wq + 2 * q); cols(1, 3, wq + q, wq + 3 * q);
            cols(0, 1, wp0, wp0 + q); cols(2, 3, wp1, wp1 + q);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int row = i + r * q, col = j + c * q;
                const float2 a = v[r][2 * c], b = v[r][2 * c + 1];
                if (S.gp.base) store_split2(S.gp, planes, row, col, a, b);
                if (S.ck_re) {
                    const long long o = (long long)row * n + col;
                    *reinterpret_cast<float2 *>(S.ck_re + o) = make_float2(a.x, b.x);
                    *reinterpret_cast<float2 *>(S.ck_im + o) = make_float2(a.y, b.y);
                }
            }
    };
    if (J.s[0].re) source(J.s[0], x);
    if (!TWO && !J.out) return;
    // X = K + sgn G.  K: 4 - k^2 eps on the diagonal, -1 on the periodic neighbours,
    // the circulants Sigma_bot / Sigma_top on the first / last slab row; float64 only
    // on the diagonal
    const float s0 = J.s[0].re && J.s[0].use ? J.sgn : 0.f;
    const bool c0 = J.row == 0, c1 = J.row == g.h - 1;
    // off the end rows K touches a thread's elements only where i and j are (almost) equal modulo q
    const int off = i > j ? i - j : j - i;
    if (J.row >= 0 && (c0 || c1 || off <= 2 || off >= q - 2)) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                float kr = 0.f, ki = 0.f;
                const int row = i + r * q, col = j + (c & 1) + (c >> 1) * q, dx = row - col;
                if (dx == 0) kr = (float)(4.0 - g.k * g.k * J.eps[(long long)J.row * n + row]);
                if (dx == 1 || dx == -1 || dx == n - 1 || dx == 1 - n) kr -= 1.f;
                const int d = dx < 0 ? dx + n : dx;
                if (c0) { kr += (float)circ[d].x; ki += (float)circ[d].y; }
                if (c1) { kr += (float)circ[n + d].x; ki += (float)circ[n + d].y; }
                // (sgn = +-1: the product is exact)
                x[r][c] = s0 != 0.f ? make_float2(__fadd_rn(kr, s0 * x[r][c].x), __fadd_rn(ki, s0 * x[r][c].y)) : make_float2(kr, ki);
            }
    } else {
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 8; ++c) x[r][c] = s0 != 0.f ? make_float2(s0 * x[r][c].x, s0 * x[r][c].y) : make_float2(0.f, 0.f);
    }
    if constexpr (TWO) {
        if (J.s[1].re) {
            float2 v[4][8];
            source(J.s[1], v);
            if (J.s[1].use)
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        x[r][c] = make_float2(__fadd_rn(x[r][c].x, J.sgn * v[r][c].x), __fadd_rn(x[r][c].y, J.sgn * v[r][c].y));
        }
        if (!J.out) return;
    }
    if (BF) {  // X' = U^T X U: rows and columns, P^T then Q^T
        auto rows = [&](int a, int b, float wa, float wb) {
#pragma unroll
            for (int c = 0; c < 8; ++c) bf_fwd(x[a][c], x[b][c], wa, wb);
        };
        auto cols = [&](int a, int b, const float *wa, const float *wb) {
            const float2 fa = *reinterpret_cast<const float2 *>(wa + j), fb = *reinterpret_cast<const float2 *>(wb + j);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                bf_fwd(x[r][2 * a], x[r][2 * b], fa.x, fb.x);
                bf_fwd(x[r][2 * a + 1], x[r][2 * b + 1], fa.y, fb.y);
            }
        };
        rows(0, 1, wp0[i], wp0[q + i]); rows(2, 3, wp1[i], wp1[q + i]);
        rows(0, 2, wq[i], wq[2 * q + i]); rows(1, 3, wq[q + i], wq[3 * q + i]);
        cols(0, 1, wp0, wp0 + q); cols(2, 3, wp1, wp1 + q);
        cols(0, 2, wq, wq + 2 * q); cols(1, 3, wq + q, wq + 3 * q);
    }
    const int ls = 31 - __clz(leaf);  // leaf sizes are powers of two
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int row = i + r * q, col = j + c * q;
            const int br = row >> ls, bc = col >> ls;
            if (bc > br) continue;
            const float2 a = x[r][2 * c], b = x[r][2 * c + 1];
            const long long o = (long long)row * n + col;
            *reinterpret_cast<float2 *>(J.Xre + o) = make_float2(a.x, b.x);
            *reinterpret_cast<float2 *>(J.Xim + o) = make_float2(a.y, b.y);
            if (J.XP.base && bc < br) store_split2(J.XP, planes, row, col, a, b);
        }
}

// Float32 Gauss-Jordan inverse of an n x n (n <= 128) diagonal block with
// partial pivoting, in shared memory (planar in global memory).
__global__ void __launch_bounds__(512) k_leaf_inv32(const __grid_constant__ Tab<float *> ret, const __grid_constant__ Tab<float *> imt, long long ld, int n, const __grid_constant__ Tab<int *> flt) {
    float *re = ret.v[blockIdx.x], *im = imt.v[blockIdx.x];
    int *flags = flt.v[blockIdx.x];
    extern __shared__ float2 a32[];
    __shared__ float2 colk[128];
    __shared__ int piv[128];
    __shared__ int s_p;
    __shared__ float2 s_inv;
    int tid = threadIdx.x, nt = blockDim.x;
    for (int e = tid; e < n * n; e += nt) {
        long long gidx = (long long)(e / n) * ld + (e % n);
        a32[e] = make_float2(re[gidx], im[gidx]);
    }
    __syncthreads();
    for (int k = 0; k < n; ++k) {
        if (tid < 32) {
            float best = -1.f;
            int bi = k;
            for (int i = k + tid; i < n; i += 32) {
                float2 v = a32[i * n + k];
                float m = v.x * v.x + v.y * v.y;
                if (m > best) { best = m; bi = i; }
            }
            for (int off = 16; off > 0; off >>= 1) {
                float ob = __shfl_down_sync(0xffffffffu, best, off);
                int oi = __shfl_down_sync(0xffffffffu, bi, off);
                if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
            }
            if (tid == 0) {
                s_p = bi;
                piv[k] = bi;
                if (!(best > 0.f) || !isfinite(best)) atomicOr(flags, FLAG_SINGULAR);
            }
        }
        __syncthreads();
        int p = s_p;
        if (p != k) {
            for (int j = tid; j < n; j += nt) {
                float2 t = a32[k * n + j];
                a32[k * n + j] = a32[p * n + j];
                a32[p * n + j] = t;
            }
            __syncthreads();
        }
        if (tid == 0) {
            float2 d = a32[k * n + k];
            float den = d.x * d.x + d.y * d.y;
            s_inv = make_float2(d.x / den, -d.y / den);
        }
        __syncthreads();
        float2 inv = s_inv;
        for (int j = tid; j < n; j += nt) a32[k * n + j] = (j == k) ? inv : fmul(a32[k * n + j], inv);
        for (int i = tid; i < n; i += nt) colk[i] = a32[i * n + k];
        __syncthreads();
        for (int e = tid; e < n * n; e += nt) {
            int i = e / n, j = e - i * n;
            if (i == k) continue;
            float2 f = colk[i];
            if (j == k) {
                float2 t = fmul(f, inv);
                a32[e] = make_float2(-t.x, -t.y);
            } else {
                float2 t = fmul(f, a32[k * n + j]);
                a32[e] = make_float2(a32[e].x - t.x, a32[e].y - t.y);
            }
        }
        __syncthreads();
    }
    for (int k = n - 1; k >= 0; --k) {
        int p = piv[k];
        if (p != k) {
            for (int i = tid; i < n; i += nt) {
                float2 t = a32[i * n + k];
                a32[i * n + k] = a32[i * n + p];
                a32[i * n + p] = t;
            }
        }
        __syncthreads();
    }
    for (int e = tid; e < n * n; e += nt) {
        long long gidx = (long long)(e / n) * ld + (e % n);
        re[gidx] = a32[e].x;
        im[gidx] = a32[e].y;
    }
}

template <int NB>
__global__ void __launch_bounds__(NB * 4) k_leaf32(const __grid_constant__ Tab<float *> re, const __grid_constant__ Tab<float *> im, long long ld, const __grid_constant__ Tab<int *> flags) {
    const int b = blockIdx.x;
    LeafIO<float, true> io{re.v[b], im.v[b], nullptr, ld};
    leaf_gj<float, NB, true>(io, flags.v[b]);
}

template <int NB>
__global__ void __launch_bounds__(NB * 4) k_leaf32r(const __grid_constant__ Tab<float *> re, const __grid_constant__ Tab<float *> im, long long ld, const __grid_constant__ Tab<int *> flags) {
    const int b = blockIdx.x;
    leaf_gj_regs<NB>(re.v[b], im.v[b], ld, flags.v[b]);
}

// 128 x 128 and 64 x 64 diagonal blocks (NP = 4, 2; one cluster of NP CTAs each): the inverse in place
// and in split form (XP.base null: float32 only).
template <int NP>
__global__ void __launch_bounds__(lc::NT) __cluster_dims__(NP, 1, 1) k_leaf_cluster(const __grid_constant__ Tab<float *> ret, const __grid_constant__ Tab<float *> imt, long long ld, const __grid_constant__ Tab<Mirror> XP, int planes, const __grid_constant__ Tab<int *> flags) {
    extern __shared__ __align__(16) unsigned char lc_smem[];
    constexpr int N = 32 * NP;
    lc::Smem<NP> &sm = *reinterpret_cast<lc::Smem<NP> *>(lc_smem);
    const int b = blockIdx.x / NP, rank = blockIdx.x % NP;
    float *re = ret.v[b], *im = imt.v[b];
    const Mirror m = XP.v[b];
    const bool sound = lc::invert<NP>(sm, re, im, ld, rank, [&](int r, int c, float2 u, float2 v) {
        if (m.base) store_split2(m, planes, r, c, u, v);
    });
    if (sound) return;
    if (rank != 0 || threadIdx.x >= 4 * N) return;
    if (threadIdx.x == 0) atomicAdd(flags.v[b] + 1, 1);  // fallback count (flags[1])
    leaf_gj_regs<N>(re, im, ld, flags.v[b]);
    if (!m.base) return;
    __syncthreads();  // the block's float32 stores are read back by other threads
    for (int e = threadIdx.x; e < N * N / 2; e += 4 * N) {
        const int r = e / (N / 2), c = 2 * (e % (N / 2));
        const float2 a = *reinterpret_cast<const float2 *>(re + (long long)r * ld + c);
        const float2 d = *reinterpret_cast<const float2 *>(im + (long long)r * ld + c);
        store_split2(m, planes, r, c, make_float2(a.x, d.x), make_float2(a.y, d.y));
    }
}

template <int NB>
__global__ void __launch_bounds__(NB * 4) k_leaf32r2(const __grid_constant__ Tab<float *> re, const __grid_constant__ Tab<float *> im, long long ld, const __grid_constant__ Tab<int *> flags) {
    const int b = blockIdx.x;
    leaf_gj_regs2<NB>(re.v[b], im.v[b], ld, flags.v[b]);
}

// Element-wise step of a field sweep between two products: o = the product's
// rows (float32 planes O for columns [o0, o1), plus O2 for [p0, p1)), v = o + add
// (float64 rows, columns [a0, a1)); out = v, out = o or out += o; and v in split
// form as the next product's operand (row c - c0 for column c).  Two x per thread.
struct FieldJob {
    const float *O, *O2;      // re plane, im plane at + olen (null: none)
    long long olen;
    int o0, o1, p0, p1;
    const double2 *add;
    int a0, a1;
    double2 *out;
    int mode;                 // 1: out = v, 2: out = o, 3: out += o
    Mirror m;
    int c0, c1;               // columns of this job
};
template <int N>
struct FieldJobs {
    FieldJob j[N];
};

template <int N>
__global__ void __launch_bounds__(128) k_field_step(const __grid_constant__ FieldJobs<N> jobs, int nx, int planes) {
    const FieldJob &J = jobs.j[blockIdx.z];
    const int x = 2 * (blockIdx.x * blockDim.x + threadIdx.x), c = J.c0 + blockIdx.y;
    if (x >= nx || c >= J.c1) return;
    double2 o[2] = {cmk(0.0, 0.0), cmk(0.0, 0.0)};
    if (J.O && c >= J.o0 && c < J.o1) {
        const float *p = J.O + (long long)(c - J.o0) * nx + x;
        const float2 a = *reinterpret_cast<const float2 *>(p), b = *reinterpret_cast<const float2 *>(p + J.olen);
        o[0] = cmk(a.x, b.x);
        o[1] = cmk(a.y, b.y);
    }
    if (J.O2 && c >= J.p0 && c < J.p1) {
        const float *p = J.O2 + (long long)(c - J.p0) * nx + x;
        const float2 a = *reinterpret_cast<const float2 *>(p), b = *reinterpret_cast<const float2 *>(p + J.olen);
        o[0] = cadd(o[0], cmk(a.x, b.x));
        o[1] = cadd(o[1], cmk(a.y, b.y));
    }
    const long long g = (long long)c * nx + x;
    double2 v[2] = {o[0], o[1]};
    if (J.add && c >= J.a0 && c < J.a1) {
        v[0] = cadd(J.add[g], v[0]);
        v[1] = cadd(J.add[g + 1], v[1]);
    }
    if (J.mode == 1) {
        J.out[g] = v[0];
        J.out[g + 1] = v[1];
    } else if (J.mode == 2) {
        J.out[g] = o[0];
        J.out[g + 1] = o[1];
    } else if (J.mode == 3) {
        J.out[g] = cadd(J.out[g], o[0]);
        J.out[g + 1] = cadd(J.out[g + 1], o[1]);
    }
    if (J.m.base)
        store_split2(J.m, planes, c - J.c0, x, make_float2((float)v[0].x, (float)v[0].y),
                     make_float2((float)v[1].x, (float)v[1].y));
}

// out = Sigma in, Sigma = U diag(sigma) U^H (a circulant), per column, in shared
// memory: a radix-4 decimation-in-frequency transform (natural order in, digits
// reversed out), the product with sigma where the values lie, and the transposed
// transform back to natural order, so that nothing is permuted.  An odd power of
// two takes one radix-2 stage first (and last).  blockIdx.y: 0 the first slab row
// (Sigma_bot, out cb), 1 the last (Sigma_top, ct); blockIdx.z: design.
// Bound by the float64 pipe: 28 operations per four points and two stages (16
// where all factors are 1) against 32 of radix 2; 4096 x 260: 1.04 ms against
// 1.24 ms.
__global__ void __launch_bounds__(256) k_circ_apply(const __grid_constant__ Tab<const double2 *> Et, long long last, const __grid_constant__ Tab<double2 *> cbt, const __grid_constant__ Tab<double2 *> ctt,
                             int n, int logn, const double2 *__restrict__ sigma, const double2 *__restrict__ tw) {
    extern __shared__ double2 a[];
    const double2 *src = Et.v[blockIdx.z] + (blockIdx.y ? last : 0) + (long long)blockIdx.x * n;
    double2 *out = (blockIdx.y ? ctt.v[blockIdx.z] : cbt.v[blockIdx.z]) + (long long)blockIdx.x * n;
    sigma += blockIdx.y * n;
    const int t0 = threadIdx.x, nt = blockDim.x;
    // w = exp(-2 pi i k / n), k < n: the table holds the first half
    auto root = [&](int k) {
        const double2 w = tw[k & (n / 2 - 1)];
        return k < n / 2 ? w : make_double2(-w.x, -w.y);
    };
    for (int i = t0; i < n; i += nt) a[i] = src[i];
    __syncthreads();
    int len = n;
    if (logn & 1) {
        for (int k = t0; k < n / 2; k += nt) {
            const double2 u = a[k], v = a[k + n / 2];
            a[k] = cadd(u, v);
            a[k + n / 2] = cmul(csub(u, v), tw[k]);
        }
        len = n / 2;
        __syncthreads();
    }
    for (; len >= 4; len >>= 2) {
        const int q = len >> 2, lq = __ffs(q) - 1, st = n / len;
        for (int t = t0; t < n / 4; t += nt) {
            const int k = t & (q - 1), i = ((t >> lq) << (lq + 2)) + k;
            const double2 x0 = a[i], x1 = a[i + q], x2 = a[i + 2 * q], x3 = a[i + 3 * q];
            const double2 s0 = cadd(x0, x2), s1 = csub(x0, x2), s2 = cadd(x1, x3), s3 = csub(x1, x3);
            const double2 y1 = make_double2(s1.x + s3.y, s1.y - s3.x), y2 = csub(s0, s2), y3 = make_double2(s1.x - s3.y, s1.y + s3.x);
            a[i] = cadd(s0, s2);
            if (q > 1) {
                a[i + q] = cmul(y1, tw[k * st]);
                a[i + 2 * q] = cmul(y2, tw[2 * k * st]);
                a[i + 3 * q] = cmul(y3, root(3 * k * st));
            } else {
                a[i + 1] = y1;
                a[i + 2] = y2;
                a[i + 3] = y3;
            }
        }
        __syncthreads();
    }
    // position p holds the coefficient whose base-4 digits (below the radix-2 bit) are p's reversed
    const int bits = logn & ~1;
    const double inv_n = 1.0 / n;
    for (int p = t0; p < n; p += nt) {
        unsigned r = __brev((unsigned)(p & ((1 << bits) - 1))) >> (32 - bits);
        r = ((r & 0x55555555u) << 1) | ((r >> 1) & 0x55555555u);
        const int m = (logn & 1) ? (int)(2 * r + (p >> bits)) : (int)r;
        const double2 s = sigma[m];
        a[p] = cmul(a[p], make_double2(s.x * inv_n, s.y * inv_n));
    }
    __syncthreads();
    auto cmul_conj = [](double2 x, double2 w) { return cmul(x, make_double2(w.x, -w.y)); };
    for (len = 4; len <= (1 << bits); len <<= 2) {
        const int q = len >> 2, lq = __ffs(q) - 1, st = n / len;
        for (int t = t0; t < n / 4; t += nt) {
            const int k = t & (q - 1), i = ((t >> lq) << (lq + 2)) + k;
            double2 x1 = a[i + q], x2 = a[i + 2 * q], x3 = a[i + 3 * q];
            const double2 x0 = a[i];
            if (q > 1) {
                x1 = cmul_conj(x1, tw[k * st]);
                x2 = cmul_conj(x2, tw[2 * k * st]);
                x3 = cmul_conj(x3, root(3 * k * st));
            }
            const double2 s0 = cadd(x0, x2), s1 = csub(x0, x2), s2 = cadd(x1, x3), s3 = csub(x1, x3);
            a[i] = cadd(s0, s2);
            a[i + q] = make_double2(s1.x - s3.y, s1.y + s3.x);
            a[i + 2 * q] = csub(s0, s2);
            a[i + 3 * q] = make_double2(s1.x + s3.y, s1.y - s3.x);
        }
        __syncthreads();
    }
    if (logn & 1) {
        for (int k = t0; k < n / 2; k += nt) {
            const double2 u = a[k], v = cmul_conj(a[k + n / 2], tw[k]);
            out[k] = cadd(u, v);
            out[k + n / 2] = csub(u, v);
        }
    } else {
        for (int i = t0; i < n; i += nt) out[i] = a[i];
    }
}

// r_j = R_j - K E restricted to the slab, float64.  K E at a pixel is
// d E - (sum of the four neighbours) + boundary terms, d = 4 - k^2 eps; the
// neighbour sum and the boundary terms are gathered first so that the
// diagonal term is one fused multiply-add per component.  One thread walks the
// slab rows of RC columns at one x, so each field value is loaded three times (as
// centre, left, right) instead of five, with the next row's loads in flight, and
// the squared norms of the columns are summed on the way (part: one value per
// block and column, see k_normsum).  R is zero except on the first and last slab
// rows (Rt: those two rows; null: r = K E).  Bound by the float64 pipe: 10.5
// operations per point at 2 per clock and SM (4096 x 260, 686 columns: 0.82 ms of
// them, 1.15 ms measured; 1.62 ms with the end rows' conditions in the loop).
constexpr int RC = 2;
__global__ void __launch_bounds__(128) k_residual(GridDev g, const __grid_constant__ Tab<const double *> epst, const __grid_constant__ Tab<const double2 *> Et, const __grid_constant__ Tab<const double2 *> Rt, const __grid_constant__ Tab<double2 *> cbt,
                                                  const __grid_constant__ Tab<double2 *> ctt, const __grid_constant__ Tab<double2 *> rt, const __grid_constant__ Tab<double *> partt, int ncol) {
    const int b = blockIdx.z, n = g.nx, h = g.h, c0 = RC * blockIdx.y;
    const int x = blockIdx.x * 128 + threadIdx.x;
    const long long L = (long long)ncol * n;
    double acc[RC] = {};
    if (x < n) {
        const double *eps = epst.v[b] + x;
        const double2 *R = Rt.v[b];
        const double k2 = -(g.k * g.k);
        const int xr = (x + 1 == n) ? 0 : x + 1, xl = (x == 0) ? n - 1 : x - 1;
        long long col[RC];
        const double2 *e[RC];
#pragma unroll
        for (int u = 0; u < RC; ++u) {
            col[u] = (long long)min(c0 + u, ncol - 1) * n;  // (an odd last column is computed twice, written once)
            e[u] = Et.v[b] + col[u];
        }
        double2 below[RC], here[RC], above[RC], lr[RC], rr[RC];
        double ep = eps[0];
#pragma unroll
        for (int u = 0; u < RC; ++u) {
            below[u] = cmk(0.0, 0.0);
            here[u] = e[u][x];
            lr[u] = e[u][xl];
            rr[u] = e[u][xr];
            above[u] = h > 1 ? e[u][L + x] : cmk(0.0, 0.0);
        }
        // extra: what an end row adds to the neighbour sum.  The rows between them
        // run without a condition (one would be turned into float64 operations
        // that are always executed: 21 per point instead of 10.5).
        auto row = [&](int j, const double2 (&extra)[RC], bool end) {
            // the next row's neighbours and the row above it
            double2 nl[RC], nr[RC], na[RC];
            double en = 0.0;
#pragma unroll
            for (int u = 0; u < RC; ++u) {
                e[u] += L;
                nl[u] = nr[u] = na[u] = cmk(0.0, 0.0);
                if (j + 1 < h) {
                    nl[u] = e[u][xl];
                    nr[u] = e[u][xr];
                    if (j + 2 < h) na[u] = e[u][L + x];
                }
            }
            if (j + 1 < h) en = eps[(long long)(j + 1) * n];
            const double d = fma(k2, ep, 4.0);
#pragma unroll
            for (int u = 0; u < RC; ++u) {
                double2 nbr = cadd(cadd(rr[u], lr[u]), cadd(below[u], above[u]));  // neighbours, zero outside the slab
                if (end) nbr = cadd(nbr, extra[u]);
                const double2 v = make_double2(fma(-d, here[u].x, nbr.x), fma(-d, here[u].y, nbr.y));
                if (c0 + u < ncol) rt.v[b][j * L + col[u] + x] = R ? v : make_double2(-v.x, -v.y);  // without R: K E
                acc[u] = fma(v.x, v.x, fma(v.y, v.y, acc[u]));
                below[u] = here[u];
                here[u] = above[u];
                above[u] = na[u];
                lr[u] = nl[u];
                rr[u] = nr[u];
            }
            ep = en;
        };
        double2 first[RC], last[RC];
#pragma unroll
        for (int u = 0; u < RC; ++u) {
            const double2 sb = cbt.v[b][col[u] + x], st = ctt.v[b][col[u] + x];
            first[u] = R ? csub(R[col[u] + x], sb) : make_double2(-sb.x, -sb.y);
            last[u] = R && h > 1 ? csub(R[L + col[u] + x], st) : make_double2(-st.x, -st.y);
            if (h == 1) first[u] = cadd(first[u], last[u]);
        }
        row(0, first, true);
#pragma unroll 1
        for (int j = 1; j < h - 1; ++j) row(j, first, false);
        if (h > 1) row(h - 1, last, true);
    }
    double *part = partt.v[b];
    if (!part) return;
    __shared__ double red[RC][4];
#pragma unroll
    for (int u = 0; u < RC; ++u) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], off);
        if ((threadIdx.x & 31) == 0) red[u][threadIdx.x >> 5] = acc[u];
    }
    __syncthreads();
    const int u = threadIdx.x;
    if (u < RC && c0 + u < ncol)
        part[(long long)(c0 + u) * gridDim.x + blockIdx.x] = (red[u][0] + red[u][1]) + (red[u][2] + red[u][3]);
}

// out[c] = the sum of column c's np partial sums, in a fixed order (one warp per column).
__global__ void __launch_bounds__(32) k_normsum(const __grid_constant__ Tab<double *> partt, int np, const __grid_constant__ Tab<double *> outt) {
    const double *p = partt.v[blockIdx.z] + (long long)blockIdx.x * np;
    double a = 0.0;
    for (int i = threadIdx.x; i < np; i += 32) a += p[i];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
    if (threadIdx.x == 0) outt.v[blockIdx.z][blockIdx.x] = a;
}

// out[c] = sum_{j,x} |X_j[c][x]|^2 (one block of 256 threads per column, a
// fixed summation order; two independent loads in flight per thread).
__global__ void __launch_bounds__(256) k_colnorm(const double2 *X, int h, int ncol, int nx, double *out) {
    __shared__ double red[256];
    const int c = blockIdx.x;
    double a0 = 0.0, a1 = 0.0;
    for (int j = 0; j < h; ++j) {
        const long long o = ((long long)j * ncol + c) * nx;
        const double2 *p = X + o;
        int x = threadIdx.x;
        for (; x + 256 < nx; x += 512) {
            const double2 u = p[x], v = p[x + 256];
            a0 += cabs2(u);
            a1 += cabs2(v);
        }
        if (x < nx) {
            const double2 u = p[x];
            a0 += cabs2(u);
        }
    }
    red[threadIdx.x] = a0 + a1;
    __syncthreads();
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if ((int)threadIdx.x < off) red[threadIdx.x] += red[threadIdx.x + off];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[c] = red[0];
}

// Krylov helpers over fields [row][column][x]: per-column dot products
// (conj(A) . B, one block per column, fixed order), Y += sgn coef[c] X, and
// Y = X / sqrt(nrm2[c]) (zero when the norm is zero).
__global__ void k_coldot(const double2 *A, const double2 *B, int h, int ncol, int nx, double2 *out) {
    __shared__ double2 red[256];
    const int c = blockIdx.x;
    double2 acc = cmk(0.0, 0.0);
    for (int j = 0; j < h; ++j) {
        const long long o = ((long long)j * ncol + c) * nx;
        for (int x = threadIdx.x; x < nx; x += blockDim.x) acc = cadd(acc, cmul(cconj(A[o + x]), B[o + x]));
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if ((int)threadIdx.x < off) red[threadIdx.x] = cadd(red[threadIdx.x], red[threadIdx.x + off]);
        __syncthreads();
    }
    if (threadIdx.x == 0) out[c] = red[0];
}

__global__ void k_colaxpy(double2 *Y, const double2 *X, const double2 *coef, double sgn, int ncol, int nx) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x, c = blockIdx.y, j = blockIdx.z;
    if (x >= nx) return;
    const long long i = ((long long)j * ncol + c) * nx + x;
    Y[i] = cadd(Y[i], cscale(cmul(coef[c], X[i]), sgn));
}

__global__ void k_colscale(double2 *Y, const double2 *X, const double *nrm2, int ncol, int nx) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x, c = blockIdx.y, j = blockIdx.z;
    if (x >= nx) return;
    const long long i = ((long long)j * ncol + c) * nx + x;
    const double n2 = nrm2[c];
    Y[i] = n2 > 0.0 ? cscale(X[i], 1.0 / sqrt(n2)) : cmk(0.0, 0.0);
}

// g_j(x) = 2 k^2 Re sum_b Phi_j[b][x] Q[b][x].  Block: 32 consecutive x (lanes)
// x 8 warps, warp w summing b = w, w + 8, ...; the 8 partial sums are added in
// a fixed order (deterministic).
__global__ void __launch_bounds__(256) k_grad_rowdot32(const __grid_constant__ Tab<const double2 *> Et, const __grid_constant__ Tab<const float *> Qret,
                                                       const __grid_constant__ Tab<const float *> Qimt, int j, int nx, int n_in, int n_out,
                                                       double k2, const __grid_constant__ Tab<double *> gt) {
    __shared__ double part[8][32];
    const double2 *E = Et.v[blockIdx.z];
    const float *Qre = Qret.v[blockIdx.z], *Qim = Qimt.v[blockIdx.z];
    double *g = gt.v[blockIdx.z];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int x = blockIdx.x * 32 + lane;
    const int ncol = n_in + n_out;
    double acc = 0.0;
    if (x < nx) {
        const double2 *phi = E + ((long long)j * ncol + n_in) * nx + x;
        for (int b = w; b < n_out; b += 8) {
            const double2 p = phi[(long long)b * nx];
            acc = fma(p.x, (double)Qre[(long long)b * nx + x], acc);
            acc = fma(-p.y, (double)Qim[(long long)b * nx + x], acc);
        }
    }
    part[w][lane] = acc;
    __syncthreads();
    if (w == 0 && x < nx) {
        double t = part[0][lane];
#pragma unroll
        for (int i = 1; i < 8; ++i) t += part[i][lane];
        g[(long long)j * nx + x] = 2.0 * k2 * t;
    }
}

long long round_up(long long a, long long b) { return (a + b - 1) / b * b; }

template <typename T>
int walloc(apf_ctx *c, MixedWork *w, T **p, long long count) {
    void *q = nullptr;
    size_t bytes = (size_t)std::max<long long>(count, 1) * sizeof(T);
    cudaError_t e = cudaMalloc(&q, bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return set_err(c, APF_ENOMEM, "cudaMalloc(%zu) for the mixed workspace failed", bytes);
    }
    w->allocs.push_back(q);
    c->ws_bytes += (long long)bytes;
    *p = (T *)q;
    return APF_OK;
}

// ---- host-side helpers ----------------------------------------------------
struct PV {  // planar complex view
    float *re, *im;
    long long ld;
    PV off(long long r, long long c) const { return PV{re + r * ld + c, im + r * ld + c, ld}; }
};

// The problems of one launch: designs, and for the elimination and the sweeps
// also the two chains of each (sd[b]); they share grid, slab height, channel set
// and settings, each has its own buffers.
struct Bat {
    int n = 0;
    apf_ctx *c[CG_MAX_PROB] = {};
    int sd[CG_MAX_PROB] = {};
    apf_ctx *lead() const { return c[0]; }
    SideWork &w(int b) const { return c[b]->mw->sd[sd[b]]; }
    void add(apf_ctx *ctx, int side) {
        c[n] = ctx;
        sd[n++] = side;
    }
};

Bat one(apf_ctx *c) {
    Bat b;
    b.add(c, 0);
    return b;
}

template <typename T, typename F>
Tab<T> tab(const Bat &bt, F f) {
    Tab<T> t{};
    for (int b = 0; b < bt.n; ++b) t.v[b] = f(b);
    return t;
}

void pack64A_b(const Bat &bt, PackView *v, __nv_bfloat16 *const *dst, const double2 *const *src, long long ld, int R,
               int K, int nsplit, cudaStream_t s) {
    const long long kp = round_up(2LL * K, 64);
    for (int b = 0; b < bt.n; ++b) {
        if (kp != 2LL * K) cudaMemsetAsync(dst[b], 0, sizeof(__nv_bfloat16) * R * kp * nsplit, s);
        v[b] = PackView{dst[b], R, kp, nsplit, (long long)R * kp};
    }
    dim3 grid((K + 255) / 256, R, bt.n);
    APF_LAUNCH(bt.lead(), k_pack64_A, grid, 256, 0, s, tab<const double2 *>(bt, [&](int b) { return src[b]; }), ld, R, K, nsplit,
               tab<__nv_bfloat16 *>(bt, [&](int b) { return dst[b]; }), kp, (long long)R * kp);
}

void pack64BT_b(const Bat &bt, PackView *v, __nv_bfloat16 *const *dst, const double2 *const *src, long long ld, int R,
                int K, int nsplit, cudaStream_t s) {
    const long long kp = round_up(2LL * K, 64);
    const long long rows = 2LL * R;
    for (int b = 0; b < bt.n; ++b) {
        if (kp != 2LL * K) cudaMemsetAsync(dst[b], 0, sizeof(__nv_bfloat16) * rows * kp * nsplit, s);
        v[b] = PackView{dst[b], rows, kp, nsplit, rows * kp};
    }
    dim3 grid((K + 31) / 32, (R + 31) / 32, bt.n);
    APF_LAUNCH(bt.lead(), k_pack64_BT, grid, dim3(32, 8), 0, s,
               tab<const double2 *>(bt, [&](int b) { return src[b]; }), ld, R, K, nsplit,
               tab<__nv_bfloat16 *>(bt, [&](int b) { return dst[b]; }), kp, rows * kp);
}

int leaf_size(const MixedWork *w) { return w->leaf; }

void mirror_b(const Bat &bt, const PV *X, const Mirror *m, int R, int C, bool trans, int planes, cudaStream_t s) {
    for (int b = 0; b < bt.n; ++b)
        APF_LAUNCH(bt.lead(), k_mirror, dim3((C + 127) / 128, R), 128, 0, s, (const float *)X[b].re,
                   (const float *)X[b].im, X[b].ld, R, C, trans ? 1 : 0, m[b], planes);
}

// Diagonal blocks of the recursion, one CTA or cluster per problem (kernel variant per the
// context's knobs); m: where the split form of the inverse goes (null base: nowhere).
void leaf_b(const Bat &bt, const PV *X, int n, const Mirror *m, cudaStream_t s) {
    apf_ctx *c = bt.lead();
    const MixedWork *w = c->mw;
    const int nb = bt.n, v = w->leaf_variant;
    const long long ld = X[0].ld;
    const auto re = tab<float *>(bt, [&](int b) { return X[b].re; }), im = tab<float *>(bt, [&](int b) { return X[b].im; });
    const auto fl = tab<int *>(bt, [&](int b) { return bt.c[b]->d_flags; });
    // 128 and 64: block elimination by a cluster (default); variants 1-3 are the single-level Gauss-Jordan kernels.
    if (n == 128 && v == 0) {
        APF_LAUNCH(c, k_leaf_cluster<4>, 4 * nb, lc::NT, (int)sizeof(lc::Smem<4>), s, re, im, ld, tab<Mirror>(bt, [&](int b) { return m[b]; }),
                  w->nsplit_elim, fl);
        return;
    }
    if (n == 64 && v == 0) {
        APF_LAUNCH(c, k_leaf_cluster<2>, 2 * nb, lc::NT, (int)sizeof(lc::Smem<2>), s, re, im, ld, tab<Mirror>(bt, [&](int b) { return m[b]; }),
                  w->nsplit_elim, fl);
        return;
    }
    if (n == 128 && v == 1) APF_LAUNCH(c, k_leaf32r2<128>, nb, 512, 0, s, re, im, ld, fl);
    else if (n == 128 && v == 2) APF_LAUNCH(c, k_leaf32<128>, nb, 512, leaf_smem_bytes<128>(8), s, re, im, ld, fl);
    else if (n == 128) APF_LAUNCH(c, k_leaf32r<128>, nb, 512, 0, s, re, im, ld, fl);
    else if (n == 64 && v == 1) APF_LAUNCH(c, k_leaf32r2<64>, nb, 256, 0, s, re, im, ld, fl);
    else if (n == 64) APF_LAUNCH(c, k_leaf32r<64>, nb, 256, 0, s, re, im, ld, fl);
    else if (n == 32) APF_LAUNCH(c, k_leaf32<32>, nb, 128, leaf_smem_bytes<32>(8), s, re, im, ld, fl);
    else if (n == 16) APF_LAUNCH(c, k_leaf32<16>, nb, 64, leaf_smem_bytes<16>(8), s, re, im, ld, fl);
    else APF_LAUNCH(c, k_leaf_inv32, nb, 256, n * n * (int)sizeof(float2), s, re, im, ld, n, fl);
    if (m[0].base) mirror_b(bt, X, m, n, n, false, w->nsplit_elim, s);
}

// X[b] <- X[b]^-1 in place for complex-symmetric X[b] (n a power of two), by the
// 2x2 block Schur recursion of the float64 path,
//   [A B; C D]^-1 = [Ai + T^T V, -V^T; -V, Si],  T = C Ai, S = D - T C^T, V = Si T,
// with all four products on the tensor cores, two of them symmetric.  X holds the
// block in float32 (on and below its diagonal blocks) and XP the split form of
// what lies below them; they come out as the whole inverse, XP with want_mirror
// only.  Every product reads split operands where the previous steps' epilogues
// left them (T only exists split, as T and T^T; V is written as -V to C and,
// transposed, to B, and read back from B as the operand of T^T V), so nothing
// runs between the products.
// toff: offset of this level's T in the T buffers.  upper: the result is wanted in
// float32 above the diagonal (outside its leaves) too, which nothing inside the recursion
// reads: an SM stores 32 bytes per clock, and half of a product's time can be stores.
int inv32_b(const Bat &bt, const PV *X, const Mirror *XP, int n, bool want_mirror, long long toff, cudaStream_t s, bool upper = true) {
    apf_ctx *c = bt.lead();
    MixedWork *w = c->mw;
    const int nb = bt.n, planes = w->nsplit_elim;
    if (n <= leaf_size(w)) {
        Mirror none[CG_MAX_PROB];
        leaf_b(bt, X, n, want_mirror ? XP : none, s);
        return APF_OK;
    }
    const int h = n / 2;
    const long long hh = (long long)h * h, sub = toff + 2 * planes * hh;
    PV A[CG_MAX_PROB], B[CG_MAX_PROB], C[CG_MAX_PROB], D[CG_MAX_PROB];
    Mirror mA[CG_MAX_PROB], mB[CG_MAX_PROB], mC[CG_MAX_PROB], mD[CG_MAX_PROB], mT[CG_MAX_PROB], mTT[CG_MAX_PROB];
    for (int b = 0; b < nb; ++b) {
        A[b] = X[b]; B[b] = X[b].off(0, h); C[b] = X[b].off(h, 0); D[b] = X[b].off(h, h);
        mA[b] = XP[b]; mB[b] = XP[b].off(0, h); mC[b] = XP[b].off(h, 0); mD[b] = XP[b].off(h, h);
        mT[b] = Mirror{bt.w(b).TP + toff, h, hh};
        mTT[b] = Mirror{bt.w(b).TT + toff, h, hh};
    }
    auto out = [](const PV &v, const Mirror &m) { return CgOut{v.re, v.im, v.ld, m}; };
    CgProblem pb[CG_MAX_PROB];
    const Mirror none[CG_MAX_PROB];
    auto product = [&](const Mirror *P, const Mirror *Q, float alpha, const PV *in, const PV *o, const Mirror *om,
                       const PV *ot, const Mirror *otm, bool sym, int t_block = 0) {
        for (int b = 0; b < nb; ++b) {
            pb[b] = CgProblem{};
            pb[b].A = P[b];
            pb[b].B = Q[b];
            pb[b].M = h;
            pb[b].out = out(o ? o[b] : PV{}, om[b]);
            pb[b].outT = out(ot ? ot[b] : PV{}, otm[b]);
            if (in) {
                pb[b].in_re = in[b].re;
                pb[b].in_im = in[b].im;
                pb[b].ldi = in[b].ld;
            }
            pb[b].flags = bt.c[b]->d_flags;
            pb[b].t_block = t_block;
        }
        return cgemm_n(c, nb, pb, planes, h, h, h, alpha, in ? 1.f : 0.f, sym, false, s);
    };
    int rc;
    if ((rc = inv32_b(bt, A, mA, h, true, sub, s, false))) return rc;
    // T = C Ai (Ai symmetric: its rows are its columns)
    if ((rc = product(mC, mA, 1.f, nullptr, nullptr, mT, nullptr, mTT, false))) return rc;
    // D = D - T C^T, as the inversion of D reads it
    const bool deep = h > leaf_size(w);
    if ((rc = product(mT, mC, -1.f, D, D, deep ? mD : none, D, none, true, leaf_size(w)))) return rc;
    if ((rc = inv32_b(bt, D, mD, h, true, sub, s, upper))) return rc;
    // C = -Si T, B = its transpose
    if ((rc = product(mD, mTT, -1.f, nullptr, C, want_mirror ? mC : none, upper ? B : nullptr, mB, false))) return rc;
    // A = Ai + V^T T = Ai - B T
    const Mirror *const sA = want_mirror ? mA : none;
    return product(mB, mTT, -1.f, A, A, sA, upper ? A : nullptr, sA, true);
}

// The G_j of a context in split form: slot j, or with recomputation the slot of j's position.
int row_pos(const apf_ctx *c, int row) {
    const int m = c->h / 2;
    return row < m ? row : row == m ? c->h - 1 : m + (c->h - 1 - row);
}
int pos_row(const apf_ctx *c, int p) {
    const int m = c->h / 2;
    return p < m ? p : p == c->h - 1 ? m : c->h - 1 - (p - m);
}
Mirror gp_view(const apf_ctx *c, int row) {
    const MixedWork *w = c->mw;
    const int slot = w->seg_rows > 0 ? row_pos(c, row) % w->seg_rows : row;
    return Mirror{w->GP + slot * w->gp_stride, c->nx, (long long)c->nx * c->nx};
}

// Launch one k_row_step per problem of `bt` (n: block size; jobs without an
// output and sources do nothing).
void row_step_b(const Bat &bt, const RowJob *jobs, int nj, int n, bool bf, cudaStream_t s) {
    apf_ctx *c = bt.lead();
    const MixedWork *w = c->mw;
    const int leaf = std::min(leaf_size(w), n);
    const GridDev g = make_grid(c);
    const dim3 grid((unsigned)(((long long)(n / 4) * (n / 8) + 127) / 128), 1, nj);
    bool two = false;
    for (int i = 0; i < nj; ++i) two = two || jobs[i].s[1].re;
    auto run = [&](auto &pack) {
        for (int i = 0; i < nj; ++i) pack.j[i] = jobs[i];
        constexpr int N = sizeof(pack.j) / sizeof(RowJob);
        auto launch = [&](auto kernel) {
            APF_LAUNCH(c, kernel, grid, 128, 0, s, g, pack, n, (const double2 *)c->d_circ, (const float *)w->BW, w->nsplit_elim, leaf);
        };
        if (bf) two ? launch(k_row_step<true, true, N>) : launch(k_row_step<true, false, N>);
        else two ? launch(k_row_step<false, true, N>) : launch(k_row_step<false, false, N>);
    };
    if (nj <= 2) {
        RowJobs<2> p{};
        run(p);
    } else {
        RowJobs<CG_MAX_PROB> p{};
        run(p);
    }
}

bool uses_butterfly(const MixedWork *w, int n) { return w->bfly && n > leaf_size(w) && n >= 16; }

// The working block of problem b, as a source (its transformed inverse) and as
// the block to write.
RowSrc work_src(const SideWork &w, bool use) {
    RowSrc s{};
    s.re = w.Xre; s.im = w.Xim;
    s.yspace = 1;
    s.use = use ? 1 : 0;
    return s;
}
RowJob row_job(const apf_ctx *c, const SideWork &w, int row) {
    RowJob j{};
    j.eps = c->d_eps;
    j.row = row;
    j.out = row >= 0 ? 1 : 0;
    j.sgn = -1.f;
    j.Xre = w.Xre; j.Xim = w.Xim;
    j.XP = w.XP;
    return j;
}

int invert_work_b(const Bat &bt, cudaStream_t s) {
    const int n = bt.lead()->nx;
    PV X[CG_MAX_PROB];
    Mirror XP[CG_MAX_PROB];
    for (int b = 0; b < bt.n; ++b) {
        X[b] = PV{bt.w(b).Xre, bt.w(b).Xim, n};
        XP[b] = bt.w(b).XP;
    }
    return inv32_b(bt, X, XP, n, false, 0, s);
}

// E ~= Khat^-1 R with the stored (or recomputed) G_j of each design: the
// right-hand sides are carried along both chains to the middle row, solved
// there, and substituted back outwards.  R(b, j): row j of design b's right-hand
// side (null: zero); Y: rows kept on the way in; E: the solution, written, or
// added to with `accumulate` (then Y is another array).  full: all columns are
// carried by both chains, else the inputs [0, cf) by the lower and the outputs
// [cf, ncol) by the upper one (where R is not zero).
template <typename F>
int approx_solve_b(const Bat &bt, F R, double2 *const *Y, double2 *const *E, bool accumulate, bool full, cudaStream_t s) {
    apf_ctx *c = bt.lead();
    MixedWork *w = c->mw;
    const int nb = bt.n, ncol = c->cf + c->ca, nx = c->nx, h = c->h, m = h / 2, top = h - 1 - m;
    const int planes = w->nsplit_elim, K = w->seg_rows;
    const long long L = (long long)ncol * nx;
    const int lo[2] = {0, full ? 0 : c->cf}, hi[2] = {full ? ncol : c->cf, ncol};  // columns of each chain
    // with recomputation: the segment whose inverses `row` needs must be loaded
    auto need = [&](int row) -> int {
        if (K <= 0) return APF_OK;
        const int sg = row_pos(c, row) / K;
        if (sg == w->seg_loaded) return APF_OK;
        return recompute_segment_b(bt, sg, s);
    };
    auto side = [&](int b, int sd) -> SideWork & { return bt.c[b]->mw->sd[sd]; };
    const int form_rows = full ? ncol : std::max(c->cf, c->ca);  // the same for both chains and in every step
    // O32 of each chain <- (operand of the chain) G_row^T for the chains that take part
    auto multiply = [&](const int *row, const int *cols) -> int {
        CgProblem pb[CG_MAX_PROB];
        int n = 0, M = 0;
        for (int sd = 0; sd < 2; ++sd) {
            if (row[sd] < 0 || cols[sd] <= 0) continue;
            if (int rc = need(row[sd])) return rc;
            M = std::max(M, cols[sd]);
            for (int b = 0; b < nb; ++b) {
                SideWork &sw = side(b, sd);
                CgProblem &p = pb[n++];
                p.A = sw.PA;
                p.B = gp_view(bt.c[b], row[sd]);
                p.M = cols[sd];
                p.out = CgOut{sw.O32, sw.O32 + L, nx, Mirror{}};
                p.flags = bt.c[b]->d_flags;
            }
        }
        return n ? cgemm_n(c, n, pb, planes, M, nx, nx, 1.f, 0.f, false, true, s, form_rows) : APF_OK;
    };
    FieldJob fj[CG_MAX_PROB];
    int nj = 0;
    auto push = [&](const FieldJob &j) {
        if (j.c1 > j.c0) fj[nj++] = j;
    };
    auto flush = [&]() {
        if (!nj) return;
        int rows = 0;
        for (int i = 0; i < nj; ++i) rows = std::max(rows, fj[i].c1 - fj[i].c0);
        const int threads = nx >= 256 ? 128 : 32;
        const dim3 grid((nx / 2 + threads - 1) / threads, rows, nj);
        auto run = [&](auto &pack) {
            for (int i = 0; i < nj; ++i) pack.j[i] = fj[i];
            constexpr int N = sizeof(pack.j) / sizeof(FieldJob);
            APF_LAUNCH(c, k_field_step<N>, grid, threads, 0, s, pack, nx, planes);
        };
        if (nj <= 2) {
            FieldJobs<2> p{};
            run(p);
        } else {
            FieldJobs<CG_MAX_PROB> p{};
            run(p);
        }
        nj = 0;
    };
    // one design's jobs at a time in Y / R rows; chain sd's row t steps from its end
    auto chain_row = [&](int sd, int t) { return sd ? h - 1 - t : t; };
    const int len[2] = {m, top};
    // carried rows: row t's operand (Y_t = R_t + O) and, past the end row, Y_t itself
    auto carry = [&](int b, int sd, int t) {
        SideWork &sw = side(b, sd);
        const int row = chain_row(sd, t);
        FieldJob j{};
        j.O = t > 0 ? sw.O32 : nullptr;
        j.olen = L;
        j.o0 = lo[sd]; j.o1 = hi[sd];
        j.add = R(b, row);
        j.a0 = 0; j.a1 = ncol;
        if (t > 0) { j.out = Y[b] + row * L; j.mode = 1; }
        j.m = sw.PA;
        j.c0 = lo[sd]; j.c1 = hi[sd];
        push(j);
    };
    // inwards; with recomputation one chain after the other, so that each segment is loaded once
    auto inwards = [&](bool s0, bool s1) -> int {
        const bool on[2] = {s0 && m > 0 && hi[0] > lo[0], s1 && top > 0 && hi[1] > lo[1]};
        for (int sd = 0; sd < 2; ++sd)
            if (on[sd])
                for (int b = 0; b < nb; ++b) carry(b, sd, 0);
        flush();
        for (int t = 1; t <= std::max(on[0] ? m : 0, on[1] ? top : 0); ++t) {
            int row[2], cols[2];
            for (int sd = 0; sd < 2; ++sd) {
                row[sd] = on[sd] && t <= len[sd] ? chain_row(sd, t - 1) : -1;
                cols[sd] = hi[sd] - lo[sd];
            }
            if (int e = multiply(row, cols)) return e;
            for (int sd = 0; sd < 2; ++sd)
                if (on[sd] && t < len[sd])
                    for (int b = 0; b < nb; ++b) carry(b, sd, t);
            flush();
        }
        return APF_OK;
    };
    int rc = inwards(true, K <= 0);
    if (rc == APF_OK && K > 0) rc = inwards(false, true);
    if (rc) return rc;
    // the middle row: both chains' contributions, then its own inverse
    for (int b = 0; b < nb; ++b) {
        FieldJob j{};
        j.O = m > 0 && hi[0] > lo[0] ? side(b, 0).O32 : nullptr;
        j.O2 = top > 0 && hi[1] > lo[1] ? side(b, 1).O32 : nullptr;
        j.olen = L;
        j.o0 = lo[0]; j.o1 = hi[0]; j.p0 = lo[1]; j.p1 = hi[1];
        j.add = R(b, m);
        j.a0 = 0; j.a1 = ncol;
        j.m = side(b, 0).PA;
        j.c0 = 0; j.c1 = ncol;
        push(j);
    }
    flush();
    {
        const int row[2] = {m, -1}, cols[2] = {ncol, 0};
        if ((rc = multiply(row, cols))) return rc;
    }
    // outwards: E_row = o (in O32 of `from`), and chain sd's next operand, Y_next + o
    auto outward = [&](int b, int sd, int row, const SideWork &from, bool store) {
        const int next = sd ? row + 1 : row - 1;
        FieldJob j{};
        j.O = from.O32;
        j.olen = L;
        j.o0 = 0; j.o1 = ncol;
        if (store) { j.out = E[b] + row * L; j.mode = accumulate ? 3 : 2; }
        if (next >= 0 && next < h) {
            // (on the chain's end row nothing was added to R)
            j.add = next == chain_row(sd, 0) ? R(b, next) : Y[b] + next * L;
            j.a0 = lo[sd]; j.a1 = hi[sd];
            j.m = side(b, sd).PA;
        }
        j.c0 = 0; j.c1 = ncol;
        push(j);
    };
    for (int b = 0; b < nb; ++b) {
        outward(b, 0, m, side(b, 0), true);
        if (top > 0) outward(b, 1, m, side(b, 0), false);
    }
    flush();
    auto outwards = [&](bool s0, bool s1) -> int {
        for (int t = 1; t <= std::max(s0 ? m : 0, s1 ? top : 0); ++t) {
            const int row[2] = {s0 && t <= m ? m - t : -1, s1 && t <= top ? m + t : -1}, cols[2] = {ncol, ncol};
            if (int e = multiply(row, cols)) return e;
            for (int sd = 0; sd < 2; ++sd)
                if (row[sd] >= 0)
                    for (int b = 0; b < nb; ++b) outward(b, sd, row[sd], side(b, sd), true);
            flush();
        }
        return APF_OK;
    };
    if (K <= 0) return outwards(true, true);
    if ((rc = outwards(false, true))) return rc;  // the upper chain first: segment 0 is loaded at the end
    return outwards(true, false);
}

// r = R - K E and the squared column norms of r (rhs), or r = K E (not rhs), for
// every design: E(b), r(b) fields.
template <typename FE, typename FR>
void residual_b(const Bat &bt, FE E, FR r, bool rhs, cudaStream_t s) {
    apf_ctx *c = bt.lead();
    const int ncol = c->cf + c->ca, nx = c->nx, nb = bt.n;
    const long long L = (long long)ncol * nx;
    int logn = 0;
    while ((1 << logn) < nx) ++logn;
    const int threads = nx / 2 < 256 ? nx / 2 : 256;
    const auto Et = tab<const double2 *>(bt, [&](int b) { return (const double2 *)E(b); });
    const auto cb = tab<double2 *>(bt, [&](int b) { return bt.c[b]->mw->cb; });
    const auto ct = tab<double2 *>(bt, [&](int b) { return bt.c[b]->mw->ct; });
    const auto part = tab<double *>(bt, [&](int b) { return rhs ? bt.c[b]->mw->rpart : nullptr; });
    APF_LAUNCH(c, k_circ_apply, dim3(ncol, 2, nb), threads, nx * (int)sizeof(double2), s, Et, (c->h - 1) * L, cb, ct, nx,
               logn, (const double2 *)c->d_modes, (const double2 *)c->d_tw);
    const dim3 grid((nx + 127) / 128, (ncol + RC - 1) / RC, nb);
    APF_LAUNCH(c, k_residual, grid, 128, 0, s, make_grid(c),
               tab<const double *>(bt, [&](int b) { return (const double *)bt.c[b]->d_eps; }), Et,
               tab<const double2 *>(bt, [&](int b) { return rhs ? (const double2 *)bt.c[b]->d_R : nullptr; }), cb, ct,
               tab<double2 *>(bt, [&](int b) { return (double2 *)r(b); }), part, ncol);
    if (rhs)
        APF_LAUNCH(c, k_normsum, dim3(ncol, 1, nb), 32, 0, s, part, (int)grid.x,
                   tab<double *>(bt, [&](int b) { return bt.c[b]->mw->rnorm + ncol; }));
}

}  // namespace

void mixed_init_attrs() {
    tc_init_attrs();
    cgemm_init_attrs();
    cudaFuncSetAttribute(k_leaf_inv32, cudaFuncAttributeMaxDynamicSharedMemorySize, 128 * 128 * (int)sizeof(float2));
    cudaFuncSetAttribute(k_leaf32<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, leaf_smem_bytes<128>(8));
    cudaFuncSetAttribute(k_leaf_cluster<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(lc::Smem<4>));
    cudaFuncSetAttribute(k_leaf_cluster<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(lc::Smem<2>));
    cudaFuncSetAttribute(k_circ_apply, cudaFuncAttributeMaxDynamicSharedMemorySize, 8192 * (int)sizeof(double2));
}

void mixed_free(apf_ctx *c) {
    if (!c->mw) return;
    for (void *p : c->mw->allocs) cudaFree(p);
    delete c->mw;
    c->mw = nullptr;
}

int mixed_alloc(apf_ctx *c) {
    mixed_free(c);
    MixedWork *w = new MixedWork();
    c->mw = w;
    w->nsplit_elim = c->elim_planes;
    if (const char *e = getenv("APF_NSPLIT_ELIM")) {  // tuning knob: bf16 planes of the elimination (2 or 3)
        int v = atoi(e);
        if (v == 2 || v == 3) w->nsplit_elim = v;
    }
    if (const char *e = getenv("APF_LEAF_VARIANT")) {  // tuning knob: 128-block leaf kernel (0..3)
        int v = atoi(e);
        if (v >= 0 && v <= 3) w->leaf_variant = v;
    }
    const long long n = c->nx, h = c->h, q = 2 * w->nsplit_elim;  // q: component planes of a split matrix
    const int nin = c->nin, nout = c->nout;
    const long long ncol = std::max(nin + nout, nin);
    w->seg_rows = (c->schur_seg > 0 && c->schur_seg < h) ? c->schur_seg : 0;
    w->nseg = w->seg_rows > 0 ? (int)((h + w->seg_rows - 1) / w->seg_rows) : 1;
    w->nside = w->seg_rows > 0 || h < 3 ? 1 : 2;  // chains eliminated at the same time
    int rc;
#define WA(p, cnt) if ((rc = walloc(c, w, &(p), (cnt))) != APF_OK) return rc;
    for (int sd = 0; sd < 2; ++sd) {
        SideWork &sw = w->sd[sd];
        if (sd < w->nside) {
            WA(sw.Xre, n * n); WA(sw.Xim, n * n);
            WA(sw.XP.base, q * n * n);
            sw.XP.pitch = n; sw.XP.qpitch = n * n;
            // T of the levels n/2, n/4, ..: q (n^2/4 + n^2/16 + ..) < q n^2 / 3
            WA(sw.TP, q * (n * n * 11 / 32 + 64)); WA(sw.TT, q * (n * n * 11 / 32 + 64));
        }
        WA(sw.O32, 2 * ncol * n);
        WA(sw.PA.base, q * ncol * n);
        sw.PA.pitch = n; sw.PA.qpitch = ncol * n;
    }
    const long long kp_g = round_up(2LL * nin, 64);
    WA(w->GA, (long long)nout * kp_g * w->nsplit_grad);
    WA(w->GB, 2 * n * kp_g * w->nsplit_grad);
    if (const char *e = getenv("APF_BUTTERFLY")) w->bfly = (e[0] == '1');  // diagnostic knob; default from ctx
    else w->bfly = c->butterfly;
    WA(w->BW, 2 * n);
    {
        // random diagonals exp(rho / 10), rho uniform in [-1/2, 1/2) (splitmix64, fixed seed)
        std::vector<float> bw(2 * n);
        uint64_t z = 0x9E3779B97F4A7C15ull ^ (uint64_t)n;
        for (long long i = 0; i < 2 * n; ++i) {
            z += 0x9E3779B97F4A7C15ull;
            uint64_t x = z;
            x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
            x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
            x ^= x >> 31;
            const double rho = (double)(x >> 11) * (1.0 / 9007199254740992.0) - 0.5;
            bw[i] = (float)exp(rho / 10.0);
        }
        cudaError_t e = cudaMemcpyAsync(w->BW, bw.data(), sizeof(float) * 2 * n, cudaMemcpyHostToDevice, c->cap_stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(c->cap_stream);
        if (e != cudaSuccess) return check_cuda(c, e, "butterfly weights");
    }
    w->gp_stride = q * n * n;
    const long long slots = w->seg_rows > 0 ? w->seg_rows : h;
    WA(w->GP, slots * w->gp_stride);
    if (w->seg_rows > 0) {
        WA(w->CK, (long long)(w->nseg - 1) * 2 * n * n);
        WA(w->CKB, 2 * n * n);
    }
    WA(w->r, h * ncol * n); WA(w->delta, h * ncol * n);
    WA(w->cb, ncol * n); WA(w->ct, ncol * n);
    WA(w->rnorm, 2 * ncol); WA(w->rpart, ncol * ((n + 127) / 128));
    w->km = c->krylov_m;
    if (w->km > 0) {
        WA(w->KV, (long long)(w->km + 1) * h * ncol * n);
        WA(w->KZ, (long long)w->km * h * ncol * n);
        WA(w->kdot, (long long)(w->km + 1) * w->km * ncol);
        WA(w->ky, (long long)w->km * ncol);
        WA(w->knrm, (long long)w->km * ncol);
    }
#undef WA
    return APF_OK;
}

// Positions [p0, p1) of the chain order, one row at a time on the first side's
// work arrays (recomputation of the slab inverses): the elimination (p0 = 0, p1 =
// h) or one segment from the checkpoint before it.
static int eliminate_positions(const Bat &bt, int p0, int p1, cudaStream_t s) {
    apf_ctx *c = bt.lead();
    const MixedWork *w = c->mw;
    const int n = c->nx, h = c->h, m = h / 2, K = w->seg_rows, nb = bt.n;
    const long long nn = (long long)n * n;
    const bool bf = uses_butterfly(w, n);
    RowJob jobs[CG_MAX_PROB];
    auto plane = [&](float *p) {  // a checkpoint as a source
        RowSrc src{};
        src.re = p; src.im = p + nn;
        src.use = 1;
        return src;
    };
    for (int p = p0; p <= p1; ++p) {
        const bool more = p < p1;
        const bool middle = p == h - 1, first_up = p == m && !middle;
        const bool two = middle && m < h - 1;  // the middle row takes both chains
        for (int b = 0; b < nb; ++b) {
            MixedWork *wb = bt.c[b]->mw;
            RowJob &j = jobs[b];
            j = row_job(bt.c[b], wb->sd[0], more ? pos_row(c, p) : -1);
            RowSrc prev{};
            if (p > p0) {  // the inverse just computed: into its slot, and kept where a later step starts from it
                prev = work_src(wb->sd[0], more && !first_up);
                prev.gp = gp_view(bt.c[b], pos_row(c, p - 1));
                float *ck = p == m && m < h - 1 ? wb->CKB : p < h && p % K == 0 ? wb->CK + (long long)(p / K - 1) * 2 * nn : nullptr;
                if (ck) { prev.ck_re = ck; prev.ck_im = ck + nn; }
            } else if (p > 0 && !first_up) {
                prev = plane(wb->CK + (long long)(p / K - 1) * 2 * nn);
            }
            if (two && more) {
                if (m > 0) j.s[0] = plane(wb->CKB);
                j.s[1] = prev;
            } else {
                j.s[0] = prev;
            }
        }
        row_step_b(bt, jobs, nb, n, bf, s);
        if (more)
            if (int rc = invert_work_b(bt, s)) return rc;
    }
    return APF_OK;
}

int mixed_eliminate_b(const Bat &bt, cudaStream_t s) {
    apf_ctx *c = bt.lead();
    for (int b = 0; b < bt.n; ++b)
        if (!bt.c[b]->mw) return set_err(bt.c[b], APF_ESTATE, "mixed workspace missing");
    MixedWork *w = c->mw;
    const int n = c->nx, h = c->h, m = h / 2, top = h - 1 - m, nb = bt.n;
    if (w->seg_rows > 0) {
        int rc = eliminate_positions(bt, 0, h, s);
        for (int b = 0; b < nb; ++b) bt.c[b]->mw->seg_loaded = (h - 1) / w->seg_rows;
        return rc;
    }
    const bool bf = uses_butterfly(w, n);
    RowJob jobs[CG_MAX_PROB];
    // both chains: the rows t and h - 1 - t of every design in the same launches
    for (int t = 0; t < m; ++t) {
        Bat both;
        for (int sd = 0; sd < (t < top ? 2 : 1); ++sd)
            for (int b = 0; b < nb; ++b) both.add(bt.c[b], sd);
        for (int b = 0; b < both.n; ++b) {
            const int sd = both.sd[b], row = sd ? h - 1 - t : t;
            jobs[b] = row_job(both.c[b], both.w(b), row);
            if (t > 0) {
                jobs[b].s[0] = work_src(both.w(b), true);
                jobs[b].s[0].gp = gp_view(both.c[b], sd ? row + 1 : row - 1);
            }
        }
        row_step_b(both, jobs, both.n, n, bf, s);
        if (int rc = invert_work_b(both, s)) return rc;
    }
    // the middle row
    for (int b = 0; b < nb; ++b) {
        MixedWork *wb = bt.c[b]->mw;
        jobs[b] = row_job(bt.c[b], wb->sd[0], m);
        if (m > 0) {
            jobs[b].s[0] = work_src(wb->sd[0], true);
            jobs[b].s[0].gp = gp_view(bt.c[b], m - 1);
        }
        if (top > 0) {
            jobs[b].s[1] = work_src(wb->sd[1], true);
            jobs[b].s[1].gp = gp_view(bt.c[b], m + 1);
        }
    }
    row_step_b(bt, jobs, nb, n, bf, s);
    if (int rc = invert_work_b(bt, s)) return rc;
    for (int b = 0; b < nb; ++b) {
        jobs[b] = row_job(bt.c[b], bt.c[b]->mw->sd[0], -1);
        jobs[b].s[0] = work_src(bt.c[b]->mw->sd[0], false);
        jobs[b].s[0].gp = gp_view(bt.c[b], m);
    }
    row_step_b(bt, jobs, nb, n, bf, s);
    return APF_OK;
}

int mixed_eliminate(apf_ctx *c, cudaStream_t s) { return mixed_eliminate_b(one(c), s); }

// Recompute the split inverses of segment `seg` into the GP slots of every
// design, from the float32 checkpoint before it and by the same kernels as the
// elimination (bit-identical results).
int recompute_segment_b(const Bat &bt, int seg, cudaStream_t s) {
    apf_ctx *c = bt.lead();
    const int K = c->mw->seg_rows;
    int rc = eliminate_positions(bt, seg * K, std::min(c->h, (seg + 1) * K), s);
    for (int b = 0; b < bt.n; ++b) bt.c[b]->mw->seg_loaded = seg;
    return rc;
}

// The column norms of the right-hand side (its two rows in d_R, see
// launch_build_rhs) and the first low-precision solve E = Khat^-1 R.
int mixed_fields_begin_b(const Bat &bt, cudaStream_t s) {
    double2 *E[CG_MAX_PROB];
    apf_ctx *c0 = bt.lead();
    const int ncol = c0->cf + c0->ca, h = c0->h;
    const long long L = (long long)ncol * c0->nx;
    for (int b = 0; b < bt.n; ++b) {
        apf_ctx *c = bt.c[b];
        APF_LAUNCH(c, k_colnorm, ncol, 256, 0, s, (const double2 *)c->d_R, std::min(h, 2), ncol, c->nx, c->mw->rnorm);
        E[b] = c->d_Ew;
    }
    auto R = [&](int b, int row) -> const double2 * {
        return row == 0 ? bt.c[b]->d_R : row == h - 1 ? bt.c[b]->d_R + L : nullptr;
    };
    return approx_solve_b(bt, R, E, E, false, false, s);
}

int mixed_fields_begin(apf_ctx *c, cudaStream_t s) { return mixed_fields_begin_b(one(c), s); }

static void resid_b(const Bat &bt, cudaStream_t s) {
    residual_b(bt, [&](int b) { return bt.c[b]->d_Ew; }, [&](int b) { return bt.c[b]->mw->r; }, true, s);
}

static int resid_body(apf_ctx *c, cudaStream_t s) {
    resid_b(one(c), s);
    return APF_OK;
}

// E += Khat^-1 r for every design of the batch.
static int correct_b(const Bat &bt, cudaStream_t s) {
    double2 *Y[CG_MAX_PROB], *E[CG_MAX_PROB];
    for (int b = 0; b < bt.n; ++b) {
        Y[b] = bt.c[b]->mw->delta;
        E[b] = bt.c[b]->d_Ew;
    }
    const long long L = (long long)(bt.lead()->cf + bt.lead()->ca) * bt.lead()->nx;
    auto R = [&](int b, int row) -> const double2 * { return bt.c[b]->mw->r + row * L; };
    return approx_solve_b(bt, R, Y, E, true, true, s);
}

static int correct_body(apf_ctx *c, cudaStream_t s) { return correct_b(one(c), s); }

// Diagnostics: APF_IR_VERBOSE=1 prints the residual of every refinement step.
static const bool g_ir_verbose = [] {
    const char *e = getenv("APF_IR_VERBOSE");
    return e && e[0] == '1';
}();

// K E (the slab operator in float64) into out.
static void apply_K(apf_ctx *c, const double2 *E, double2 *out, cudaStream_t s) {
    residual_b(one(c), [&](int) { return E; }, [&](int) { return out; }, false, s);
}

// min || beta e1 - H y || for one column by complex Givens rotations; H is
// (m+1) x m upper Hessenberg, H[i][j] at h[i * m + j].
static void hessenberg_lsq(int m, std::vector<std::complex<double>> &h, double beta, std::complex<double> *y) {
    std::vector<std::complex<double>> g(m + 1, 0.0), cs(m), sn(m);
    std::vector<double> cr(m);
    g[0] = beta;
    for (int j = 0; j < m; ++j) {
        for (int i = 0; i < j; ++i) {
            const std::complex<double> a = h[i * m + j], b = h[(i + 1) * m + j];
            h[i * m + j] = cr[i] * a + sn[i] * b;
            h[(i + 1) * m + j] = -std::conj(sn[i]) * a + cr[i] * b;
        }
        const std::complex<double> a = h[j * m + j], b = h[(j + 1) * m + j];
        const double na = std::abs(a), nb = std::abs(b);
        if (nb == 0.0) {
            cr[j] = 1.0; sn[j] = 0.0;
        } else if (na == 0.0) {
            cr[j] = 0.0; sn[j] = std::conj(b) / nb;
        } else {
            const double nr = std::sqrt(na * na + nb * nb);
            cr[j] = na / nr;
            sn[j] = (a / na) * std::conj(b) / nr;
        }
        h[j * m + j] = cr[j] * a + sn[j] * b;
        h[(j + 1) * m + j] = 0.0;
        const std::complex<double> g0 = g[j], g1 = g[j + 1];
        g[j] = cr[j] * g0 + sn[j] * g1;
        g[j + 1] = -std::conj(sn[j]) * g0 + cr[j] * g1;
    }
    for (int j = m - 1; j >= 0; --j) {
        std::complex<double> t = g[j];
        for (int k = j + 1; k < m; ++k) t -= h[j * m + k] * y[k];
        y[j] = std::abs(h[j * m + j]) > 0.0 ? t / h[j * m + j] : 0.0;
    }
}

// Float64 refinement by restarted GMRES(m), right-preconditioned by the
// low-precision factorization Khat^-1 (a fixed linear operator), one Krylov
// space per right-hand-side column: from the true residual r = R - K E,
// V_0 = r / ||r||; Z_j = Khat^-1 V_j, W = K Z_j orthogonalised against
// V_0..V_j (modified Gram-Schmidt, per-column coefficients kept on the
// device), V_{j+1} = W / ||W||; then E += sum_j y_j Z_j with y the
// per-column least-squares solution of the (m+1) x m Hessenberg system.
// The stopping rule and the iteration count (preconditioner applications)
// are those of the plain refinement.
static int mixed_refine_gmres(apf_ctx *c, cudaStream_t s) {
    MixedWork *w = c->mw;
    const int m = w->km, ncol = c->cf + c->ca, nx = c->nx;
    const long long L = (long long)c->h * ncol * nx;
    const dim3 fgrid((nx + 255) / 256, ncol, c->h);
    std::vector<double> nr(ncol), ne(ncol), hn((size_t)m * ncol);
    std::vector<double2> hd((size_t)(m + 1) * m * ncol), yh((size_t)m * ncol);
    std::vector<std::complex<double>> H((size_t)(m + 1) * m), y(m);
    int iters = 0, rc, rising = 0;
    double ratio = 0.0, prev = INFINITY;
    cudaMemcpyAsync(nr.data(), w->rnorm, sizeof(double) * ncol, cudaMemcpyDeviceToHost, s);
    for (;;) {
        resid_b(one(c), s);
        cudaMemcpyAsync(ne.data(), w->rnorm + ncol, sizeof(double) * ncol, cudaMemcpyDeviceToHost, s);
        cudaError_t e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return check_cuda(c, e, "refinement");
        if (c->prof_on && iters == 0) prof_collect_range(c, c->g_main[c->lay].prof_lo, c->g_main[c->lay].prof_hi);
        ratio = 0.0;
        for (int i = 0; i < ncol; ++i) ratio = std::max(ratio, sqrt(ne[i] / std::max(nr[i], 1e-300)));
        if (g_ir_verbose)
            fprintf(stderr, "apf refinement (GMRES(%d)): %d preconditioner applications, max relative residual %.3e\n",
                    m, iters, ratio);
        if (!(ratio == ratio)) { ratio = INFINITY; break; }
        if (ratio <= c->ir_tol || iters >= c->ir_max) break;
        rising = ratio > prev ? rising + 1 : 0;
        if (rising >= 2) break;
        prev = ratio;
        // Arnoldi on K Khat^-1 from V_0 = r / ||r||
        APF_LAUNCH(c, k_colscale, fgrid, 256, 0, s, w->KV, w->r, w->rnorm + ncol, ncol, nx);
        for (int j = 0; j < m; ++j) {
            double2 *Vj = w->KV + j * L, *Wn = w->KV + (j + 1) * L, *Zj = w->KZ + j * L;
            const long long row = (long long)ncol * nx;
            auto R = [&](int, int j2) -> const double2 * { return Vj + j2 * row; };
            if ((rc = approx_solve_b(one(c), R, &Zj, &Zj, false, true, s))) return rc;
            apply_K(c, Zj, Wn, s);
            for (int i = 0; i <= j; ++i) {
                double2 *hij = w->kdot + ((long long)j * (m + 1) + i) * ncol;
                APF_LAUNCH(c, k_coldot, ncol, 256, 0, s, w->KV + i * L, Wn, c->h, ncol, nx, hij);
                APF_LAUNCH(c, k_colaxpy, fgrid, 256, 0, s, Wn, w->KV + i * L, hij, -1.0, ncol, nx);
            }
            APF_LAUNCH(c, k_colnorm, ncol, 256, 0, s, Wn, c->h, ncol, nx, w->knrm + (long long)j * ncol);
            APF_LAUNCH(c, k_colscale, fgrid, 256, 0, s, Wn, Wn, w->knrm + (long long)j * ncol, ncol, nx);
        }
        cudaMemcpyAsync(hd.data(), w->kdot, sizeof(double2) * hd.size(), cudaMemcpyDeviceToHost, s);
        cudaMemcpyAsync(hn.data(), w->knrm, sizeof(double) * hn.size(), cudaMemcpyDeviceToHost, s);
        e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return check_cuda(c, e, "arnoldi");
        for (int col = 0; col < ncol; ++col) {
            std::fill(H.begin(), H.end(), std::complex<double>(0.0, 0.0));
            for (int j = 0; j < m; ++j) {
                for (int i = 0; i <= j; ++i) {
                    const double2 v = hd[((size_t)j * (m + 1) + i) * ncol + col];
                    H[(size_t)i * m + j] = std::complex<double>(v.x, v.y);
                }
                H[(size_t)(j + 1) * m + j] = std::sqrt(std::max(hn[(size_t)j * ncol + col], 0.0));
            }
            hessenberg_lsq(m, H, std::sqrt(std::max(ne[col], 0.0)), y.data());
            for (int j = 0; j < m; ++j) yh[(size_t)j * ncol + col] = make_double2(y[j].real(), y[j].imag());
        }
        cudaMemcpyAsync(w->ky, yh.data(), sizeof(double2) * yh.size(), cudaMemcpyHostToDevice, s);
        for (int j = 0; j < m; ++j)
            APF_LAUNCH(c, k_colaxpy, fgrid, 256, 0, s, c->d_Ew, w->KZ + j * L, w->ky + (long long)j * ncol, 1.0,
                       ncol, nx);
        iters += m;
    }
    c->stats.refine_iters = iters;
    c->stats.residual = ratio;
    return ratio <= c->ir_tol ? APF_OK : APF_ENOCONV;
}

// Float64 iterative refinement: r = R - K E, E += Khat^-1 r until
// max_c ||r_c|| / ||R_c|| <= tol (or max_iters corrections).
int mixed_refine(apf_ctx *c, cudaStream_t s) {
    MixedWork *w = c->mw;
    if (w->km > 0) return mixed_refine_gmres(c, s);
    int ncol = c->cf + c->ca;
    std::vector<double> nr(ncol), ne(ncol);
    int iters = 0, rc, rising = 0;
    double ratio = 0.0, prev = INFINITY;
    for (;;) {
        if ((rc = run_graph(c, c->g_resid[c->lay], s, resid_body))) return rc;
        cudaMemcpyAsync(nr.data(), w->rnorm, sizeof(double) * ncol, cudaMemcpyDeviceToHost, s);
        cudaMemcpyAsync(ne.data(), w->rnorm + ncol, sizeof(double) * ncol, cudaMemcpyDeviceToHost, s);
        cudaError_t e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return check_cuda(c, e, "refinement");
        if (c->prof_on) {
            const GraphSlot &g = iters == 0 ? c->g_main[c->lay] : c->g_correct[c->lay];
            prof_collect_range(c, g.prof_lo, g.prof_hi);
        }
        ratio = 0.0;
        for (int i = 0; i < ncol; ++i) ratio = std::max(ratio, sqrt(ne[i] / std::max(nr[i], 1e-300)));
        if (g_ir_verbose) fprintf(stderr, "apf refinement: iteration %d, max relative residual %.3e\n", iters, ratio);
        if (!(ratio == ratio)) { ratio = INFINITY; break; }
        if (ratio <= c->ir_tol || iters >= c->ir_max) break;
        // diverging: the residual grew on two consecutive sweeps
        rising = ratio > prev ? rising + 1 : 0;
        if (rising >= 2) break;
        prev = ratio;
        if ((rc = run_graph(c, c->g_correct[c->lay], s, correct_body))) return rc;
        ++iters;
    }
    c->stats.refine_iters = iters;
    c->stats.residual = ratio;
    return ratio <= c->ir_tol ? APF_OK : APF_ENOCONV;
}

// Gradient contraction with tensor-core products for every design of the
// batch: Q_j = Gamma F_j, then g_j(x) = 2 k^2 Re sum_b Phi_j[b][x] Q_j[b][x] in
// float64.  Gamma[b]: the design's n_out x n_in Gamma on the device.
int mixed_gradient_b(const Bat &bt, const double2 *const *Gamma, cudaStream_t s) {
    apf_ctx *c = bt.lead();
    MixedWork *w = c->mw;
    const int nin = c->nin, nout = c->nout, ncol = nin + nout;
    const int nx = c->nx, ns = w->nsplit_grad, nb = bt.n;
    const long long L = (long long)ncol * nx;
    PackView pa[APF_MAX_BATCH], pb[APF_MAX_BATCH];
    __nv_bfloat16 *padst[APF_MAX_BATCH], *pbdst[APF_MAX_BATCH];
    PV Q[APF_MAX_BATCH];
    const double2 *src[APF_MAX_BATCH];
    for (int b = 0; b < nb; ++b) {
        MixedWork *wb = bt.c[b]->mw;
        padst[b] = wb->GA;
        pbdst[b] = wb->GB;
        Q[b] = PV{wb->sd[0].O32, wb->sd[0].O32 + (long long)nout * nx, nx};
    }
    pack64A_b(bt, pa, padst, Gamma, nin, nout, nin, ns, s);
    for (int j = 0; j < c->h; ++j) {
        for (int b = 0; b < nb; ++b) src[b] = bt.c[b]->d_E + j * L;
        pack64BT_b(bt, pb, pbdst, src, nx, nx, nin, ns, s);
        TcProblem pr[APF_MAX_BATCH];
        for (int b = 0; b < nb; ++b)
            pr[b] = TcProblem{pa[b], pb[b], Q[b].re, Q[b].im, bt.c[b]->d_flags};
        if (int rc = tc_gemm_n(c, nb, pr, ns, nout, 2 * nx, nx, nx, s)) return rc;
        APF_LAUNCH(c, k_grad_rowdot32, dim3((nx + 31) / 32, 1, nb), 256, 0, s,
                   tab<const double2 *>(bt, [&](int b) { return (const double2 *)bt.c[b]->d_E; }),
                   tab<const float *>(bt, [&](int b) { return (const float *)Q[b].re; }),
                   tab<const float *>(bt, [&](int b) { return (const float *)Q[b].im; }), j, nx, nin, nout,
                   c->k * c->k, tab<double *>(bt, [&](int b) { return bt.c[b]->d_grad; }));
    }
    return APF_OK;
}

int mixed_gradient(apf_ctx *c, const double2 *Gamma, cudaStream_t s) { return mixed_gradient_b(one(c), &Gamma, s); }

// Refinement of a batch of designs (no captured graphs): every sweep checks
// the residual of each design, and designs still above tolerance take one
// more correction, all of them in the same launches.  The stopping rule per
// design is that of mixed_refine.  rc[b]: APF_OK or APF_ENOCONV.
int mixed_refine_b(const Bat &bt, cudaStream_t s, int *rcs) {
    const int nb = bt.n;
    apf_ctx *c0 = bt.lead();
    const int ncol = c0->cf + c0->ca;
    std::vector<std::vector<double>> nr(nb, std::vector<double>(ncol)), ne(nb, std::vector<double>(ncol));
    std::vector<int> iters(nb, 0), rising(nb, 0), active(nb, 1);
    std::vector<double> ratio(nb, 0.0), prev(nb, INFINITY);
    for (;;) {
        Bat act;
        for (int b = 0; b < nb; ++b)
            if (active[b]) act.add(bt.c[b], 0);
        resid_b(act, s);
        for (int b = 0; b < nb; ++b) {
            if (!active[b]) continue;
            apf_ctx *c = bt.c[b];
            cudaMemcpyAsync(nr[b].data(), c->mw->rnorm, sizeof(double) * ncol, cudaMemcpyDeviceToHost, s);
            cudaMemcpyAsync(ne[b].data(), c->mw->rnorm + ncol, sizeof(double) * ncol, cudaMemcpyDeviceToHost, s);
        }
        cudaError_t e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return check_cuda(c0, e, "refinement");
        Bat next;
        for (int b = 0; b < nb; ++b) {
            if (!active[b]) continue;
            apf_ctx *c = bt.c[b];
            double r = 0.0;
            for (int i = 0; i < ncol; ++i) r = std::max(r, sqrt(ne[b][i] / std::max(nr[b][i], 1e-300)));
            ratio[b] = (r == r) ? r : INFINITY;
            bool stop = !(r == r) || r <= c->ir_tol || iters[b] >= c->ir_max;
            if (!stop) {
                rising[b] = r > prev[b] ? rising[b] + 1 : 0;
                stop = rising[b] >= 2;
            }
            prev[b] = r;
            if (stop) active[b] = 0;
            else next.add(c, 0);
        }
        if (next.n == 0) break;
        int rc = correct_b(next, s);
        if (rc) return rc;
        for (int b = 0; b < nb; ++b)
            if (active[b]) ++iters[b];
    }
    for (int b = 0; b < nb; ++b) {
        apf_ctx *c = bt.c[b];
        c->stats.refine_iters = iters[b];
        c->stats.residual = ratio[b];
        rcs[b] = ratio[b] <= c->ir_tol ? APF_OK : APF_ENOCONV;
    }
    return APF_OK;
}

// Entry points for a batch of contexts (apf_solve_S_grad_batch).
static Bat make_bat(apf_ctx *const *cs, int nb) {
    Bat bt;
    for (int b = 0; b < nb; ++b) bt.add(cs[b], 0);
    return bt;
}
int mixed_eliminate_n(apf_ctx *const *cs, int nb, cudaStream_t s) { return mixed_eliminate_b(make_bat(cs, nb), s); }
int mixed_fields_begin_n(apf_ctx *const *cs, int nb, cudaStream_t s) {
    return mixed_fields_begin_b(make_bat(cs, nb), s);
}
int mixed_refine_n(apf_ctx *const *cs, int nb, cudaStream_t s, int *rcs) {
    return mixed_refine_b(make_bat(cs, nb), s, rcs);
}
int mixed_gradient_n(apf_ctx *const *cs, int nb, cudaStream_t s) {
    const double2 *g[APF_MAX_BATCH];
    for (int b = 0; b < nb; ++b) g[b] = cs[b]->d_Gam;
    return mixed_gradient_b(make_bat(cs, nb), g, s);
}
// Settings that must agree across the designs of a batch (the launches are shared).
bool mixed_batch_compatible(const apf_ctx *a, const apf_ctx *b) {
    const MixedWork *x = a->mw, *y = b->mw;
    if (!x || !y) return false;
    return x->nsplit_elim == y->nsplit_elim && x->nsplit_grad == y->nsplit_grad && x->leaf == y->leaf &&
           x->leaf_variant == y->leaf_variant && x->seg_rows == y->seg_rows && x->bfly == y->bfly && x->km == 0 &&
           y->km == 0;
}

// ---------------------------------------------------------------------------
// Test hooks (not part of the public ABI in include/): exercise the splitting +
// tensor-core product and the mixed recursive inversion in isolation.  They
// allocate their own temporaries.
// ---------------------------------------------------------------------------
extern "C" int apf_debug_cgemm(apf_ctx *c, int m, int n, int k, const float *Are, const float *Aim,
                               const float *Bre, const float *Bim, float *Cre, float *Cim, int nsplit) {
    if (!c) return APF_EINVAL;
    SolveGate gate(c->device);
    if (m < 1 || n < 1 || k < 1 || nsplit < 1 || nsplit > 3) return APF_EINVAL;
    cudaSetDevice(c->device);
    const long long kp = round_up(k, 64);
    Mirror A{nullptr, kp, m * kp}, B{nullptr, kp, n * kp};
    const size_t abytes = sizeof(__nv_bfloat16) * 2 * nsplit * m * kp, bbytes = sizeof(__nv_bfloat16) * 2 * nsplit * n * kp;
    if (cudaMalloc(&A.base, abytes) != cudaSuccess) return APF_ENOMEM;
    if (cudaMalloc(&B.base, bbytes) != cudaSuccess) { cudaFree(A.base); return APF_ENOMEM; }
    int *flags = nullptr;
    if (cudaMalloc(&flags, 16) != cudaSuccess) { cudaFree(A.base); cudaFree(B.base); return APF_ENOMEM; }
    cudaStream_t s = 0;
    cudaMemsetAsync(A.base, 0, abytes, s);
    cudaMemsetAsync(B.base, 0, bbytes, s);
    cudaMemsetAsync(flags, 0, 16, s);
    const PV av{(float *)Are, (float *)Aim, k}, bv{(float *)Bre, (float *)Bim, n};
    mirror_b(one(c), &av, &A, m, k, false, nsplit, s);
    mirror_b(one(c), &bv, &B, n, k, true, nsplit, s);
    CgProblem p;
    p.A = A;
    p.B = B;
    p.M = m;
    p.out = CgOut{Cre, Cim, n, Mirror{}};
    p.flags = flags;
    int rc = cgemm_n(c, 1, &p, nsplit, m, n, k, 1.f, 0.f, false, true, s);
    cudaError_t e = cudaDeviceSynchronize();
    if (c->prof_on) prof_collect(c);  // GEMM event timings of this call
    int fl = 0;
    cudaMemcpy(&fl, flags, sizeof(int), cudaMemcpyDeviceToHost);
    cudaFree(flags);
    cudaFree(A.base);
    cudaFree(B.base);
    if (rc) return rc;
    if (e != cudaSuccess) return check_cuda(c, e, "debug cgemm");
    if (fl & FLAG_TIMEOUT) return set_err(c, APF_ETIMEOUT, "cgemm wait gave up");
    return APF_OK;
}

// In-place inverse of an n x n complex-symmetric planar float32 matrix using
// the workspace of a prepared mixed-precision context (n <= its nx).
extern "C" int apf_debug_inv32(apf_ctx *c, int n, float *re, float *im, int leaf) {
    if (!c) return APF_EINVAL;
    SolveGate gate(c->device);
    if (!c->mw || n < 1 || n > c->nx || (n & (n - 1))) return APF_EINVAL;
    cudaSetDevice(c->device);
    MixedWork *w = c->mw;
    const int old = w->leaf, oldv = w->leaf_variant;
    // leaf = block size + 1000 * kernel variant (test and tuning hook);
    // + 100000: through the symmetric random butterfly transform
    const bool bf = leaf >= 100000 && n >= 16;
    leaf %= 100000;
    // (blocks below 8 are taken as 8: a row of a product's operand is at least 16 bytes)
    if (leaf > 0) { w->leaf = std::max(8, leaf % 1000); w->leaf_variant = leaf / 1000; }
    cudaStream_t s = 0;
    cudaMemsetAsync(c->d_flags, 0, 16, s);
    const Bat bt = one(c);
    const PV X{w->sd[0].Xre, w->sd[0].Xim, n}, user{re, im, n};
    const Mirror XP{w->sd[0].XP.base, n, (long long)n * n};
    int rc = APF_OK;
    if (n < 8) {
        Mirror none;
        leaf_b(bt, &user, n, &none, s);
    } else {
        RowJob j = row_job(c, w->sd[0], -1);  // load: X = U^T user U
        j.s[0].re = re; j.s[0].im = im;
        j.s[0].use = 1;
        j.out = 1;
        j.sgn = 1.f;
        j.XP = XP;
        row_step_b(bt, &j, 1, n, bf, s);
        rc = inv32_b(bt, &X, &XP, n, false, 0, s);
        j = row_job(c, w->sd[0], -1);  // store: user = U X U^T
        j.s[0] = work_src(w->sd[0], false);
        j.s[0].ck_re = re; j.s[0].ck_im = im;
        if (rc == APF_OK) row_step_b(bt, &j, 1, n, bf, s);
    }
    cudaError_t e = cudaDeviceSynchronize();
    w->leaf = old;
    w->leaf_variant = oldv;
    if (rc) return rc;
    if (e != cudaSuccess) return check_cuda(c, e, "debug inv32");
    int fl2[2] = {0, 0};
    cudaMemcpy(fl2, c->d_flags, sizeof fl2, cudaMemcpyDeviceToHost);
    const int fl = fl2[0];
    c->stats.leaf_fallbacks = fl2[1];
    if (fl & FLAG_TIMEOUT) return set_err(c, APF_ETIMEOUT, "cgemm wait gave up");
    if (fl & FLAG_SINGULAR) return set_err(c, APF_ESINGULAR, "singular leaf");
    return APF_OK;
}
