// Float64 slab elimination: assembly of the slab Schur blocks X_j, a complex
// float64 GEMM, diagonal-block inversion, and the recursive inversion of the
// complex-symmetric X_j.
//
// In the pixel basis the slab rows j = 0..h-1 form a block-tridiagonal system
// with diagonal blocks K_j = T_x + 2 I - k^2 diag(eps_j) + 2 I (T_x the
// periodic second difference; the two y-couplings give the other 2 I),
// plus the boundary Schur blocks Sigma_bot on row 0 and Sigma_top on row h-1
// (circulants, diagonal in the Fourier basis), and off-diagonal blocks -I.
// Block elimination from both ends (eliminate64): X_0 = K_0, X_j = K_j - X_{j-1}^-1
// below the middle row, X_j = K_j - X_{j+1}^-1 above it (Schur complements of the
// rows outside; paper Sec. 2: S is a Schur complement of the augmented K,
// obtained here block row by block row).  Every X_j is complex symmetric
// (reciprocity, A = A^T), which the inversion exploits.
#include "apf_internal.h"
#include "leaf.cuh"

#include <algorithm>
#include <stdint.h>

namespace {

// X = K_row - Gp - Gq (either may be null).  blockIdx.z = 1: the second row of a
// pair (see eliminate64), at X + dX with its own previous inverse at Gp + dG.
__global__ void k_assemble64(GridDev g, int row, int row2, const double *eps, const double2 *circ,
                             const double2 *Gp, long long dG, const double2 *Gq, double2 *X, long long dX) {
    int xp = blockIdx.x * blockDim.x + threadIdx.x;
    int x = blockIdx.y;
    int n = g.nx;
    if (xp >= n) return;
    if (blockIdx.z == 1) {
        row = row2;
        X += dX;
        if (Gp) Gp += dG;
    }
    double2 v = cmk(0.0, 0.0);
    if (xp == x) v.x += 4.0 - g.k * g.k * eps[(long long)row * n + x];
    if (xp == (x + 1) % n) v.x -= 1.0;
    if (xp == (x + n - 1) % n) v.x -= 1.0;
    int d = (x - xp + n) % n;
    if (row == 0) v = cadd(v, circ[d]);
    if (row == g.h - 1) v = cadd(v, circ[n + d]);
    long long idx = (long long)x * n + xp;
    if (Gp) v = csub(v, Gp[idx]);
    if (Gq) v = csub(v, Gq[idx]);
    X[idx] = v;
}

// C = alpha op(A) B + beta C, row-major complex float64, batched over
// blockIdx.z (M2 > 0: the second entry of the batch has M2 rows instead of M).
//
// What bounds it is the float64 pipe: 2 FMA per clock and SM on GB300, so a
// product costs the same wherever it runs and only the split over the SMs
// counts (a 32^3 product on one SM is 65k clocks).  Hence small T x T tiles, one
// output per thread and k slice, as many of them as fill the chip: T = 16,
// 256 outputs, where that gives at least two tiles per SM, else T = 8 or 4
// with 4 or 16 k slices whose sums are added in a fixed order.  Operand traffic
// does not matter at this rate (T = 16: 0.5 KB of shared memory per 512 clocks).
// Measured inside a solve on GB300 against the 64 x 64 tiles these replace:
// two 32^3 products 177 -> 5.4 us, and with the elimination from both ends
// (eliminate64) the 1024 x 240 evaluation 658 -> 90 ms, 64 x 100 8.3 -> 0.84 ms.
//
// SYM: the result is known to be symmetric (Schur complements): only the tiles
// on and below the diagonal are computed and each element is written to both
// places, half the work.
struct ZArgs {
    int M, M2, N, K;
    double2 alpha, beta;
    const double2 *A, *B;
    double2 *C;
    long long lda, sA, ldb, sB, ldc, sC;
};

template <int T, bool TA, bool SYM>
__global__ void __launch_bounds__(256) k_zgemm(const ZArgs a) {
    constexpr int BK = 32, KS = 256 / (T * T), NL = (BK * T + 255) / 256;
    __shared__ double2 As[2][BK][T + 1], Bs[2][BK][T + 1];
    const int z = blockIdx.z, tid = threadIdx.x;
    const int M = (z == 1 && a.M2 > 0) ? a.M2 : a.M, N = a.N, K = a.K;
    const double2 *__restrict__ A = a.A + z * a.sA, *__restrict__ B = a.B + z * a.sB;
    double2 *C = a.C + z * a.sC;
    int bm = blockIdx.y, bn = blockIdx.x;
    if (SYM) {  // blockIdx.x counts the tiles of the lower triangle row by row
        bm = (int)((sqrtf(8.f * (float)bn + 1.f) - 1.f) * 0.5f);
        while ((bm + 1) * (bm + 2) / 2 <= bn) ++bm;
        while (bm * (bm + 1) / 2 > bn) --bm;
        bn -= bm * (bm + 1) / 2;
    }
    const int m0 = bm * T, n0 = bn * T;
    if (m0 >= M) return;
    const int ks = tid / (T * T), ty = (tid / T) % T, tx = tid % T;
    double2 ra[NL], rb[NL];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int r = 0; r < NL; ++r) {
            const int e = tid + 256 * r;
            if (BK * T < 256 && e >= BK * T) break;
            const int ka = TA ? e / T : e % BK, ia = TA ? e % T : e / BK;  // contiguous along m / along k
            const int kb = e / T, jb = e % T;                               // contiguous along n
            const int gi = m0 + ia, gj = n0 + jb;
            ra[r] = rb[r] = cmk(0.0, 0.0);
            if (gi < M && k0 + ka < K) ra[r] = TA ? A[(long long)(k0 + ka) * a.lda + gi] : A[(long long)gi * a.lda + k0 + ka];
            if (gj < N && k0 + kb < K) rb[r] = B[(long long)(k0 + kb) * a.ldb + gj];
        }
    };
    fetch(0);
    double2 acc = cmk(0.0, 0.0);
    for (int k0 = 0, buf = 0; k0 < K; k0 += BK, buf ^= 1) {
#pragma unroll
        for (int r = 0; r < NL; ++r) {
            const int e = tid + 256 * r;
            if (BK * T < 256 && e >= BK * T) break;
            As[buf][TA ? e / T : e % BK][TA ? e % T : e / BK] = ra[r];
            Bs[buf][e / T][e % T] = rb[r];
        }
        __syncthreads();  // one per chunk: the other buffer was last read before the previous one
        if (k0 + BK < K) fetch(k0 + BK);
#pragma unroll
        for (int kk = 0; kk < BK; kk += KS) {
            const double2 u = As[buf][kk + ks][ty], v = Bs[buf][kk + ks][tx];
            acc.x = fma(u.x, v.x, fma(-u.y, v.y, acc.x));
            acc.y = fma(u.x, v.y, fma(u.y, v.x, acc.y));
        }
    }
    if constexpr (KS > 1) {
        __shared__ double2 part[KS][T * T];
        part[ks][tid % (T * T)] = acc;
        __syncthreads();
        if (ks > 0) return;
#pragma unroll
        for (int q = 1; q < KS; ++q) acc = cadd(acc, part[q][tid]);
    }
    const int gi = m0 + ty, gj = n0 + tx;
    if (gi >= M || gj >= N || (SYM && gj > gi)) return;
    double2 v = cmul(a.alpha, acc);
    if (a.beta.x != 0.0 || a.beta.y != 0.0) v = cadd(v, cmul(a.beta, C[(long long)gi * a.ldc + gj]));
    C[(long long)gi * a.ldc + gj] = v;
    if (SYM && gj < gi) C[(long long)gj * a.ldc + gi] = v;
}

// In-place inverse of an n x n (n <= 64) block by Gauss-Jordan elimination
// with partial (row) pivoting, in shared memory.  Row interchanges during the
// sweep become column interchanges of the result, undone in reverse order.
__global__ void __launch_bounds__(256) k_leaf_inv64(double2 *X, long long sX, int n, long long ld, int *flags) {
    extern __shared__ double2 a[];  // n*n
    X += blockIdx.x * sX;
    __shared__ double2 colk[64];
    __shared__ int piv[64];
    __shared__ int s_p;
    __shared__ double2 s_inv;
    int tid = threadIdx.x, nt = blockDim.x;
    for (int e = tid; e < n * n; e += nt) a[e] = X[(long long)(e / n) * ld + (e % n)];
    __syncthreads();
    for (int k = 0; k < n; ++k) {
        if (tid < 32) {
            double best = -1.0;
            int bi = k;
            for (int i = k + tid; i < n; i += 32) {
                double v = cabs2(a[i * n + k]);
                if (v > best) { best = v; bi = i; }
            }
            for (int off = 16; off > 0; off >>= 1) {
                double ob = __shfl_down_sync(0xffffffffu, best, off);
                int oi = __shfl_down_sync(0xffffffffu, bi, off);
                if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
            }
            if (tid == 0) {
                s_p = bi;
                piv[k] = bi;
                if (!(best > 0.0) || !isfinite(best)) atomicOr(flags, FLAG_SINGULAR);
            }
        }
        __syncthreads();
        int p = s_p;
        if (p != k) {
            for (int j = tid; j < n; j += nt) {
                double2 t = a[k * n + j];
                a[k * n + j] = a[p * n + j];
                a[p * n + j] = t;
            }
            __syncthreads();
        }
        if (tid == 0) s_inv = cinv(a[k * n + k]);
        __syncthreads();
        double2 inv = s_inv;
        for (int j = tid; j < n; j += nt) {
            a[k * n + j] = (j == k) ? inv : cmul(a[k * n + j], inv);
        }
        for (int i = tid; i < n; i += nt) colk[i] = a[i * n + k];
        __syncthreads();
        for (int e = tid; e < n * n; e += nt) {
            int i = e / n, j = e - i * n;
            if (i == k) continue;
            double2 f = colk[i];
            if (j == k) a[e] = cscale(cmul(f, inv), -1.0);
            else a[e] = csub(a[e], cmul(f, a[k * n + j]));
        }
        __syncthreads();
    }
    for (int k = n - 1; k >= 0; --k) {
        int p = piv[k];
        if (p != k) {
            for (int i = tid; i < n; i += nt) {
                double2 t = a[i * n + k];
                a[i * n + k] = a[i * n + p];
                a[i * n + p] = t;
            }
        }
        __syncthreads();
    }
    for (int e = tid; e < n * n; e += nt) X[(long long)(e / n) * ld + (e % n)] = a[e];
}

template <int NB>
__global__ void __launch_bounds__(NB * 4) k_leaf64(double2 *X, long long sX, long long ld, int *flags) {
    LeafIO<double, false> io{nullptr, nullptr, X + blockIdx.x * sX, ld};
    leaf_gj<double, NB, false>(io, flags);
}

// 1 / d for a pivot d with |d|^2 = den: the reciprocal of den by Newton's
// iteration from a float32 start (24 -> 48 -> 96 bits, 4 dependent float64
// operations instead of a division's long chain), a division outside the
// range that float32 covers.
__device__ __forceinline__ double2 pivot_inverse(double2 d, double den) {
    double r;
    if (den > 1e-30 && den < 1e30) {
        r = (double)__frcp_rn((float)den);
        r = fma(r, fma(-den, r, 1.0), r);
        r = fma(r, fma(-den, r, 1.0), r);
    } else {
        r = 1.0 / den;
    }
    return make_double2(d.x * r, -d.y * r);
}

// Inverse of a 32 x 32 block, Gauss-Jordan with partial (row) pivoting, one
// block per CTA.  Lane i of every warp holds row i, warp w the columns 8w .. 8w+7,
// in registers; rows are not swapped (step k takes the unused row with the
// largest max(|re|, |im|) in column k, found on the integer pipe from the high
// words), so at the end inv[step(i)][piv(c)] = x[i][c].
// Bound by the SM's float64 pipe (36 warp instructions per warp and step, 4
// warps: 2304 clocks a step); everything else is kept off that pipe or beside
// it: the warp that owns the next pivot column updates that column first and
// finds the next pivot and its inverse while the others still multiply.
// Measured: 142 -> 64 us per block (shared-memory form with a division, two
// row swaps and five barriers per step before).
__global__ void __launch_bounds__(128) k_leaf64_32(double2 *X, long long sX, long long ld, int *flags) {
    X += blockIdx.x * sX;
    __shared__ double2 cur[2][32][33], s_inv[2];
    __shared__ int s_p[2], piv[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    double2 x[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) x[j] = X[(long long)lane * ld + 8 * w + j];
    bool used = false;
    int mystep = 0;
    auto pivot = [&](double2 v, int k, int b) {
        const unsigned hr = (unsigned)__double2hiint(v.x) & 0x7fffffffu, hi = (unsigned)__double2hiint(v.y) & 0x7fffffffu;
        const unsigned key = used ? 0u : ((max(hr, hi) & ~31u) | (unsigned)(31 - lane));
        const unsigned best = __reduce_max_sync(0xffffffffu, key);
        const int p = 31 - (int)(best & 31u);
        const double2 d = make_double2(__shfl_sync(0xffffffffu, v.x, p), __shfl_sync(0xffffffffu, v.y, p));
        const double den = cabs2(d);
        const double2 inv = pivot_inverse(d, den);
        if (lane == 0) {
            s_p[b] = p;
            piv[k] = p;
            s_inv[b] = inv;
            if ((best & ~31u) == 0u || !(den > 0.0) || !isfinite(den)) atomicOr(flags, FLAG_SINGULAR);
        }
    };
    if (w == 0) pivot(x[0], 0, 0);
#pragma unroll
    for (int j = 0; j < 8; ++j) cur[0][lane][8 * w + j] = x[j];
    __syncthreads();
    for (int kw = 0; kw < 4; ++kw) {
#pragma unroll
        for (int kl = 0; kl < 8; ++kl) {
            const int k = 8 * kw + kl, b = kl & 1;
            const int p = s_p[b];
            const double2 inv = s_inv[b], f = cur[b][lane][k];
            double2 r[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) r[j] = cur[b][p][8 * w + j];
            // other rows: x - (f inv) row_p; the pivot row: 0 - (-inv) row_p
            const bool isp = lane == p;
            const double2 g = isp ? make_double2(-inv.x, -inv.y) : cmul(f, inv);
            if (isp) {
                used = true;
                mystep = k;
#pragma unroll
                for (int j = 0; j < 8; ++j) x[j] = cmk(0.0, 0.0);
            }
            auto update = [&](int j) {
                x[j].x = fma(-g.x, r[j].x, fma(g.y, r[j].y, x[j].x));
                x[j].y = fma(-g.x, r[j].y, fma(-g.y, r[j].x, x[j].y));
            };
            constexpr int LAST = 7;
            const int jn = kl < LAST ? kl + 1 : 0;  // the next pivot column, in warp kw (or kw + 1)
            update(jn);
            if (w == (kl < LAST ? kw : kw + 1) && k + 1 < 32) pivot(x[jn], k + 1, b ^ 1);
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (j != jn) update(j);
            if (w == kw) x[kl] = make_double2(-g.x, -g.y);
            if (k + 1 < 32) {
#pragma unroll
                for (int j = 0; j < 8; ++j) cur[b ^ 1][lane][8 * w + j] = x[j];
            }
            __syncthreads();
        }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) X[(long long)mystep * ld + piv[8 * w + j]] = x[j];
}

// C block <- -V, B block <- -V^T  (the off-diagonal blocks of the inverse).
__global__ void k_neg_offdiag(double2 *Bblk, double2 *Cblk, long long sX, long long ld, const double2 *V, long long sV,
                              int h) {
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    int i = blockIdx.y;
    if (j >= h) return;
    double2 v = V[blockIdx.z * sV + (long long)i * h + j];
    Cblk[blockIdx.z * sX + (long long)i * ld + j] = cscale(v, -1.0);
    Bblk[blockIdx.z * sX + (long long)j * ld + i] = cscale(v, -1.0);
}

// T = a + b for the field rows of a back-substitution step (b null: T = a);
// blockIdx.y = 1: the second row of the pair, at a + da, b + db, T + dT.
__global__ void k_add2(double2 *T, long long dT, const double2 *a, long long da, const double2 *b, long long db, long long n) {
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (blockIdx.y == 1) {
        T += dT;
        a += da;
        b += db;
    }
    T[i] = b ? cadd(a[i], b[i]) : a[i];
}

constexpr int LEAF64 = 32;

}  // namespace

void launch_assemble64(apf_ctx *c, int row, int row2, const double2 *Gp, long long dG, const double2 *Gq, double2 *X,
                       long long dX, cudaStream_t s) {
    GridDev g = make_grid(c);
    dim3 grid((c->nx + 255) / 256, c->nx, row2 >= 0 ? 2 : 1);
    APF_LAUNCH(c, k_assemble64, grid, 256, 0, s, g, row, row2, c->d_eps, c->d_circ, Gp, dG, Gq, X, dX);
}

namespace {

template <int T>
void launch_zgemm(apf_ctx *c, bool ta, bool sym, int batch, const ZArgs &a, cudaStream_t s) {
    const int mt = (std::max(a.M, a.M2) + T - 1) / T, nt = (a.N + T - 1) / T;
    dim3 grid(sym ? mt * (mt + 1) / 2 : nt, sym ? 1 : mt, batch);
    if (sym && ta) APF_LAUNCH(c, (k_zgemm<T, true, true>), grid, 256, 0, s, a);
    else if (sym) APF_LAUNCH(c, (k_zgemm<T, false, true>), grid, 256, 0, s, a);
    else APF_LAUNCH(c, (k_zgemm<T, false, false>), grid, 256, 0, s, a);
}

}  // namespace

// Products the float64 path needs: A B, and with `sym` (M = N, a symmetric
// result) A B or A^T B.  M2: rows of the second entry of the batch (0: M).
void zgemm(apf_ctx *c, bool ta, bool sym, int M, int N, int K, double2 alpha, const double2 *A, long long lda,
           long long sA, const double2 *B, long long ldb, long long sB, double2 beta, double2 *C, long long ldc,
           long long sC, int batch, cudaStream_t s, int M2) {
    if ((M <= 0 && M2 <= 0) || N <= 0 || batch <= 0) return;
    const ZArgs a{M, M2, N, K, alpha, beta, A, B, C, lda, sA, ldb, sB, ldc, sC};
    auto tiles = [&](int t) {
        const long long mt = (std::max(M, M2) + t - 1) / t, nt = (N + t - 1) / t;
        return (sym ? mt * (mt + 1) / 2 : mt * nt) * batch;
    };
    // at least two tiles per SM (304 on 152 SMs): with fewer, the last wave of
    // the larger tile costs more than the smaller tile's extra loads
    if (tiles(16) >= 304) launch_zgemm<16>(c, ta, sym, batch, a, s);
    else if (tiles(8) >= 304) launch_zgemm<8>(c, ta, sym, batch, a, s);
    else launch_zgemm<4>(c, ta, sym, batch, a, s);
}

// X <- X^-1 in place for complex-symmetric X (n a power of two), by the
// 2x2 block Schur recursion
//   [A B; C D]^-1 = [Ai + T^T V, -V^T; -V, Si],  T = C Ai, S = D - T B,
//   Si = S^-1, V = Si T,
// which uses B = C^T and Ai = Ai^T, so four GEMMs per level, two of them with
// a symmetric result.  Pivoting is confined to the diagonal leaf blocks.
// nz (1 or 2) blocks sX apart are inverted by the same launches, with scratch
// (n^2 / 3 elements at each of scr1 and scr2) sS apart.
void invert_sym64(apf_ctx *c, double2 *X, long long sX, int nz, int n, long long ld, double2 *scr1, double2 *scr2,
                  long long sS, cudaStream_t s) {
    if (n <= LEAF64) {
        if (n == 32) APF_LAUNCH(c, k_leaf64_32, nz, 128, 0, s, X, sX, ld, c->d_flags);
        else if (n == 16) APF_LAUNCH(c, k_leaf64<16>, nz, 64, leaf_smem_bytes<16>(16), s, X, sX, ld, c->d_flags);
        else APF_LAUNCH(c, k_leaf_inv64, nz, 256, n * n * (int)sizeof(double2), s, X, sX, n, ld, c->d_flags);
        return;
    }
    int h = n / 2;
    double2 *A = X, *B = X + h, *C = X + (long long)h * ld, *D = X + (long long)h * ld + h;
    double2 *T = scr1, *V = scr2;
    long long hh = (long long)h * h;
    const double2 one = cmk(1, 0), zero = cmk(0, 0), mone = cmk(-1, 0);
    invert_sym64(c, A, sX, nz, h, ld, scr1 + hh, scr2 + hh, sS, s);
    zgemm(c, false, false, h, h, h, one, C, ld, sX, A, ld, sX, zero, T, h, sS, nz, s);
    zgemm(c, false, true, h, h, h, mone, T, h, sS, B, ld, sX, one, D, ld, sX, nz, s);
    invert_sym64(c, D, sX, nz, h, ld, scr1 + hh, scr2 + hh, sS, s);
    zgemm(c, false, false, h, h, h, one, D, ld, sX, T, h, sS, zero, V, h, sS, nz, s);
    zgemm(c, true, true, h, h, h, one, T, h, sS, V, h, sS, one, A, ld, sX, nz, s);
    dim3 grid((h + 255) / 256, h, nz);
    APF_LAUNCH(c, k_neg_offdiag, grid, 256, 0, s, B, C, sX, ld, V, sS, h);
}

// From a to b, which may lie in different allocations (all of them aligned to 256 bytes).
static long long elements_between(const double2 *a, const double2 *b) {
    return ((long long)(uintptr_t)b - (long long)(uintptr_t)a) / (long long)sizeof(double2);
}

// Block elimination of the slab rows from both ends towards the middle row
// m = h / 2: rows 0, 1, .., m - 1 upwards (X_j = K_j - G_{j-1}) and rows h - 1, ..,
// m + 1 downwards (X_j = K_j - G_{j+1}) are independent chains, so rows t and
// h - 1 - t are inverted by the same launches; the middle row takes both
// neighbours, X_m = K_m - G_{m-1} - G_{m+1}.  The same h inversions, but only
// about h / 2 dependent steps of them, each with twice the parallel work.  The
// second chain's scratch lies in the middle row's block, which is not assembled
// before both chains are done.
void eliminate64(apf_ctx *c, cudaStream_t s) {
    const long long n = c->nx, nn = n * n;
    const int h = c->h, m = h / 2, top = h - 1 - m;  // top <= m
    double2 *G = c->d_G, *scr1 = c->d_scr, *scr2 = scr1 + nn / 2;
    const long long dS = elements_between(scr1, G + m * nn);
    for (int t = 0; t < m; ++t) {
        const int u = h - 1 - t, nz = t < top ? 2 : 1;
        const long long d = (u - t) * nn;  // from row t's block to row u's
        launch_assemble64(c, t, nz == 2 ? u : -1, t > 0 ? G + (t - 1) * nn : nullptr, d + 2 * nn, nullptr, G + t * nn,
                          d, s);
        invert_sym64(c, G + t * nn, d, nz, c->nx, n, scr1, scr2, dS, s);
    }
    launch_assemble64(c, m, -1, m > 0 ? G + (m - 1) * nn : nullptr, 0, top > 0 ? G + (m + 1) * nn : nullptr, G + m * nn,
                      0, s);
    invert_sym64(c, G + m * nn, 0, 1, c->nx, n, scr1, scr2, 0, s);
}

// Slab fields from the inverses of eliminate64: the right-hand sides (inputs
// on row 0, outputs on row h - 1) are carried to the middle row, solved there,
// and substituted back outwards.
void fields64(apf_ctx *c, cudaStream_t s) {
    const int nf = c->cf, na = c->ca, ncol = nf + na, h = c->h, m = h / 2, top = h - 1 - m;
    const long long nx = c->nx, L = (long long)ncol * nx, nn = nx * nx, of = (long long)nf * nx;
    double2 *E = c->d_Ew, *T = c->d_T;
    const long long dT = elements_between(T, c->d_fft);  // the second row of a pair: in the transforms' buffer, not in use yet
    const double2 *G = c->d_G;
    const double2 one = cmk(1, 0), zero = cmk(0, 0);
    // inwards: Y_t = G_{t-1} Y_{t-1} (inputs) and Y_u = G_{u+1} Y_{u+1} (outputs), u = h - 1 - t
    for (int t = 1; t <= m; ++t) {
        const int u = h - 1 - t;
        const long long d = (u - t) * L + of, dg = (u - t + 2) * nn;
        if (t <= top && na > 0)
            zgemm(c, false, false, nf, c->nx, c->nx, one, E + (t - 1) * L, nx, d + 2 * L, G + (t - 1) * nn, nx, dg,
                  zero, E + t * L, nx, d, 2, s, na);
        else
            zgemm(c, false, false, nf, c->nx, c->nx, one, E + (t - 1) * L, nx, 0, G + (t - 1) * nn, nx, 0, zero,
                  E + t * L, nx, 0, 1, s, 0);
    }
    // the middle row, then outwards E_t = G_t (Y_t + E_{t+1}), E_u = G_u (Y_u + E_{u-1})
    launch_add(c, T, 0, E + m * L, 0, nullptr, 0, L, 1, s);
    zgemm(c, false, false, ncol, c->nx, c->nx, one, T, nx, 0, G + m * nn, nx, 0, zero, E + m * L, nx, 0, 1, s);
    for (int t = m - 1; t >= 0; --t) {
        const int u = h - 1 - t, nz = t < top ? 2 : 1;
        launch_add(c, T, dT, E + t * L, (u - t) * L, E + (t + 1) * L, (u - t - 2) * L, L, nz, s);
        zgemm(c, false, false, ncol, c->nx, c->nx, one, T, nx, dT, G + t * nn, nx, (u - t) * nn, zero, E + t * L, nx,
              (u - t) * L, nz, s);
    }
}

void launch_add(apf_ctx *c, double2 *T, long long dT, const double2 *a, long long da, const double2 *b, long long db,
                long long n, int nz, cudaStream_t s) {
    APF_LAUNCH(c, k_add2, dim3((unsigned)((n + 255) / 256), nz), 256, 0, s, T, dT, a, da, b, db, n);
}

void launch_zero(apf_ctx *c, void *dst, long long bytes, cudaStream_t s) {
    (void)c;
    cudaMemsetAsync(dst, 0, (size_t)bytes, s);
}

void slab64_init_attrs() {
    cudaFuncSetAttribute(k_leaf_inv64, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 64 * (int)sizeof(double2));
}
