// Spectral-convolution surrogate of the efficiencies (training and inference
// kernels).  Not part of the paper's method: it screens line-search
// candidates before the exact solve judges them.
//
// Network (x is the periodic axis, n positions; the slab rows are channels):
//   h0 = W0 eps + b0                                   (CI -> C, per position)
//   for l = 1..L:
//     X = DFT_M(h_{l-1})          (first M Fourier modes, e^{-2 pi i m x / n})
//     Y[o, m] = sum_i W_l[i, o, m] X[i, m]             (complex, per mode)
//     z_l = synth_M(Y) + P_l h_{l-1} + c_l              (synth: real inverse DFT
//                                                        of the M modes, zero-padded)
//     h_l = gelu(z_l)  (l < L),   h_L = z_L
//   out = Wh mean_x(h_L) + bh                          (C -> NO)
// Loss: mean squared error.  Weights are used in bf16 (a bf16 copy of the
// fp32 master parameters, refreshed after every Adam step); activations and
// every sum are fp32.
#include "apf_internal.h"
#include "../../include/apf_surrogate.h"

#include <math.h>

#include <algorithm>
#include <vector>

struct apf_sno {
    int device = 0;
    int n = 0, ci = 0, c = 0, m = 0, layers = 0, no = 0, bmax = 0;
    long long nparams = 0;
    // parameter offsets (floats)
    long long oW0, ob0, oWr, oWi, oP, oc, oWh, obh;
    float *p = nullptr, *g = nullptr, *mom1 = nullptr, *mom2 = nullptr;
    __nv_bfloat16 *pb = nullptr;
    float2 *tw = nullptr;          // M x n: (cos, sin)(2 pi m x / n)
    float *h = nullptr, *z = nullptr;       // (L+1) x B x C x n, L x B x C x n
    float2 *X = nullptr, *Y = nullptr;      // L x B x C x M
    float *dh = nullptr, *dz = nullptr;     // B x C x n each
    float2 *dY = nullptr, *dX = nullptr;    // B x C x M
    float *pooled = nullptr, *out = nullptr, *dout = nullptr, *dpooled = nullptr, *loss = nullptr;
    long long step = 0;
    std::vector<void *> allocs;
    std::string err;
};

namespace {

__device__ __forceinline__ float bf(const __nv_bfloat16 *p, long long i) { return __bfloat162float(p[i]); }

__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_d(float x) {
    const float phi = 0.39894228040143268f * expf(-0.5f * x * x);
    return 0.5f * (1.f + erff(x * 0.70710678118654752f)) + x * phi;
}

__global__ void k_tw(float2 *tw, int n, int M) {
    int x = blockIdx.x * blockDim.x + threadIdx.x;
    int m = blockIdx.y;
    if (x >= n) return;
    long long t = ((long long)m * x) % n;
    float s, c;
    sincospif(2.f * (float)t / (float)n, &s, &c);
    tw[(long long)m * n + x] = make_float2(c, s);
}

// h0[b][o][x] = b0[o] + sum_i W0[o][i] eps[b][i][x].  Block: 64 positions of one
// sample, staged in shared memory; each of the 4 thread rows takes every fourth
// group of 8 outputs.
__global__ void __launch_bounds__(256) k_lift(const float *eps, const __nv_bfloat16 *pb, long long oW0, long long ob0,
                                              float *h0, int CI, int C, int n) {
    __shared__ __align__(16) float es[64][64], ws[64][72];  // [i][x], [i][o]
    const int b = blockIdx.y, x0 = blockIdx.x * 64, tx = threadIdx.x & 63, ty = threadIdx.x >> 6;
    const int Cp = (C + 7) & ~7;
    for (int i = ty; i < CI; i += 4) es[i][tx] = eps[((long long)b * CI + i) * n + x0 + tx];
    for (int e = threadIdx.x; e < CI * Cp; e += 256) {
        const int i = e / Cp, o = e - i * Cp;
        ws[i][o] = o < C ? bf(pb, oW0 + (long long)o * CI + i) : 0.f;
    }
    __syncthreads();
    for (int o0 = 8 * ty; o0 < Cp; o0 += 32) {
        float acc[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) acc[u] = o0 + u < C ? bf(pb, ob0 + o0 + u) : 0.f;
        for (int i = 0; i < CI; ++i) {
            const float e = es[i][tx];
            const float4 w0 = *reinterpret_cast<const float4 *>(&ws[i][o0]), w1 = *reinterpret_cast<const float4 *>(&ws[i][o0 + 4]);
            acc[0] = fmaf(w0.x, e, acc[0]); acc[1] = fmaf(w0.y, e, acc[1]);
            acc[2] = fmaf(w0.z, e, acc[2]); acc[3] = fmaf(w0.w, e, acc[3]);
            acc[4] = fmaf(w1.x, e, acc[4]); acc[5] = fmaf(w1.y, e, acc[5]);
            acc[6] = fmaf(w1.z, e, acc[6]); acc[7] = fmaf(w1.w, e, acc[7]);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (o0 + u < C) h0[((long long)b * C + o0 + u) * n + x0 + tx] = acc[u];
    }
}

// The transforms use the symmetries of cos and sin: with theta = 2 pi m x / n, the
// four positions x, n/2 - x, n/2 + x, n - x (0 <= x < n/4) share cos theta and
// sin theta up to signs that depend on the parity of m only.  So the analysis
// first folds a row into four sums per x (cos / sin part, even / odd m), and the
// synthesis makes the four positions' values from four sums (even / odd m, cos /
// sin part): a quarter of the multiply-adds of the plain transforms.  x = 0 has
// only the positions 0 and n/2; x = n/4 (positions n/4, 3n/4), where cos and sin
// are 0 or +-1, is added separately.

// out[row][m] = scale_m * sum_x in[row][x] (cos, -sin)(theta_mx), rows = B*C.
// scale_m = 1 (analysis) or the synthesis weights (1/n, 2/n) for the backward.
// Block: 16 rows x 64 modes, x in chunks of 32; thread: 4 rows x 4 modes of every
// fourth x, the four partial sums added in a fixed order.  Bound by the float32
// pipe (32 multiply-adds per 6 shared-memory loads), and for few rows by latency: the
// next chunk is loaded during this one's products.  64 samples of 48 channels,
// 1024 positions, 64 modes 212 -> 20 us, 1 sample 15 -> 10 us (one thread per mode
// and quarter of x, two loads per multiply-add pair, before).
__global__ void __launch_bounds__(256) k_dft(const float *__restrict__ in, float2 *out, const float2 *__restrict__ tw,
                                             int rows, int n, int M, int synth_weights) {
    constexpr int XC = 32, RP = 17;
    __shared__ __align__(16) float4 sm[3 * XC * RP];
    float4 *fold = sm, *ta = sm + XC * RP, *tb = ta + XC * RP;  // [x][row]; [x][mode group]: modes 4g, 4g+1 and 4g+2, 4g+3
    const int tid = threadIdx.x, mg = tid & 15, ks = (tid >> 4) & 3, rg = tid >> 6;
    const int r0 = blockIdx.x * 16, m0 = blockIdx.y * 64, q = n >> 2;
    float re[4][4] = {}, im[4][4] = {};
    float4 pf[2];  // the next chunk's loads, in flight during this one's products
    float2 pw[8];
    auto fetch = [&](int x0) {
        const int x = x0 + (tid & (XC - 1));
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int r = tid / XC + 8 * k;
            pf[k] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (x < q && r0 + r < rows) {
                const float *p = in + (long long)(r0 + r) * n;
                pf[k] = make_float4(p[x], p[n / 2 - x], x ? p[n / 2 + x] : 0.f, x ? p[n - x] : 0.f);
            }
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int m = m0 + tid / XC + 8 * k;
            pw[k] = x < q && m < M ? tw[(long long)m * n + x] : make_float2(0.f, 0.f);
        }
    };
    fetch(0);
    for (int x0 = 0; x0 < q; x0 += XC) {
        __syncthreads();
        const int xx = tid & (XC - 1);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const float ad = pf[k].x + pf[k].w, bc = pf[k].y + pf[k].z, am = pf[k].x - pf[k].w, bm = pf[k].y - pf[k].z;
            fold[xx * RP + tid / XC + 8 * k] = make_float4(ad + bc, ad - bc, am - bm, am + bm);  // cos even, cos odd, sin even, sin odd
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int m = tid / XC + 8 * k;
            reinterpret_cast<float2 *>((m & 2 ? tb : ta) + xx * RP + (m >> 2))[m & 1] = pw[k];
        }
        if (x0 + XC < q) fetch(x0 + XC);
        __syncthreads();
#pragma unroll
        for (int xx = 0; xx < XC; xx += 4) {
            const float4 wa = ta[(xx + ks) * RP + mg], wb = tb[(xx + ks) * RP + mg];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float4 f = fold[(xx + ks) * RP + 4 * rg + r];
                re[r][0] = fmaf(f.x, wa.x, re[r][0]); im[r][0] = fmaf(-f.z, wa.y, im[r][0]);
                re[r][1] = fmaf(f.y, wa.z, re[r][1]); im[r][1] = fmaf(-f.w, wa.w, im[r][1]);
                re[r][2] = fmaf(f.x, wb.x, re[r][2]); im[r][2] = fmaf(-f.z, wb.y, im[r][2]);
                re[r][3] = fmaf(f.y, wb.z, re[r][3]); im[r][3] = fmaf(-f.w, wb.w, im[r][3]);
            }
        }
    }
    // add the four x slices: lane bit 4 by shuffle, the warp pair through shared memory
    __syncthreads();
    float *red = reinterpret_cast<float *>(sm);
    const int slot = rg * 16 + mg;
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            re[r][j] += __shfl_xor_sync(0xffffffffu, re[r][j], 16);
            im[r][j] += __shfl_xor_sync(0xffffffffu, im[r][j], 16);
            if (ks == 2) {
                red[(8 * r + 2 * j) * 64 + slot] = re[r][j];
                red[(8 * r + 2 * j + 1) * 64 + slot] = im[r][j];
            }
        }
    __syncthreads();
    if (ks != 0) return;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int row = r0 + 4 * rg + r;
        if (row >= rows) break;
        const float a = in[(long long)row * n + q], d = in[(long long)row * n + 3 * q];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int m = m0 + 4 * mg + j;
            if (m >= M) break;
            float vr = re[r][j] + red[(8 * r + 2 * j) * 64 + slot], vi = im[r][j] + red[(8 * r + 2 * j + 1) * 64 + slot];
            const float sg = (m >> 1) & 1 ? -1.f : 1.f;
            if (m & 1) vi -= sg * (a - d);
            else vr += sg * (a + d);
            const float s = !synth_weights ? 1.f : (m == 0 ? 1.f : 2.f) / (float)n;
            out[(long long)row * M + m] = make_float2(vr * s, vi * s);
        }
    }
}

// Y[b][o][m] = sum_i W[i][o][m] X[b][i][m], or its adjoint (BWD) dX[b][i][m] =
// sum_o conj(W[i][o][m]) dY[b][o][m].  Thread: one mode, two outputs, four samples,
// so that a weight serves four samples and a spectrum value two outputs; bound by
// the latency of L2, so four i are loaded before the first use (128 samples of 48
// channels, 64 modes: 15.5 us; 27 us as the compiler ordered the loads).
template <bool BWD>
__global__ void __launch_bounds__(256) k_mix(const float2 *__restrict__ X, const __nv_bfloat16 *__restrict__ pb, long long oWr,
                                             long long oWi, float2 *Y, int B, int C, int M) {
    constexpr int OT = 2;
    const int idx = blockIdx.x * 256 + threadIdx.x, groups = (C + OT - 1) / OT;
    if (idx >= groups * M) return;
    const int m = idx % M, o0 = OT * (idx / M), b0 = 4 * blockIdx.y;
    const int nb = min(4, B - b0);
    const long long sb = (long long)C * M;
    const float2 *x = X + (long long)b0 * sb + m;
    const unsigned short *wrp[OT], *wip[OT];
#pragma unroll
    for (int j = 0; j < OT; ++j) {
        const int o = min(o0 + j, C - 1);
        const long long w = (BWD ? (long long)o * C : (long long)o) * M + m;
        wrp[j] = reinterpret_cast<const unsigned short *>(pb) + oWr + w;
        wip[j] = reinterpret_cast<const unsigned short *>(pb) + oWi + w;
    }
    const long long ws = BWD ? M : (long long)C * M;
    float2 y[OT][4] = {};
    constexpr int IC = 4;  // loads before their first use
    for (int i0 = 0; i0 < C; i0 += IC) {
        float2 v[IC][4];
        unsigned r[IC][OT], q[IC][OT];
#pragma unroll
        for (int k = 0; k < IC; ++k) {
            const long long i = min(i0 + k, C - 1);
#pragma unroll
            for (int u = 0; u < 4; ++u) v[k][u] = x[(u < nb ? u : 0) * sb + i * M];
#pragma unroll
            for (int j = 0; j < OT; ++j) {
                r[k][j] = wrp[j][i * ws];
                q[k][j] = wip[j][i * ws];
            }
        }
#pragma unroll
        for (int k = 0; k < IC; ++k)
#pragma unroll
            for (int j = 0; j < OT; ++j) {
                const float wr = i0 + k < C ? __uint_as_float(r[k][j] << 16) : 0.f, wi = i0 + k < C ? __uint_as_float(q[k][j] << 16) : 0.f;
                const float wim = BWD ? -wi : wi;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    y[j][u].x = fmaf(wr, v[k][u].x, fmaf(-wim, v[k][u].y, y[j][u].x));
                    y[j][u].y = fmaf(wr, v[k][u].y, fmaf(wim, v[k][u].x, y[j][u].y));
                }
            }
    }
#pragma unroll
    for (int j = 0; j < OT; ++j)
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (u < nb && o0 + j < C) Y[(long long)(b0 + u) * sb + (long long)(o0 + j) * M + m] = y[j][u];
}

// The same, and k_synth below, for small calls, one output per thread: as many
// threads as there are, each with a short chain of loads (SMALL_BATCH at a time
// before their first use; the compiler's own unrolling waited for each).
constexpr int SMALL_BATCH = 8;
__host__ __device__ constexpr int small_pad(int k) { return (k + SMALL_BATCH - 1) / SMALL_BATCH * SMALL_BATCH; }
template <bool BWD>
__global__ void __launch_bounds__(128) k_mix_small(const float2 *__restrict__ X, const __nv_bfloat16 *__restrict__ pb, long long oWr,
                                                   long long oWi, float2 *__restrict__ Y, int B, int C, int M) {
    const int idx = blockIdx.x * 128 + threadIdx.x;
    if (idx >= B * C * M) return;
    const int m = idx % M, o = (idx / M) % C, b = idx / (M * C), ws = BWD ? M : C * M;
    const float2 *x = X + (long long)b * C * M + m;
    const unsigned short *w = reinterpret_cast<const unsigned short *>(pb) + (BWD ? (long long)o * C : (long long)o) * M + m;
    const unsigned short *wr = w + oWr, *wi = w + oWi;
    float yr = 0.f, yi = 0.f;
    for (int i0 = 0; i0 < C; i0 += SMALL_BATCH) {
        float2 v[SMALL_BATCH];
        unsigned r[SMALL_BATCH], q[SMALL_BATCH];
#pragma unroll
        for (int k = 0; k < SMALL_BATCH; ++k) {
            const int i = min(i0 + k, C - 1);
            v[k] = x[i * M];
            r[k] = wr[i * ws];
            q[k] = wi[i * ws];
        }
#pragma unroll
        for (int k = 0; k < SMALL_BATCH; ++k) {
            const float a = i0 + k < C ? __uint_as_float(r[k] << 16) : 0.f, d = i0 + k < C ? __uint_as_float(q[k] << 16) : 0.f;
            yr = fmaf(a, v[k].x, fmaf(BWD ? d : -d, v[k].y, yr));
            yi = fmaf(a, v[k].y, fmaf(BWD ? -d : d, v[k].x, yi));
        }
    }
    Y[idx] = make_float2(yr, yi);
}

// Block: 128 positions (blockIdx.x) of one channel of a sample (blockIdx.y).  Every sum
// is taken in k_synth's order (modes folded, n/4 and 3n/4 by a warp), so that a
// sample's result does not depend on how many others are in the call (0.3 to 0.5 us
// of a launch's 3.5 to 7 us: 1 sample of 16 channels, 128 positions; of 48 and 1024).
template <bool BWD>
__global__ void __launch_bounds__(128) k_synth_small(const float2 *__restrict__ Y, const float *__restrict__ h, const __nv_bfloat16 *__restrict__ pb,
                                                     long long oP, long long oc, const float2 *__restrict__ tw, float *z, float *hn, int C,
                                                     int n, int M, int act) {
    extern __shared__ __align__(16) unsigned char ss_smem[];
    const int Mp = small_pad(M), Cp = small_pad(C);  // with zeros up to whole batches
    float2 *ys = reinterpret_cast<float2 *>(ss_smem);  // [m]: w Y
    float *ps = reinterpret_cast<float *>(ys + Mp);     // [i]
    const int b = blockIdx.y / C, o = blockIdx.y - b * C, x = blockIdx.x * 128 + threadIdx.x, q = n >> 2;
    // x is one of f, n/2 - f, n/2 + f, n - f
    const int quarter = (x >= q) + (x >= n / 2) + (x >= 3 * q), f = quarter == 0 ? x : quarter == 1 ? n / 2 - x : quarter == 2 ? x - n / 2 : n - x;
    const float *hb = h + (long long)b * C * n;
    // n/4 or 3n/4 if it is one of this warp's positions; its first loads go out with the others
    const int lane = threadIdx.x & 31, x0 = x - lane, p = (q - x0) >> 5 == 0 ? q : (3 * q - x0) >> 5 == 0 ? 3 * q : -1;
    const float2 yp = p >= 0 && lane < M ? Y[(long long)blockIdx.y * M + lane] : make_float2(0.f, 0.f);
    const float hp = p >= 0 && lane < C ? hb[lane * n + p] : 0.f;
    auto weight = [&](int m) { return m >= M ? 0.f : BWD ? 1.f : (m == 0 ? 1.f : 2.f) / (float)n; };
    float2 w[SMALL_BATCH];  // one batch ahead
    float v[SMALL_BATCH];
    if (x < n) {
#pragma unroll
        for (int k = 0; k < SMALL_BATCH; ++k) {
            w[k] = tw[min(k, M - 1) * n + f];
            v[k] = hb[min(k, C - 1) * n + x];
        }
    }
    for (int m = threadIdx.x; m < Mp; m += 128) {
        const float2 y = Y[(long long)blockIdx.y * M + min(m, M - 1)];
        const float s = weight(m);
        ys[m] = make_float2(s * y.x, s * y.y);
    }
    for (int i = threadIdx.x; i < Cp; i += 128) ps[i] = i < C ? bf(pb, oP + (BWD ? (long long)i * C + o : (long long)o * C + i)) : 0.f;
    __syncthreads();
    if (x >= n) return;
    const long long at = (long long)blockIdx.y * n + x;
    const float zv = BWD && z ? z[at] : 0.f;
    float a[4] = {};  // even cos, odd cos, even sin, odd sin
    for (int m0 = 0; m0 < M; m0 += SMALL_BATCH) {
        float2 c[SMALL_BATCH];
#pragma unroll
        for (int k = 0; k < SMALL_BATCH; ++k) {
            c[k] = w[k];
            if (m0 + SMALL_BATCH < M) w[k] = tw[min(m0 + SMALL_BATCH + k, M - 1) * n + f];
        }
#pragma unroll
        for (int k = 0; k < SMALL_BATCH; ++k) {
            a[k & 1] = fmaf(ys[m0 + k].x, c[k].x, a[k & 1]);
            a[2 + (k & 1)] = fmaf(ys[m0 + k].y, c[k].y, a[2 + (k & 1)]);
        }
    }
    const float cp = a[0] + a[1], cm = a[0] - a[1], sp = a[2] + a[3], sd = a[2] - a[3];
    float acc = quarter == 0 ? cp - sp : quarter == 1 ? cm + sd : quarter == 2 ? cm - sd : cp + sp;
    for (int i0 = 0; i0 < C; i0 += SMALL_BATCH) {
        float c[SMALL_BATCH];
#pragma unroll
        for (int k = 0; k < SMALL_BATCH; ++k) {
            c[k] = v[k];
            if (i0 + SMALL_BATCH < C) v[k] = hb[min(i0 + SMALL_BATCH + k, C - 1) * n + x];
        }
#pragma unroll
        for (int k = 0; k < SMALL_BATCH; ++k) acc = fmaf(ps[i0 + k], c[k], acc);
    }
    if (p >= 0) {
        float even = 0.f, odd = 0.f, part = 0.f;
        for (int m = lane; m < M; m += 32) {
            const float s = (m >> 1) & 1 ? -weight(m) : weight(m);
            const float2 y = m == lane ? yp : Y[(long long)blockIdx.y * M + m];
            if (m & 1) odd = fmaf(s, y.y, odd);
            else even = fmaf(s, y.x, even);
        }
        for (int i = lane; i < C; i += 32) part = fmaf(ps[i], i == lane ? hp : hb[i * n + p], part);
        float t = p == q ? even - odd + part : even + odd + part;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
        if (x == p) acc = t;
    }
    if (BWD) {
        hn[at] = z ? acc * gelu_d(zv) : acc;
    } else {
        acc += bf(pb, oc + o);
        z[at] = acc;
        hn[at] = act ? gelu(acc) : acc;
    }
}

// v[b][o][x] = sum_m w_m Re(Y_om e^{i theta}) + sum_i P[o][i] h[b][i][x] (+ c[o]).
// Forward: w = (1/n, 2/n, ..), z = v + c, hn = act(z).  Backward (BWD): w = 1, P
// transposed, Y the mixing's gradient, h = dz of this layer; hn = v times the
// derivative of the previous layer's activation at z (z null: none).
// Block: one sample, 32 XT values of x below n/4 (so 128 XT positions), all
// channels, 8 per warp; thread: 8 channels x XT x x 4 positions.  Bound by the
// float32 pipe: 32 XT multiply-adds per 8 + XT (transform) or 2 + XT (map)
// shared-memory loads.  64 samples of 48 channels, 1024 positions, 64 modes: 104 ->
// 36 us inside a forward pass (the activation included).
constexpr int SY_MC = 16, SY_IC = 16;  // mode pairs and channels staged at a time
template <bool BWD, int XT>
__global__ void __launch_bounds__(256, 2) k_synth(const float2 *__restrict__ Y, const float *__restrict__ h, const __nv_bfloat16 *__restrict__ pb,
                                               long long oP, long long oc, const float2 *__restrict__ tw, float *z, float *hn, int C, int n,
                                               int M, int act) {
    constexpr int XW = 32 * XT;
    extern __shared__ __align__(16) unsigned char sy_smem[];
    const int Cp = (C + 7) & ~7;
    float4 *ys = reinterpret_cast<float4 *>(sy_smem);  // [mode pair][o]: w Y of modes 2q, 2q + 1
    float4 *ts = ys + SY_MC * Cp;                       // [mode pair][x]
    float4 *hs = ts + SY_MC * XW;                       // [i][x]: the four positions
    float *ps = reinterpret_cast<float *>(hs + SY_IC * XW);  // [i][o]
    const int b = blockIdx.y, x0 = blockIdx.x * XW, q = n >> 2;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, o0 = 8 * (tid >> 5);
    for (int e = tid; e < C * Cp; e += nt) {
        const int i = e / Cp, o = e - i * Cp;
        ps[e] = o < C ? bf(pb, oP + (BWD ? (long long)i * C + o : (long long)o * C + i)) : 0.f;
    }
    auto weight = [&](int m) { return m >= M ? 0.f : BWD ? 1.f : (m == 0 ? 1.f : 2.f) / (float)n; };
    float acc[XT][8][4];  // even cos, odd cos, even sin, odd sin
#pragma unroll
    for (int u = 0; u < XT; ++u)
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[u][j][k] = 0.f;
    const int pairs = (M + 1) / 2;
    for (int p0 = 0; p0 < pairs; p0 += SY_MC) {
        const int np = min(SY_MC, pairs - p0);
        __syncthreads();
#pragma unroll 4
        for (int e = tid; e < SY_MC * Cp; e += nt) {
            const int o = e / SY_MC, pr = e % SY_MC, m = 2 * (p0 + pr);
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (o < C && pr < np) {
                const float2 *y = Y + ((long long)b * C + o) * M + m;
                const float w0 = weight(m), w1 = weight(m + 1);
                const float2 a = y[0], d = m + 1 < M ? y[1] : make_float2(0.f, 0.f);
                v = make_float4(w0 * a.x, w0 * a.y, w1 * d.x, w1 * d.y);
            }
            ys[pr * Cp + o] = v;
        }
#pragma unroll 4
        for (int e = tid; e < np * XW; e += nt) {
            const int pr = e / XW, xx = e - pr * XW, x = x0 + xx, m = 2 * (p0 + pr);
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (x < q) {
                const float2 a = tw[(long long)m * n + x], d = m + 1 < M ? tw[(long long)(m + 1) * n + x] : make_float2(0.f, 0.f);
                v = make_float4(a.x, a.y, d.x, d.y);
            }
            ts[e] = v;
        }
        __syncthreads();
        if (o0 < C) {
            for (int pr = 0; pr < np; ++pr) {
                float4 t[XT];
#pragma unroll
                for (int u = 0; u < XT; ++u) t[u] = ts[pr * XW + 32 * u + lane];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float4 y = ys[pr * Cp + o0 + j];
#pragma unroll
                    for (int u = 0; u < XT; ++u) {
                        acc[u][j][0] = fmaf(y.x, t[u].x, acc[u][j][0]);
                        acc[u][j][1] = fmaf(y.z, t[u].z, acc[u][j][1]);
                        acc[u][j][2] = fmaf(y.y, t[u].y, acc[u][j][2]);
                        acc[u][j][3] = fmaf(y.w, t[u].w, acc[u][j][3]);
                    }
                }
            }
        }
    }
    // positions x, n/2 - x, n/2 + x, n - x
#pragma unroll
    for (int u = 0; u < XT; ++u)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            float *a = acc[u][j];
            const float cp = a[0] + a[1], cm = a[0] - a[1], sp = a[2] + a[3], sd = a[2] - a[3];
            a[0] = cp - sp;
            a[1] = cm + sd;
            a[2] = cm - sd;
            a[3] = cp + sp;
        }
    for (int i0 = 0; i0 < C; i0 += SY_IC) {
        const int ni = min(SY_IC, C - i0);
        __syncthreads();
#pragma unroll 4
        for (int e = tid; e < ni * XW; e += nt) {
            const int i = e / XW, xx = e - i * XW, x = x0 + xx;
            const float *p = h + ((long long)b * C + i0 + i) * n;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (x < q) v = make_float4(p[x], p[n / 2 - x], x ? p[n / 2 + x] : 0.f, x ? p[n - x] : 0.f);
            hs[e] = v;
        }
        __syncthreads();
        if (o0 >= C) continue;
        for (int i = 0; i < ni; ++i) {
            const float *pr = ps + (i0 + i) * Cp + o0;
            const float4 p0 = *reinterpret_cast<const float4 *>(pr), p1 = *reinterpret_cast<const float4 *>(pr + 4);
            const float pw[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
#pragma unroll
            for (int u = 0; u < XT; ++u) {
                const float4 v = hs[i * XW + 32 * u + lane];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    acc[u][j][0] = fmaf(pw[j], v.x, acc[u][j][0]);
                    acc[u][j][1] = fmaf(pw[j], v.y, acc[u][j][1]);
                    acc[u][j][2] = fmaf(pw[j], v.z, acc[u][j][2]);
                    acc[u][j][3] = fmaf(pw[j], v.w, acc[u][j][3]);
                }
            }
        }
    }
    if (o0 >= C) return;
    const long long base = ((long long)b * C + o0) * n;
    const float *zr = BWD && z ? z + base : nullptr;
    float *zw = BWD ? nullptr : z + base, *hw = hn + base;
    auto store = [&](int at, float v, float bias, float zv) {
        if (BWD) {
            hw[at] = zr ? v * gelu_d(zv) : v;
        } else {
            v += bias;
            zw[at] = v;
            hw[at] = act ? gelu(v) : v;
        }
    };
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        if (o0 + j >= C) break;
        const float bias = BWD ? 0.f : bf(pb, oc + o0 + j);
        int at[XT][4];
        float zv[XT][4];
#pragma unroll
        for (int u = 0; u < XT; ++u) {
            const int x = x0 + 32 * u + lane;
            const int pos[4] = {x, n / 2 - x, n / 2 + x, n - x};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                at[u][k] = x < q && (x > 0 || k < 2) ? j * n + pos[k] : -1;
                zv[u][k] = BWD && zr && at[u][k] >= 0 ? zr[at[u][k]] : 0.f;  // all loads before the first store
            }
        }
#pragma unroll
        for (int u = 0; u < XT; ++u)
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (at[u][k] >= 0) store(at[u][k], acc[u][j][k], bias, zv[u][k]);
    }
    if (blockIdx.x != 0) return;
    // positions n/4 and 3n/4 of the warp's 8 channels: lanes share modes and channels
    float even[8] = {}, odd[8] = {};
    for (int m = lane; m < M; m += 32) {
        const float w = (m >> 1) & 1 ? -weight(m) : weight(m);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float2 y = Y[((long long)b * C + min(o0 + j, C - 1)) * M + m];
            if (m & 1) odd[j] = fmaf(w, y.y, odd[j]);
            else even[j] = fmaf(w, y.x, even[j]);
        }
    }
    float p1[8] = {}, p3[8] = {};
    for (int i = lane; i < C; i += 32) {
        const float *hp = h + ((long long)b * C + i) * n;
        const float h1 = hp[q], h3 = hp[3 * q];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            p1[j] = fmaf(ps[i * Cp + o0 + j], h1, p1[j]);
            p3[j] = fmaf(ps[i * Cp + o0 + j], h3, p3[j]);
        }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        float v1 = even[j] - odd[j] + p1[j], v3 = even[j] + odd[j] + p3[j];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            v1 += __shfl_xor_sync(0xffffffffu, v1, off);
            v3 += __shfl_xor_sync(0xffffffffu, v3, off);
        }
        if (o0 + j < C && lane < 2) {
            const int at = j * n + (lane ? 3 * q : q);
            store(at, lane ? v3 : v1, BWD ? 0.f : bf(pb, oc + o0 + j), zr ? zr[at] : 0.f);
        }
    }
}

// pooled[b][c] = mean_x h[b][c][x]
__global__ void k_pool(const float *h, float *pooled, int n) {
    __shared__ float red[256];
    const long long r = blockIdx.x;
    float acc = 0.f;
    for (int x = threadIdx.x; x < n; x += blockDim.x) acc += h[r * n + x];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if ((int)threadIdx.x < off) red[threadIdx.x] += red[threadIdx.x + off];
        __syncthreads();
    }
    if (threadIdx.x == 0) pooled[r] = red[0] / (float)n;
}

__global__ void k_head(const float *pooled, const __nv_bfloat16 *pb, long long oWh, long long obh, float *out, int B,
                       int C, int NO) {
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= B * NO) return;
    int k = idx % NO, b = idx / NO;
    float acc = bf(pb, obh + k);
    for (int c = 0; c < C; ++c) acc += bf(pb, oWh + (long long)k * C + c) * pooled[(long long)b * C + c];
    out[idx] = acc;
}

// Loss, d_out, head gradients and d_pooled (one block).
__global__ void k_head_bwd(const float *out, const float *tgt, const float *pooled, const __nv_bfloat16 *pb,
                           long long oWh, float *g, long long gWh, long long gbh, float *dout, float *dpooled,
                           float *loss, int B, int C, int NO) {
    __shared__ float red[256];
    float acc = 0.f;
    for (int i = threadIdx.x; i < B * NO; i += blockDim.x) {
        float d = out[i] - tgt[i];
        acc += d * d;
        dout[i] = 2.f * d / (float)(B * NO);
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if ((int)threadIdx.x < off) red[threadIdx.x] += red[threadIdx.x + off];
        __syncthreads();
    }
    if (threadIdx.x == 0) loss[0] = red[0] / (float)(B * NO);
    for (int e = threadIdx.x; e < NO * C; e += blockDim.x) {
        int k = e / C, c = e % C;
        float s = 0.f;
        for (int b = 0; b < B; ++b) s += dout[b * NO + k] * pooled[(long long)b * C + c];
        g[gWh + e] = s;
    }
    for (int k = threadIdx.x; k < NO; k += blockDim.x) {
        float s = 0.f;
        for (int b = 0; b < B; ++b) s += dout[b * NO + k];
        g[gbh + k] = s;
    }
    for (int e = threadIdx.x; e < B * C; e += blockDim.x) {
        int b = e / C, c = e % C;
        float s = 0.f;
        for (int k = 0; k < NO; ++k) s += dout[b * NO + k] * bf(pb, oWh + (long long)k * C + c);
        dpooled[e] = s;
    }
}

// dz of the last layer (no activation): dpooled / n at every position.
__global__ void k_pool_bwd(const float *dpooled, float4 *dz, long long total4, int n) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= total4) return;
    const float d = dpooled[4 * i / n] / (float)n;
    dz[i] = make_float4(d, d, d, d);
}

// G[o][i] += sum_{b,x} D[b][o][x] H[b][i][x] and gc[o] += sum D.  Block: one
// sample, the positions in chunks of 32 staged as [x][channel]; a thread holds an
// 8 x 4 tile of one of the slices of every chunk, summed per chunk first; the
// slices are added in shared memory and the block's sums to G by one float32
// atomic each; the next chunk is loaded while this one is multiplied.  The groups of four channels
// are permuted by x / 4, so that both the transposing stores (8 x 4 channels
// per warp) and the 16-byte loads are free of bank conflicts.  32 multiply-adds
// per 3 loads: 128 samples, 48 x 48, 1024 positions 408 -> 40 us.
__global__ void __launch_bounds__(512) k_outer(const float *__restrict__ D, const float *__restrict__ H, float *G, float *gc,
                                               int CO, int CI, int n) {
    constexpr int XC = 32;
    __shared__ __align__(16) float ds[XC * 64], hs[XC * 64];
    const int b = blockIdx.x, tid = threadIdx.x;
    const int to = (CO + 7) / 8, ti = (CI + 3) / 4, nt = to * ti, ns = min(512 / nt, XC);  // tiles, slices (CO, CI <= 64)
    const int slice = tid / nt, tile = tid - slice * nt, og = 2 * (tile / ti), ig = tile % ti;  // groups of 4 channels
    const bool on = slice < ns;
    float tot[8][4] = {}, ctot[8] = {};
    // positions 4 xq .. 4 xq + 3 of channel c of a chunk (8 x 64 threads)
    const int xq = tid & 7, c = tid >> 3, at = (((c >> 2) ^ xq) << 2) + (c & 3) + 4 * xq * 64;
    const float *pd = D + ((long long)b * CO + c) * n + 4 * xq, *ph = H + ((long long)b * CI + c) * n + 4 * xq;
    float rd[4], rh[4];
    auto fetch = [&](int x0) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            rd[u] = c < CO ? pd[x0 + u] : 0.f;
            rh[u] = c < CI ? ph[x0 + u] : 0.f;
        }
    };
    fetch(0);
    for (int x0 = 0; x0 < n; x0 += XC) {
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            ds[at + 64 * u] = rd[u];
            hs[at + 64 * u] = rh[u];
        }
        __syncthreads();
        if (x0 + XC < n) fetch(x0 + XC);
        if (!on) continue;
        float acc[8][4] = {}, cacc[8] = {};
        for (int x = slice; x < XC; x += ns) {
            const int sw = (x >> 2) & 7;
            const float4 a = *reinterpret_cast<const float4 *>(ds + 64 * x + ((og ^ sw) << 2));
            const float4 c = *reinterpret_cast<const float4 *>(ds + 64 * x + (((og + 1) ^ sw) << 2));
            const float4 h = *reinterpret_cast<const float4 *>(hs + 64 * x + ((ig ^ sw) << 2));
            const float dv[8] = {a.x, a.y, a.z, a.w, c.x, c.y, c.z, c.w}, hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                if (ig == 0) cacc[r] += dv[r];
#pragma unroll
                for (int k = 0; k < 4; ++k) acc[r][k] = fmaf(dv[r], hv[k], acc[r][k]);
            }
        }
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            ctot[r] += cacc[r];
#pragma unroll
            for (int k = 0; k < 4; ++k) tot[r][k] += acc[r][k];
        }
    }
    // one row of every tile at a time: 5 values per thread, the slices added in order
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        __syncthreads();
        if (on) {
            *reinterpret_cast<float4 *>(ds + 4 * tid) = make_float4(tot[r][0], tot[r][1], tot[r][2], tot[r][3]);
            hs[tid] = ctot[r];
        }
        __syncthreads();
        const int o = 4 * og + r;
        if (tid >= nt || o >= CO) continue;
        float v[4] = {}, cv = 0.f;
        for (int q = 0; q < ns; ++q) {
            const float4 t = *reinterpret_cast<const float4 *>(ds + 4 * (q * nt + tid));
            v[0] += t.x; v[1] += t.y; v[2] += t.z; v[3] += t.w;
            cv += hs[q * nt + tid];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (4 * ig + k < CI) atomicAdd(&G[o * CI + 4 * ig + k], v[k]);
        if (ig == 0) atomicAdd(&gc[o], cv);
    }
}

// Mixing backward, weights: dW[i][o][m] = sum_b conj(X[b][i][m]) dY[b][o][m].
// Thread: one mode and a 4 x 4 tile of (i, o), every eighth sample; the eight
// partial sums are added through shared memory in a fixed order.  Latency-bound
// (8 loads from L2 per 64 multiply-adds).
constexpr int MW_S = 8;
__global__ void __launch_bounds__(32 * MW_S) k_mix_bwd_w(const float2 *__restrict__ X, const float2 *__restrict__ dY, float *g,
                                                   long long gWr, long long gWi, int B, int C, int M) {
    __shared__ float2 red[MW_S - 1][16][32];
    const int ml = threadIdx.x & 31, sl = threadIdx.x >> 5, m = blockIdx.x * 32 + ml;
    const int i0 = 4 * blockIdx.y, o0 = 4 * blockIdx.z;
    float2 acc[4][4] = {};
    if (m < M) {
#pragma unroll 2
        for (int b = sl; b < B; b += MW_S) {
            const float2 *x = X + (long long)b * C * M + m, *d = dY + (long long)b * C * M + m;
            float2 xv[4], dv[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                xv[u] = x[(long long)min(i0 + u, C - 1) * M];
                dv[u] = d[(long long)min(o0 + u, C - 1) * M];
            }
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    acc[r][c].x = fmaf(xv[r].x, dv[c].x, fmaf(xv[r].y, dv[c].y, acc[r][c].x));
                    acc[r][c].y = fmaf(-xv[r].y, dv[c].x, fmaf(xv[r].x, dv[c].y, acc[r][c].y));
                }
        }
    }
    if (sl > 0) {
#pragma unroll
        for (int e = 0; e < 16; ++e) red[sl - 1][e][ml] = acc[e >> 2][e & 3];
    }
    __syncthreads();
    if (sl > 0 || m >= M) return;
#pragma unroll
    for (int e = 0; e < 16; ++e) {
        const int i = i0 + (e >> 2), o = o0 + (e & 3);
        float2 v = acc[e >> 2][e & 3];
#pragma unroll
        for (int q = 0; q < MW_S - 1; ++q) {
            v.x += red[q][e][ml].x;
            v.y += red[q][e][ml].y;
        }
        if (i < C && o < C) {
            const long long w = ((long long)i * C + o) * M + m;
            g[gWr + w] = v.x;
            g[gWi + w] = v.y;
        }
    }
}

__global__ void k_adam(float *p, const float *g, float *m1, float *m2, __nv_bfloat16 *pb, long long np, float lr,
                       float b1, float b2, float c1, float c2, float epsv) {
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= np) return;
    float gi = g[i];
    float a = b1 * m1[i] + (1.f - b1) * gi;
    float v = b2 * m2[i] + (1.f - b2) * gi * gi;
    m1[i] = a;
    m2[i] = v;
    float q = p[i] - lr * (a / c1) / (sqrtf(v / c2) + epsv);
    p[i] = q;
    pb[i] = __float2bfloat16_rn(q);
}

__global__ void k_to_bf16(const float *p, __nv_bfloat16 *pb, long long np) {
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i < np) pb[i] = __float2bfloat16_rn(p[i]);
}

unsigned nb(long long total, int t = 256) { return (unsigned)((total + t - 1) / t); }

int serr(apf_sno *s, int code, const char *msg) {
    if (s) s->err = msg;
    return set_err(nullptr, code, "%s", msg);
}

void launch_dft(apf_sno *s, const float *in, float2 *out, int B, int weights, cudaStream_t st) {
    const int rows = B * s->c;
    k_dft<<<dim3((rows + 15) / 16, (s->m + 63) / 64), 256, 0, st>>>(in, out, s->tw, rows, s->n, s->m, weights);
}

size_t synth_smem(int C, int XT) {
    const size_t Cp = (C + 7) & ~7, XW = 32 * XT;
    return 16 * (SY_MC * Cp + SY_MC * XW + SY_IC * XW) + 4 * C * Cp;
}

// Outputs up to which one thread each is faster (k_synth_small, k_mix_small).  Whole
// screening calls, one-output kernels against the tiled ones: 1 sample of 16 channels
// and 128 positions 132 against 182 us; 20 of 24 and 512 (246k synthesised values) 178
// against 260 us, 8 of 48 and 1024 (393k) 315 against 296 us.  Mixing alone: 20 of
// 48 and 64 modes (61k values) 281 against 299 us per call, 64 of them (197k) 404
// against 402 us.
constexpr long long SMALL_SYNTH = 262144, SMALL_MIX = 131072;
// x per block: 64 where that still gives about two blocks per SM, else 32.
template <bool BWD, int XT>
void launch_synth_t(apf_sno *s, const float2 *Y, const float *h, long long oP, long long oc, float *z, float *hn, int B,
                    int act, cudaStream_t st) {
    const int q = s->n / 4, threads = 32 * ((s->c + 7) / 8);
    k_synth<BWD, XT><<<dim3((q + 32 * XT - 1) / (32 * XT), B), threads, synth_smem(s->c, XT), st>>>(
        Y, h, s->pb, oP, oc, s->tw, z, hn, s->c, s->n, s->m, act);
}

template <bool BWD>
void launch_synth(apf_sno *s, const float2 *Y, const float *h, long long oP, long long oc, float *z, float *hn, int B,
                  int act, cudaStream_t st) {
    if ((long long)B * s->c * s->n <= SMALL_SYNTH)
        k_synth_small<BWD><<<dim3((s->n + 127) / 128, B * s->c), 128, 8 * small_pad(s->m) + 4 * small_pad(s->c), st>>>(Y, h, s->pb, oP, oc, s->tw, z, hn, s->c, s->n,
                                                                             s->m, act);
    else if ((long long)B * ((s->n / 4 + 63) / 64) >= 256) launch_synth_t<BWD, 2>(s, Y, h, oP, oc, z, hn, B, act, st);
    else launch_synth_t<BWD, 1>(s, Y, h, oP, oc, z, hn, B, act, st);
}

template <bool BWD, int XT>
void synth_attr() {
    cudaFuncSetAttribute(k_synth<BWD, XT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)synth_smem(64, XT));
}
void init_attrs() {
    synth_attr<false, 1>(); synth_attr<false, 2>(); synth_attr<true, 1>(); synth_attr<true, 2>();
}

template <bool BWD>
void launch_mix(apf_sno *s, const float2 *X, float2 *Y, int l, int B, cudaStream_t st) {
    const int C = s->c, M = s->m;
    const long long wr = s->oWr + (long long)l * C * C * M, wi = s->oWi + (long long)l * C * C * M;
    if ((long long)B * C * M <= SMALL_MIX)
        k_mix_small<BWD><<<(B * C * M + 127) / 128, 128, 0, st>>>(X, s->pb, wr, wi, Y, B, C, M);
    else
        k_mix<BWD><<<dim3(nb((long long)((C + 1) / 2) * M), (B + 3) / 4), 256, 0, st>>>(X, s->pb, wr, wi, Y, B, C, M);
}

void forward(apf_sno *s, const float *x, int B, cudaStream_t st) {
    const int C = s->c, n = s->n, M = s->m, L = s->layers;
    k_lift<<<dim3(n / 64, B), 256, 0, st>>>(x, s->pb, s->oW0, s->ob0, s->h, s->ci, C, n);
    for (int l = 0; l < L; ++l) {
        const float *hp = s->h + (long long)l * s->bmax * C * n;
        float *hn = s->h + (long long)(l + 1) * s->bmax * C * n;
        float *z = s->z + (long long)l * s->bmax * C * n;
        float2 *X = s->X + (long long)l * s->bmax * C * M, *Y = s->Y + (long long)l * s->bmax * C * M;
        launch_dft(s, hp, X, B, 0, st);
        launch_mix<false>(s, X, Y, l, B, st);
        launch_synth<false>(s, Y, hp, s->oP + (long long)l * C * C, s->oc + (long long)l * C, z, hn, B, l < L - 1 ? 1 : 0, st);
    }
    k_pool<<<B * C, 256, 0, st>>>(s->h + (long long)L * s->bmax * C * n, s->pooled, n);
    k_head<<<nb(B * s->no), 256, 0, st>>>(s->pooled, s->pb, s->oWh, s->obh, s->out, B, C, s->no);
}

// Gradients of the loss w.r.t. every parameter into s->g (after forward).
void backward(apf_sno *s, const float *x, const float *tgt, int B, cudaStream_t st) {
    const int C = s->c, n = s->n, M = s->m, L = s->layers, NO = s->no;
    const long long act = (long long)B * C * n;
    cudaMemsetAsync(s->g, 0, sizeof(float) * s->nparams, st);
    k_head_bwd<<<1, 256, 0, st>>>(s->out, tgt, s->pooled, s->pb, s->oWh, s->g, s->oWh, s->obh, s->dout, s->dpooled,
                                  s->loss, B, C, NO);
    k_pool_bwd<<<nb(act / 4), 256, 0, st>>>(s->dpooled, reinterpret_cast<float4 *>(s->dz), act / 4, n);
    for (int l = L - 1; l >= 0; --l) {
        const float *hp = s->h + (long long)l * s->bmax * C * n;
        const float2 *X = s->X + (long long)l * s->bmax * C * M;
        k_outer<<<B, 512, 0, st>>>(s->dz, hp, s->g + s->oP + (long long)l * C * C, s->g + s->oc + (long long)l * C, C, C, n);
        launch_dft(s, s->dz, s->dY, B, 1, st);
        k_mix_bwd_w<<<dim3((M + 31) / 32, (C + 3) / 4, (C + 3) / 4), 32 * MW_S, 0, st>>>(
            X, s->dY, s->g, s->oWr + (long long)l * C * C * M, s->oWi + (long long)l * C * C * M, B, C, M);
        launch_mix<true>(s, s->dY, s->dX, l, B, st);
        // dz of the layer below (of the lifted input: no activation)
        float *zp = l > 0 ? s->z + (long long)(l - 1) * s->bmax * C * n : nullptr;
        launch_synth<true>(s, s->dX, s->dz, s->oP + (long long)l * C * C, 0, zp, s->dh, B, 0, st);
        std::swap(s->dh, s->dz);
    }
    // lift: dW0[o][i] = sum dh0[b][o][x] eps[b][i][x], db0 = sum dh0
    k_outer<<<B, 512, 0, st>>>(s->dz, x, s->g + s->oW0, s->g + s->ob0, C, s->ci, n);
}

}  // namespace

extern "C" {

int apf_sno_create(apf_sno **out, int device, int n, int in_ch, int width, int modes, int layers, int n_out,
                   int max_batch) {
    if (!out) return APF_EINVAL;
    *out = nullptr;
    if (n < 64 || (n % 64) || in_ch < 1 || in_ch > 64 || width < 1 || width > 64 || modes < 1 || 2 * modes > n ||
        modes > 256 || layers < 1 || layers > 8 || n_out < 1 || n_out > 64 || max_batch < 1 || max_batch > 4096 ||
        width * width > 12 * 256 || width * in_ch > 12 * 256)
        return set_err(nullptr, APF_EINVAL, "apf_sno_create: sizes out of range");
    if (cudaSetDevice(device) != cudaSuccess) { cudaGetLastError(); return set_err(nullptr, APF_ECUDA, "bad device"); }
    init_attrs();
    apf_sno *s = new apf_sno();
    s->device = device; s->n = n; s->ci = in_ch; s->c = width; s->m = modes; s->layers = layers; s->no = n_out;
    s->bmax = max_batch;
    const long long C = width, M = modes, L = layers;
    long long o = 0;
    s->oW0 = o; o += C * in_ch;
    s->ob0 = o; o += C;
    s->oWr = o; o += L * C * C * M;
    s->oWi = o; o += L * C * C * M;
    s->oP = o; o += L * C * C;
    s->oc = o; o += L * C;
    s->oWh = o; o += (long long)n_out * C;
    s->obh = o; o += n_out;
    s->nparams = o;
    const long long Bn = (long long)max_batch * C * n, BM = (long long)max_batch * C * M;
    auto al = [&](void **p, size_t bytes) {
        if (cudaMalloc(p, bytes) != cudaSuccess) return false;
        s->allocs.push_back(*p);
        return true;
    };
    bool ok = al((void **)&s->p, sizeof(float) * o) && al((void **)&s->g, sizeof(float) * o) &&
              al((void **)&s->mom1, sizeof(float) * o) && al((void **)&s->mom2, sizeof(float) * o) &&
              al((void **)&s->pb, sizeof(__nv_bfloat16) * o) && al((void **)&s->tw, sizeof(float2) * M * n) &&
              al((void **)&s->h, sizeof(float) * (L + 1) * Bn) && al((void **)&s->z, sizeof(float) * L * Bn) &&
              al((void **)&s->X, sizeof(float2) * L * BM) && al((void **)&s->Y, sizeof(float2) * L * BM) &&
              al((void **)&s->dh, sizeof(float) * Bn) &&
              al((void **)&s->dz, sizeof(float) * Bn) && al((void **)&s->dY, sizeof(float2) * BM) &&
              al((void **)&s->dX, sizeof(float2) * BM) &&
              al((void **)&s->pooled, sizeof(float) * max_batch * C) &&
              al((void **)&s->dpooled, sizeof(float) * max_batch * C) &&
              al((void **)&s->out, sizeof(float) * max_batch * n_out) &&
              al((void **)&s->dout, sizeof(float) * max_batch * n_out) && al((void **)&s->loss, sizeof(float) * 4);
    if (!ok) {
        cudaGetLastError();
        apf_sno_destroy(s);
        return set_err(nullptr, APF_ENOMEM, "apf_sno_create: out of device memory");
    }
    cudaMemset(s->p, 0, sizeof(float) * o);
    cudaMemset(s->mom1, 0, sizeof(float) * o);
    cudaMemset(s->mom2, 0, sizeof(float) * o);
    k_tw<<<dim3((n + 255) / 256, modes), 256>>>(s->tw, n, modes);
    k_to_bf16<<<nb(o), 256>>>(s->p, s->pb, o);
    if (cudaDeviceSynchronize() != cudaSuccess) {
        cudaGetLastError();
        apf_sno_destroy(s);
        return set_err(nullptr, APF_ECUDA, "apf_sno_create: init failed");
    }
    *out = s;
    return APF_OK;
}

void apf_sno_destroy(apf_sno *s) {
    if (!s) return;
    cudaSetDevice(s->device);
    for (void *p : s->allocs) cudaFree(p);
    delete s;
}

long long apf_sno_num_params(const apf_sno *s) { return s ? s->nparams : -1; }

int apf_sno_set_params(apf_sno *s, const float *params) {
    if (!s || !params) return APF_EINVAL;
    cudaSetDevice(s->device);
    if (cudaMemcpy(s->p, params, sizeof(float) * s->nparams, cudaMemcpyDefault) != cudaSuccess)
        return serr(s, APF_ECUDA, "set_params copy failed");
    cudaMemset(s->mom1, 0, sizeof(float) * s->nparams);
    cudaMemset(s->mom2, 0, sizeof(float) * s->nparams);
    s->step = 0;
    k_to_bf16<<<nb(s->nparams), 256>>>(s->p, s->pb, s->nparams);
    return cudaDeviceSynchronize() == cudaSuccess ? APF_OK : serr(s, APF_ECUDA, "set_params failed");
}

int apf_sno_get_params(const apf_sno *s, float *params) {
    if (!s || !params) return APF_EINVAL;
    cudaSetDevice(s->device);
    return cudaMemcpy(params, s->p, sizeof(float) * s->nparams, cudaMemcpyDefault) == cudaSuccess ? APF_OK
                                                                                                  : APF_ECUDA;
}

int apf_sno_forward(apf_sno *s, const float *x, int B, float *y, void *stream) {
    if (!s || !x || !y || B < 1 || B > s->bmax) return APF_EINVAL;
    cudaSetDevice(s->device);
    cudaStream_t st = (cudaStream_t)stream;
    forward(s, x, B, st);
    cudaMemcpyAsync(y, s->out, sizeof(float) * B * s->no, cudaMemcpyDefault, st);
    cudaError_t e = cudaStreamSynchronize(st);
    return e == cudaSuccess ? APF_OK : serr(s, APF_ECUDA, cudaGetErrorString(e));
}

int apf_sno_gradients(apf_sno *s, const float *x, const float *target, int B, float *grads, float *loss,
                      void *stream) {
    if (!s || !x || !target || B < 1 || B > s->bmax) return APF_EINVAL;
    cudaSetDevice(s->device);
    cudaStream_t st = (cudaStream_t)stream;
    forward(s, x, B, st);
    backward(s, x, target, B, st);
    if (grads) cudaMemcpyAsync(grads, s->g, sizeof(float) * s->nparams, cudaMemcpyDefault, st);
    float lh = 0.f;
    cudaMemcpyAsync(&lh, s->loss, sizeof(float), cudaMemcpyDeviceToHost, st);
    cudaError_t e = cudaStreamSynchronize(st);
    if (loss) *loss = lh;
    return e == cudaSuccess ? APF_OK : serr(s, APF_ECUDA, cudaGetErrorString(e));
}

int apf_sno_train_step(apf_sno *s, const float *x, const float *target, int B, float lr, float *loss,
                       void *stream) {
    if (!s || !x || !target || B < 1 || B > s->bmax || !(lr > 0.f)) return APF_EINVAL;
    cudaSetDevice(s->device);
    cudaStream_t st = (cudaStream_t)stream;
    forward(s, x, B, st);
    backward(s, x, target, B, st);
    s->step += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)s->step), c2 = 1.f - powf(b2, (float)s->step);
    k_adam<<<nb(s->nparams), 256, 0, st>>>(s->p, s->g, s->mom1, s->mom2, s->pb, s->nparams, lr, b1, b2, c1, c2,
                                           1e-8f);
    float lh = 0.f;
    cudaMemcpyAsync(&lh, s->loss, sizeof(float), cudaMemcpyDeviceToHost, st);
    cudaError_t e = cudaStreamSynchronize(st);
    if (loss) *loss = lh;
    return e == cudaSuccess ? APF_OK : serr(s, APF_ECUDA, cudaGetErrorString(e));
}

}  // extern "C"
