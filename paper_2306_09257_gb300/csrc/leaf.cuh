// Diagonal-block inversion shared by the float64 and the mixed path.
// (1) leaf_gj / leaf_gj_regs: Gauss-Jordan elimination with partial (row)
// pivoting of one NB x NB block.  (2) lc: the mixed path's 128 x 128 and 64 x 64
// blocks, by a cluster of four and two CTAs.
// In (1), for the shared-memory form:  Thread t owns row t/4 and the columns sub + 4q
// (sub = t%4), so the 4 threads of a row sit in adjacent lanes and the
// pivot-row reads are conflict-free; rows are padded by 4 elements.
// Row interchanges of the sweep become column interchanges of the inverse,
// undone in reverse order at the end.
#pragma once
#include "apf_internal.h"

template <typename R>
struct Cplx;
template <>
struct Cplx<double> {
    using T = double2;
    __device__ static T mk(double a, double b) { return make_double2(a, b); }
};
template <>
struct Cplx<float> {
    using T = float2;
    __device__ static T mk(float a, float b) { return make_float2(a, b); }
};

// Planar (re, im) or interleaved global layout.
template <typename R, bool PLANAR>
struct LeafIO {
    R *re, *im;
    typename Cplx<R>::T *z;
    long long ld;
    __device__ typename Cplx<R>::T load(int r, int c) const {
        long long g = (long long)r * ld + c;
        if (PLANAR) return Cplx<R>::mk(re[g], im[g]);
        return z[g];
    }
    __device__ void store(int r, int c, typename Cplx<R>::T v) const {
        long long g = (long long)r * ld + c;
        if (PLANAR) { re[g] = v.x; im[g] = v.y; }
        else z[g] = v;
    }
};

template <typename R, int NB, bool PLANAR>
__device__ void leaf_gj(LeafIO<R, PLANAR> io, int *flags) {
    using T = typename Cplx<R>::T;
    constexpr int P = NB + 4;
    constexpr int NT = NB * 4;
    constexpr int Q = NB / 4;
    extern __shared__ __align__(16) unsigned char leaf_smem[];
    T *a = reinterpret_cast<T *>(leaf_smem);
    __shared__ T rowk[NB], colk[NB];
    __shared__ R mag[NB];
    __shared__ int piv[NB];
    __shared__ int s_p;
    const int t = threadIdx.x, i = t >> 2, sub = t & 3;
    for (int e = t; e < NB * NB; e += NT) {
        int r = e / NB, c = e % NB;  // NB is a compile-time power of two
        a[r * P + c] = io.load(r, c);
    }
    __syncthreads();
    if (t < NB) {
        T v = a[t * P];
        mag[t] = v.x * v.x + v.y * v.y;
    }
    __syncthreads();
    for (int k = 0; k < NB; ++k) {
        if (t < 32) {
            R best = (R)-1;
            int bi = k;
            for (int r = k + t; r < NB; r += 32) {
                R m = mag[r];
                if (m > best) { best = m; bi = r; }
            }
            for (int off = 16; off > 0; off >>= 1) {
                R ob = __shfl_down_sync(0xffffffffu, best, off);
                int oi = __shfl_down_sync(0xffffffffu, bi, off);
                if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
            }
            if (t == 0) {
                s_p = bi;
                piv[k] = bi;
                if (!(best > (R)0) || !isfinite((double)best)) atomicOr(flags, FLAG_SINGULAR);
            }
        }
        __syncthreads();
        const int p = s_p;
        if (p != k && t < NB) {
            T x = a[k * P + t];
            a[k * P + t] = a[p * P + t];
            a[p * P + t] = x;
        }
        __syncthreads();
        if (t < NB) {
            T d = a[k * P + k];
            R den = d.x * d.x + d.y * d.y;
            T inv = Cplx<R>::mk(d.x / den, -d.y / den);
            T v = a[k * P + t];
            rowk[t] = (t == k) ? inv : Cplx<R>::mk(v.x * inv.x - v.y * inv.y, v.x * inv.y + v.y * inv.x);
            colk[t] = a[t * P + k];
        }
        __syncthreads();
        const T f = colk[i];
        T *row = a + i * P;
        if (i == k) {
#pragma unroll 8
            for (int q = 0; q < Q; ++q) row[sub + 4 * q] = rowk[sub + 4 * q];
        } else {
            R m1 = (R)-1;
#pragma unroll 8
            for (int q = 0; q < Q; ++q) {
                const int j = sub + 4 * q;
                T x = (j == k) ? Cplx<R>::mk(0, 0) : row[j];
                T rk = rowk[j];
                x.x -= f.x * rk.x - f.y * rk.y;
                x.y -= f.x * rk.y + f.y * rk.x;
                row[j] = x;
                if (j == k + 1) m1 = x.x * x.x + x.y * x.y;
            }
            if (((k + 1) & 3) == sub && k + 1 < NB) mag[i] = m1;
        }
        if (i == k && ((k + 1) & 3) == sub && k + 1 < NB) {
            T x = rowk[k + 1];
            mag[i] = x.x * x.x + x.y * x.y;
        }
        __syncthreads();
    }
    for (int k = NB - 1; k >= 0; --k) {
        int p = piv[k];
        if (p != k && t < NB) {
            T x = a[t * P + k];
            a[t * P + k] = a[t * P + p];
            a[t * P + p] = x;
        }
        __syncthreads();
    }
    for (int e = t; e < NB * NB; e += NT) {
        int r = e / NB, c = e % NB;
        io.store(r, c, a[r * P + c]);
    }
}

template <int NB>
constexpr int leaf_smem_bytes(int elem_bytes) {
    return NB * (NB + 4) * elem_bytes;
}

// Register-resident variant for the mixed path: thread t keeps row t/4,
// columns sub + 4q (q < NB/4) of the block in registers; the pivot row is the
// only data exchanged through shared memory.  Rows are never swapped: step k
// takes the largest unused |a[r][k]| as pivot row p_k and eliminates column k
// from every other row.  With piv[k] = p_k and ipiv[p_k] = k the inverse is
// inv[ipiv[r]][piv[c]] = a[r][c] (written out by a scatter at the end).
// For the non-pivot rows the update x[j] -= f * prow[j] also produces the
// new column-k entry -f / pivot, because prow[k] holds 1 + 1/pivot there and
// x[k] = f before the update.
template <int NB>
__device__ void leaf_gj_regs(float *re, float *im, long long ld, int *flags) {
    constexpr int Q = NB / 4;
    __shared__ float2 prow[NB];
    __shared__ float mag[NB];
    __shared__ int piv[NB], ipiv[NB];
    __shared__ int s_p;
    const int t = threadIdx.x, i = t >> 2, sub = t & 3, lane = t & 31;
    float2 a[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        long long g = (long long)i * ld + sub + 4 * q;
        a[q] = make_float2(re[g], im[g]);
    }
    bool used = false;
    float2 col = a[0];  // column k value, valid on the owner lanes (sub == k % 4)
    if (sub == 0) mag[i] = col.x * col.x + col.y * col.y;
    __syncthreads();
    for (int k = 0; k < NB; ++k) {
        if (t < 32) {
            float best = -1.f;
            int bi = 0;
#pragma unroll
            for (int r0 = 0; r0 < NB; r0 += 32) {
                float m = mag[r0 + t];
                if (m > best) { best = m; bi = r0 + t; }
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                float ob = __shfl_down_sync(0xffffffffu, best, off);
                int oi = __shfl_down_sync(0xffffffffu, bi, off);
                if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
            }
            if (t == 0) {
                s_p = bi;
                piv[k] = bi;
                ipiv[bi] = k;
                if (!(best > 0.f) || !isfinite(best)) atomicOr(flags, FLAG_SINGULAR);
            }
        }
        __syncthreads();
        const int p = s_p;
        const float2 f = make_float2(__shfl_sync(0xffffffffu, col.x, (lane & ~3) | (k & 3)),
                                     __shfl_sync(0xffffffffu, col.y, (lane & ~3) | (k & 3)));
        float2 pinv;
        {
            float den = f.x * f.x + f.y * f.y;
            pinv = make_float2(f.x / den, -f.y / den);
        }
        if (i == p) {
            used = true;
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int j = sub + 4 * q;
                float2 x = (j == k) ? pinv
                                    : make_float2(a[q].x * pinv.x - a[q].y * pinv.y, a[q].x * pinv.y + a[q].y * pinv.x);
                a[q] = x;
                prow[j] = (j == k) ? make_float2(1.f + pinv.x, pinv.y) : x;
            }
        }
        __syncthreads();
        if (i != p) {
            const float nfx = -f.x, fy = f.y;
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const float2 pr = prow[sub + 4 * q];
                float2 x = a[q];
                x.x = fmaf(nfx, pr.x, x.x);
                x.x = fmaf(fy, pr.y, x.x);
                x.y = fmaf(nfx, pr.y, x.y);
                x.y = fmaf(-fy, pr.x, x.y);
                a[q] = x;
            }
        }
        // next pivot column: a uniform switch on its register slot
        float2 nc = make_float2(0.f, 0.f);
        switch ((k + 1) >> 2) {
#define APF_NC_CASE(Z) case Z: if (Z < Q) nc = a[Z < Q ? Z : 0]; break;
            APF_NC_CASE(0) APF_NC_CASE(1) APF_NC_CASE(2) APF_NC_CASE(3) APF_NC_CASE(4) APF_NC_CASE(5)
            APF_NC_CASE(6) APF_NC_CASE(7) APF_NC_CASE(8) APF_NC_CASE(9) APF_NC_CASE(10) APF_NC_CASE(11)
            APF_NC_CASE(12) APF_NC_CASE(13) APF_NC_CASE(14) APF_NC_CASE(15) APF_NC_CASE(16) APF_NC_CASE(17)
            APF_NC_CASE(18) APF_NC_CASE(19) APF_NC_CASE(20) APF_NC_CASE(21) APF_NC_CASE(22) APF_NC_CASE(23)
            APF_NC_CASE(24) APF_NC_CASE(25) APF_NC_CASE(26) APF_NC_CASE(27) APF_NC_CASE(28) APF_NC_CASE(29)
            APF_NC_CASE(30) APF_NC_CASE(31)
#undef APF_NC_CASE
            default: break;
        }
        col = nc;
        if (k + 1 < NB && sub == ((k + 1) & 3)) mag[i] = used ? -1.f : nc.x * nc.x + nc.y * nc.y;
        __syncthreads();
    }
    const int r = ipiv[i];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        long long g = (long long)r * ld + piv[sub + 4 * q];
        re[g] = a[q].x;
        im[g] = a[q].y;
    }
}

// Faster register-resident variant: two barriers per elimination step.
//  * The argmax for the next pivot is reduced per warp during the update
//    (by the lanes that own the next column) and finished redundantly by
//    every thread from the per-warp partials.
//  * The pivot row is published unscaled; each thread folds 1/pivot into its
//    own row factor g = f / a_pk.  Column k of the published row carries
//    a_pk + 1, so x[k] - g (a_pk + 1) = -g, the new column-k entry.
template <int NB>
__device__ void leaf_gj_regs2(float *re, float *im, long long ld, int *flags) {
    constexpr int Q = NB / 4;
    constexpr int NW = NB * 4 / 32;  // warps
    __shared__ float2 prow[NB];
    __shared__ float pmag[2][NW];
    __shared__ int pidx[2][NW];
    __shared__ int piv[NB], ipiv[NB];
    const int t = threadIdx.x, i = t >> 2, sub = t & 3, lane = t & 31, warp = t >> 5;
    float2 a[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        long long g = (long long)i * ld + sub + 4 * q;
        a[q] = make_float2(re[g], im[g]);
    }
    bool used = false;
    float2 col = a[0];
    // warp-level partial argmax of |col|^2 over the owner lanes (sub == k % 4)
    auto publish = [&](int k, int buf) {
        float m = (sub == (k & 3) && !used) ? col.x * col.x + col.y * col.y : -1.f;
        int idx = i;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            float om = __shfl_down_sync(0xffffffffu, m, off);
            int oi = __shfl_down_sync(0xffffffffu, idx, off);
            if (om > m || (om == m && oi < idx)) { m = om; idx = oi; }
        }
        if (lane == 0) { pmag[buf][warp] = m; pidx[buf][warp] = idx; }
    };
    publish(0, 0);
    __syncthreads();
    for (int k = 0; k < NB; ++k) {
        const int buf = k & 1;
        float best = -1.f;
        int p = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            float m = pmag[buf][w];
            int idx = pidx[buf][w];
            if (m > best || (m == best && idx < p)) { best = m; p = idx; }
        }
        if (t == 0) {
            piv[k] = p;
            ipiv[p] = k;
            if (!(best > 0.f) || !isfinite(best)) atomicOr(flags, FLAG_SINGULAR);
        }
        const float2 f = make_float2(__shfl_sync(0xffffffffu, col.x, (lane & ~3) | (k & 3)),
                                     __shfl_sync(0xffffffffu, col.y, (lane & ~3) | (k & 3)));
        if (i == p) {
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int j = sub + 4 * q;
                prow[j] = (j == k) ? make_float2(a[q].x + 1.f, a[q].y) : a[q];
            }
        }
        __syncthreads();
        // pivot value from the published row (column k holds a_pk + 1)
        const float2 pk = prow[k];
        const float2 apk = make_float2(pk.x - 1.f, pk.y);
        const float den = apk.x * apk.x + apk.y * apk.y;
        const float2 pinv = make_float2(apk.x / den, -apk.y / den);
        float2 nc = make_float2(0.f, 0.f);
        if (i != p) {
            const float2 g = make_float2(f.x * pinv.x - f.y * pinv.y, f.x * pinv.y + f.y * pinv.x);
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int j = sub + 4 * q;
                const float2 pr = prow[j];
                float2 x = a[q];
                x.x -= g.x * pr.x - g.y * pr.y;
                x.y -= g.x * pr.y + g.y * pr.x;
                a[q] = x;
                if (j == k + 1) nc = x;
            }
        } else {
            used = true;
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int j = sub + 4 * q;
                float2 x = (j == k) ? pinv
                                    : make_float2(a[q].x * pinv.x - a[q].y * pinv.y, a[q].x * pinv.y + a[q].y * pinv.x);
                a[q] = x;
                if (j == k + 1) nc = x;
            }
        }
        col = nc;
        if (k + 1 < NB) publish(k + 1, buf ^ 1);
        __syncthreads();
    }
    const int r = ipiv[i];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        long long g = (long long)r * ld + piv[sub + 4 * q];
        re[g] = a[q].x;
        im[g] = a[q].y;
    }
}

// ---------------------------------------------------------------------------
// Inverse of a 128 x 128 (64 x 64) float32 block by a cluster of NP = four (two)
// CTAs of 512 threads: block Gauss-Jordan elimination in place over NP 32-column
// panels, CTA q holding the panel of columns 32 q .. 32 q + 31 in shared memory.
// Step p, with panel p as it stands (F) and the inverse P^-1 of its 32 x 32 pivot
// block in every CTA: R = P^-1 A_p, A_i -= F_i R, A_p = R (on panel p itself:
// P^-1 and -F_i P^-1).
// These blocks sit one after the other on the critical path of every inversion,
// so what counts is latency, and the chain of 32 NP pivots bounds it.  Four
// warps of the next panel's CTA invert its pivot block and store the inverse to the
// others (distributed shared memory) while these copy the panel.
// Updating the next pivot block alone first, and the rest beside its inversion,
// is no faster: the inversion then takes twice as long (it shares the SM's issue slots).
// Measured: 34 us per 128 block; 60 us with every CTA inverting the pivot block (400 clocks
// a pivot) after copying the panel, 93 us in one CTA.  64 block: 15 us; 56 us by pivots
// over all rows in one CTA.
// ---------------------------------------------------------------------------
namespace lc {
constexpr int NT = 512, PT = 34;  // threads, row pitch (float2; rows 16-byte aligned, columns conflict-free)

struct Leaf {  // of the 32 x 32 inversion
    float2 g[32 * 32], scale[32];
    int piv[32];
};
template <int NP>
struct Smem {
    static constexpr int N = 32 * NP, GROUPS = NT / N;  // rows and columns; threads per column
    float2 own[N * PT], F[N * PT], inv[32 * PT], R[32 * PT];
    float2 v[N], wpart[16][32], w[32], zpart[NP][GROUPS][N];
    float part[NP];
    Leaf leaf;
};

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// Shared-memory object `p` of cluster CTA `rank` (generic address).
template <typename T>
__device__ __forceinline__ T *peer(T *p, int rank) {
    uint64_t a;
    asm volatile("mapa.u64 %0, %1, %2;" : "=l"(a) : "l"((uint64_t)p), "r"(rank));
    return reinterpret_cast<T *>(a);
}
// Store to the same place in all CTAs of the cluster.
template <int NP, typename T>
__device__ __forceinline__ void store_all(T *p, T v) {
#pragma unroll
    for (int q = 0; q < NP; ++q) *peer(p, q) = v;
}

// Pivoted Gauss-Jordan inverse of the 32 x 32 block `a` (pitch PT) into `out`, by
// warps 0-3: lane i of every warp holds row i, warp w the columns 8w .. 8w+7.  Rows
// are not swapped: step k takes the unused row with the largest |a[p][k]| (a warp
// maximum over |.|^2 with its low five bits replaced by the row), and rows are
// divided by their pivots only at the end, so that a step leaves its own row
// alone.  All that a step's pivot needs lies in the warp that holds its column: for
// eight steps that warp runs ahead on its own (pivot row by shuffles, all issued
// before their first use; reciprocals beside the maximum) and leaves the column's
// factors in shared memory; the other warps follow two steps at a time behind
// named barriers, at which it does not wait (1-4 and 5-8 by turns: it waits for the
// next warp's while the others may still be at its own).  A zero pivot leaves
// infinities or NaN, which the caller's check of the result finds.
// Measured: 195 clocks per pivot; 400 with a barrier of all four warps and the
// pivot row through shared memory.
static __device__ void leaf32(Leaf &sm, const float2 *a, float2 *out) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    float2 x[8];
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
        const float4 q = *reinterpret_cast<const float4 *>(a + lane * PT + 8 * w + j);
        x[j] = make_float2(q.x, q.y);
        x[j + 1] = make_float2(q.z, q.w);
    }
    unsigned keep = ~31u, low = lane;  // both 0 once the row has been a pivot
    int mystep = 0;
    auto shuffle = [](float2 v, int p) {
        return make_float2(__shfl_sync(0xffffffffu, v.x, p), __shfl_sync(0xffffffffu, v.y, p));
    };
    auto apply = [](float2 &c, float2 g, float2 r) {
        c.x = fmaf(-g.x, r.x, fmaf(g.y, r.y, c.x));
        c.y = fmaf(-g.x, r.y, fmaf(-g.y, r.x, c.y));
    };
    for (int kw = 0; kw < 4; ++kw) {
        const int bar = 1 + 4 * (kw & 1);
        if (w == kw) {
            unsigned key, best;
            float2 rec;  // this lane's 1 / x
            auto search = [&](float2 v) {
                const float den = fmaf(v.x, v.x, v.y * v.y);
                key = (__float_as_uint(den) & keep) | low;
                best = __reduce_max_sync(0xffffffffu, key);
                float rd;
                asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rd) : "f"(den));
                rec = make_float2(v.x * rd, -v.y * rd);
            };
            search(x[0]);
#pragma unroll
            for (int kl = 0; kl < 8; ++kl) {
                const int k = 8 * kw + kl, p = (int)(best & 31u);
                const float2 inv = shuffle(rec, p), f = x[kl];
                float2 r[8];
#pragma unroll
                for (int i = 1; i < 8; ++i) r[(kl + i) & 7] = shuffle(x[(kl + i) & 7], p);
                const bool isp = lane == p;
                const float2 g = isp ? make_float2(0.f, 0.f)
                                     : make_float2(fmaf(f.x, inv.x, -f.y * inv.y), fmaf(f.x, inv.y, f.y * inv.x));
                if (isp) {
                    keep = low = 0u;
                    mystep = k;
                }
                apply(x[(kl + 1) & 7], g, r[(kl + 1) & 7]);
                if (kl < 7) search(x[(kl + 1) & 7]);
                sm.piv[k] = p;
                sm.scale[k] = inv;
                sm.g[32 * k + lane] = g;
                if (kl & 1) {
                    __syncwarp();
                    asm volatile("bar.arrive %0, 128;" ::"r"(bar + (kl >> 1)) : "memory");
                }
#pragma unroll
                for (int i = 2; i < 8; ++i) apply(x[(kl + i) & 7], g, r[(kl + i) & 7]);
                x[kl] = isp ? make_float2(1.f, 0.f) : make_float2(-g.x, -g.y);
            }
            __syncwarp();
        } else {
#pragma unroll
            for (int kl = 0; kl < 8; kl += 2) {
                asm volatile("bar.sync %0, 128;" ::"r"(bar + (kl >> 1)) : "memory");
                const int k = 8 * kw + kl;
                const int p0 = sm.piv[k], p1 = sm.piv[k + 1];
                const float2 g0 = sm.g[32 * k + lane], g1 = sm.g[32 * (k + 1) + lane];
                if (lane == p0 || lane == p1) {
                    keep = low = 0u;
                    mystep = lane == p0 ? k : k + 1;
                }
                float2 r[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) r[j] = shuffle(x[j], p0);
#pragma unroll
                for (int j = 0; j < 8; ++j) apply(x[j], g0, r[j]);
#pragma unroll
                for (int j = 0; j < 8; ++j) r[j] = shuffle(x[j], p1);
#pragma unroll
                for (int j = 0; j < 8; ++j) apply(x[j], g1, r[j]);
            }
        }
    }
    const float2 q = sm.scale[mystep];
#pragma unroll
    for (int j = 0; j < 8; ++j)
        out[mystep * PT + sm.piv[8 * w + j]] = make_float2(x[j].x * q.x - x[j].y * q.y, x[j].x * q.y + x[j].y * q.x);
}

// acc += S f u over 32 k: NR rows f (32 contiguous elements each) times the columns
// 0, 1, 16, 17 of u (pitch PT).  Shared memory hands out 128 bytes per clock,
// broadcasts included, so the tile counts: with two rows and four columns per
// thread R takes 1.9k clocks, 2.7k with one row and two columns.  The update (three
// rows, four columns) takes 4.8k, as with two columns; its multiply-adds alone are 3.1k.
template <int S, int NR>
__device__ __forceinline__ void multiply(float4 (&acc)[NR][2], const float2 *const (&f)[NR], const float2 *u) {
#pragma unroll 4
    for (int k = 0; k < 32; k += 2) {
        float4 q[NR];
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            q[i] = *reinterpret_cast<const float4 *>(f[i] + k);
            if (S < 0) q[i] = make_float4(-q[i].x, -q[i].y, -q[i].z, -q[i].w);
        }
#pragma unroll
        for (int kk = 0; kk < 2; ++kk)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const float4 w = *reinterpret_cast<const float4 *>(u + (k + kk) * PT + 16 * j);
#pragma unroll
                for (int i = 0; i < NR; ++i) {
                    const float qx = kk ? q[i].z : q[i].x, qy = kk ? q[i].w : q[i].y;
                    float4 &c = acc[i][j];
                    c.x = fmaf(qx, w.x, fmaf(-qy, w.y, c.x));
                    c.y = fmaf(qx, w.y, fmaf(qy, w.x, c.y));
                    c.z = fmaf(qx, w.z, fmaf(-qy, w.w, c.z));
                    c.w = fmaf(qx, w.w, fmaf(qy, w.z, c.w));
                }
            }
    }
}

// The inverse of the block at (re, im), in place; each CTA passes its panel
// (sm.own) to `also` as well.  Returns (the same in every thread of the cluster)
// whether the result passed the check below; if not, the block is as it was.
template <int NP, typename Also>
static __device__ bool invert(Smem<NP> &sm, float *re, float *im, long long ld, int rank, Also also) {
    constexpr int N = Smem<NP>::N, GROUPS = Smem<NP>::GROUPS, NI = 32 / GROUPS;
    const int t = threadIdx.x;
    cluster_arrive();
    {
        float2 x[2 * NP], f[2 * NP];
#pragma unroll
        for (int i = 0; i < 2 * NP; ++i) {
            const long long g = (long long)((t >> 5) + 16 * i) * ld + (t & 31);
            f[i] = make_float2(re[g], im[g]);
            x[i] = make_float2(re[g + 32 * rank], im[g + 32 * rank]);
        }
#pragma unroll
        for (int i = 0; i < 2 * NP; ++i) {
            const int e = ((t >> 5) + 16 * i) * PT + (t & 31);
            sm.F[e] = f[i];
            sm.own[e] = x[i];
        }
    }
    __syncthreads();
    if (t < 128) {
        leaf32(sm.leaf, sm.F, sm.inv);
    } else if (t < 128 + N) {
        float sn, cs;
        sincosf(2.3999632f * (float)(t - 128), &sn, &cs);
        sm.v[t - 128] = make_float2(cs, sn);
    }
    // this thread's share of the original block, for the check: a column, NI rows
    const int grp = t / N, col = t % N;
    float *const ore = re + (32 * rank + NI * grp) * ld + col, *const oim = im + (ore - re);
    float xr[NI], xi[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        xr[i] = ore[i * ld];
        xi[i] = oim[i * ld];
    }
    __syncthreads();
    cluster_wait();  // every CTA has started: its shared memory can be written
    const int cp = 2 * (t & 15), row = t >> 4;  // this thread's share of a copy: column pair, row of each block
    const int tc = 2 * (t & 7), tr = t >> 3;    // and of a product: columns tc, tc + 1, tc + 16, tc + 17, row
    for (int p = 0; p < NP; ++p) {
        // R = P^-1 A_p (the panel's own columns: R = P^-1), two rows and four columns per thread
        float4 r[2][2];
        if (t < 128) {
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j)
                    r[i][j] = rank == p ? *reinterpret_cast<const float4 *>(sm.inv + (tr + 16 * i) * PT + tc + 16 * j)
                                        : make_float4(0.f, 0.f, 0.f, 0.f);
            if (rank != p) {
                const float2 *const f[2] = {sm.inv + tr * PT, sm.inv + (tr + 16) * PT};
                multiply<1>(r, f, sm.own + 32 * p * PT + tc);
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j) *reinterpret_cast<float4 *>(sm.R + (tr + 16 * i) * PT + tc + 16 * j) = r[i][j];
        }
        __syncthreads();
        // A_i -= F_i R for the other row blocks, four columns of one row of each per thread.
        // On panel p F is the panel itself: its rows are read and written by the same lanes.
        if (t < 256) {
            float4 acc[NP - 1][2];
#pragma unroll
            for (int i = 0; i < NP - 1; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j)
                    acc[i][j] = rank == p ? make_float4(0.f, 0.f, 0.f, 0.f)
                                          : *reinterpret_cast<const float4 *>(sm.own + (32 * (i < p ? i : i + 1) + tr) * PT + tc + 16 * j);
            const float2 *F = rank == p ? sm.own : sm.F;
            const float2 *f[NP - 1];
#pragma unroll
            for (int i = 0; i < NP - 1; ++i) f[i] = F + (32 * (i < p ? i : i + 1) + tr) * PT;
            multiply<-1>(acc, f, sm.R + tc);
            __syncwarp();
#pragma unroll
            for (int i = 0; i < NP - 1; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j)
                    *reinterpret_cast<float4 *>(sm.own + (32 * (i < p ? i : i + 1) + tr) * PT + tc + 16 * j) = acc[i][j];
        }
        if (t < 128) {
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j)
                    *reinterpret_cast<float4 *>(sm.own + (32 * p + tr + 16 * i) * PT + tc + 16 * j) = r[i][j];
        }
        if (p == NP - 1) break;
        cluster_arrive();
        if (rank == p + 1) {
            __syncthreads();
            if (t < 128) {
                leaf32(sm.leaf, sm.own + 32 * (p + 1) * PT, sm.inv);
                asm volatile("bar.sync 9, 128;" ::: "memory");
                cluster_wait();
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float2 *e = sm.inv + (8 * i + (t >> 4)) * PT + cp;
                    const float4 v = *reinterpret_cast<const float4 *>(e);
#pragma unroll
                    for (int q = 1; q < NP; ++q) *reinterpret_cast<float4 *>(peer(e, (rank + q) % NP)) = v;
                }
            } else {
                cluster_wait();
            }
        } else {
            cluster_wait();  // panel p + 1 is up to date
            const float2 *src = peer(sm.own, p + 1);
            float4 f[NP - 1];
#pragma unroll
            for (int i = 0; i < NP - 1; ++i) {
                const int r = 32 * (i < p + 1 ? i : i + 1) + row;
                f[i] = *reinterpret_cast<const float4 *>(src + r * PT + cp);
            }
#pragma unroll
            for (int i = 0; i < NP - 1; ++i) {
                const int r = 32 * (i < p + 1 ? i : i + 1) + row;
                *reinterpret_cast<float4 *>(sm.F + r * PT + cp) = f[i];
            }
        }
        cluster_arrive();  // every CTA has panel p + 1 and its pivot block's inverse
        cluster_wait();
    }
    __syncthreads();
    for (int e = t; e < N * 16; e += NT) {
        const int r = e >> 4, c = 2 * (e & 15);
        const float2 u = sm.own[r * PT + c], v = sm.own[r * PT + c + 1];
        const long long g = r * ld + 32 * rank + c;
        *reinterpret_cast<float2 *>(re + g) = make_float2(u.x, v.x);
        *reinterpret_cast<float2 *>(im + g) = make_float2(u.y, v.y);
        also(r, 32 * rank + c, u, v);
    }
    // Self-check.  Pivoting stays inside the 32 x 32 blocks, so a nearly singular
    // leading sub-block of a block that is itself well conditioned spoils the
    // elimination; apply the computed inverse to a fixed unit-modulus probe v and
    // compare (v^T X^-1) X with v^T.  Above 2e-5 relative residual (a sound block
    // gives a few 1e-7) the block is inverted again by Gauss-Jordan with pivoting
    // over all rows.
    {
        const int g = t >> 5, c = t & 31;
        float2 y = make_float2(0.f, 0.f);
#pragma unroll
        for (int r = 2 * NP * g; r < 2 * NP * (g + 1); ++r) {
            const float2 m = sm.own[r * PT + c], v = sm.v[r];
            y.x += m.x * v.x - m.y * v.y;
            y.y += m.x * v.y + m.y * v.x;
        }
        sm.wpart[g][c] = y;
    }
    __syncthreads();
    if (t < 32) {
        float2 y = make_float2(0.f, 0.f);
#pragma unroll
        for (int g = 0; g < 16; ++g) {
            y.x += sm.wpart[g][t].x;
            y.y += sm.wpart[g][t].y;
        }
        sm.w[t] = y;
    }
    __syncthreads();
    {
        float2 z = make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const float2 y = sm.w[NI * grp + i];
            z.x += xr[i] * y.x - xi[i] * y.y;
            z.y += xr[i] * y.y + xi[i] * y.x;
        }
        store_all<NP>(&sm.zpart[rank][grp][col], z);
    }
    cluster_arrive();
    cluster_wait();  // the last access to another CTA's shared memory is done
    if (t < N) {
        float2 z = make_float2(-sm.v[t].x, -sm.v[t].y);
#pragma unroll
        for (int q = 0; q < NP * GROUPS; ++q) {
            const float2 u = sm.zpart[q / GROUPS][q % GROUPS][t];
            z.x += u.x;
            z.y += u.y;
        }
        float e2 = z.x * z.x + z.y * z.y;
#pragma unroll
        for (int off = 16; off; off >>= 1) e2 += __shfl_xor_sync(0xffffffffu, e2, off);
        if ((t & 31) == 0) sm.part[t >> 5] = e2;
    }
    __syncthreads();
    float e2 = 0.f;
#pragma unroll
    for (int i = 0; i < NP; ++i) e2 += sm.part[i];
    if (e2 <= 4e-10f * N) return true;  // (2e-5)^2 |v|^2; NaN fails
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        ore[i * ld] = xr[i];
        oim[i * ld] = xi[i];
    }
    cluster_arrive();
    cluster_wait();  // the block is whole again
    return false;
}
}  // namespace lc
