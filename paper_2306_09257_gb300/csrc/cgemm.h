// Complex tensor-core products of the slab elimination and the field sweeps (internal).
#pragma once
#include "apf_internal.h"

#include <cuda.h>

constexpr int CG_MAX_PROB = 2 * APF_MAX_BATCH;  // products of one launch (two slab rows per design)

// Split form of a complex matrix, the operand of every product: `planes` bf16
// planes x = x0 + x1 (+ x2) of the real and of the imaginary part.  Element
// (r, c) of plane p, component q (0 re, 1 im) lies at
// base + (2 p + q) * qpitch + r * pitch + c.  A sub-block is another base.
struct Mirror {
    __nv_bfloat16 *base = nullptr;
    long long pitch = 0, qpitch = 0;
    Mirror off(long long r, long long c) const { return Mirror{base + r * pitch + c, pitch, qpitch}; }
};

// Where a product goes: float32 planes and / or the split form (null: not written).
struct CgOut {
    float *re = nullptr, *im = nullptr;
    long long ld = 0;
    Mirror m;
};

// out = alpha A B^T + beta in, A: M x K, B: N x K (rows of B = columns of the
// result), and the same values transposed to outT.
struct CgProblem {
    Mirror A, B;
    int M = 0;                       // rows of this problem (at most the launch's M)
    CgOut out, outT;
    const float *in_re = nullptr, *in_im = nullptr;
    long long ldi = 0;
    int *flags = nullptr;
    int t_block = 0;  // != 0 (the same for all problems): outT in float32 only inside diagonal blocks of this size
};

// nprob products of the same N, K (and at most M rows) in one launch.  sym: the
// result is symmetric (M = N, out and outT the same matrix, or outT without what
// nobody reads above the diagonal): only elements on and below the diagonal are
// computed, each written to both places; 32 x 32 diagonal blocks come out whole.  cross: the
// smaller sums of a long product in accumulators of their own (see cgemm.cu).
// rows: the row count by which the kernel form is chosen (0: M).
int cgemm_n(apf_ctx *c, int nprob, const CgProblem *pb, int planes, int M, int N, int K, float alpha, float beta,
            bool sym, bool cross, cudaStream_t s, int rows = 0);
void cgemm_init_attrs();
