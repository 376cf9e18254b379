// One-warp Cholesky of a 32 x 32 tile with its inverse, shared by the tensor-core solver's
// diagonal blocks (k_chol_tc.cu) and the refined FP64 solve (k_solve_ref.cu).
#pragma once
#include "common.cuh"

namespace otvmc {
namespace chol {

constexpr int TB = 32;  // tile of the block algorithms

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

// Steps m0 .. m1 - 1 of factor32, two pivots at a time, with W registers of a and x still in use.
template <int W>
__device__ __forceinline__ void factor32_steps(float (&a)[TB], float (&x)[TB], int m0, int m1, float* A, int lda,
                                               float* X, int ldx, float* scr, float dmin, bool& ok, float& isd) {
    const int lane = threadIdx.x & 31;
#pragma unroll 2
    for (int m = m0; m < m1; m += 2) {
        float2* col = reinterpret_cast<float2*>(scr) + ((m >> 1) & 1) * TB;
        const float l1 = lane >= m ? a[0] * isd : 0.f;
        const float lu1 = lane > m ? l1 : 0.f;
        const float d2 = __shfl_sync(0xffffffffu, fmaf(-lu1, l1, a[1]), m + 1);  // lane m + 1's own pivot
        const float s = __shfl_sync(0xffffffffu, l1, m + 1);
        ok = ok && d2 > dmin && isfinite(d2);
        const float isd2 = rsqrtf(ok ? d2 : 1.f);
        const float l2 = lane >= m + 1 ? fmaf(-lu1, s, a[1]) * isd2 : 0.f;
        const float lu2 = lane > m + 1 ? l2 : 0.f;
        col[(lane - m - 2) & (TB - 1)] = lane > m + 1 ? make_float2(lu1, lu2) : make_float2(0.f, 0.f);
        __syncwarp();
        float4 c[W / 2];
#pragma unroll
        for (int q = 0; q < W / 2; ++q) c[q] = ld4(reinterpret_cast<const float*>(col) + 4 * q);
        const float d = __shfl_sync(0xffffffffu, fmaf(-lu2, l2, fmaf(-lu1, l1, a[2])), (m + 2) & (TB - 1));
        const float x0 = x[0] * isd, x1 = fmaf(-s, x0, x[1]) * isd2;
        A[lane * lda + m] = l1;
        A[lane * lda + m + 1] = l2;
        X[m * ldx + lane] = x0;
        X[(m + 1) * ldx + lane] = x1;
        // the next pivot's root, ahead of the updates that hide it (none after the last step)
        ok = ok && (m + 2 == TB || (d > dmin && isfinite(d)));
        isd = rsqrtf(ok ? d : 1.f);
#pragma unroll
        for (int q = 0; q < W / 2 - 1; ++q) {
            a[2 * q] = fmaf(-lu2, c[q].y, fmaf(-lu1, c[q].x, a[2 * q + 2]));
            x[2 * q] = fmaf(-c[q].y, x1, fmaf(-c[q].x, x0, x[2 * q + 2]));
            a[2 * q + 1] = fmaf(-lu2, c[q].w, fmaf(-lu1, c[q].z, a[2 * q + 3]));
            x[2 * q + 1] = fmaf(-c[q].w, x1, fmaf(-c[q].z, x0, x[2 * q + 3]));
        }
    }
}

// Factor the 32 x 32 tile at A (row stride lda; lower triangle read) into L (written in place,
// zeros above the diagonal) and write X = L^-1 to X (row stride ldx, zeros above the diagonal).
// One warp: lane i holds row i of A and column i of X.  Step m: the pivot's reciprocal root scales
// column m of L (lanes i >= m) and row m of X; column m of L goes to the scratch (scr: 128 floats),
// from where every lane reads it for both updates, A_ij -= L_im L_jm and X_ij -= L_im X_mj.
// Bound: the chain of 32 pivots (FMA, shuffle, reciprocal square root, multiply: lane m + 1 forms
// the next pivot from its own entries, before the scratch is read back) and, before that, the
// instruction fetch: fully unrolled, the body is some 50 KB of code that runs once a call (16,000
// cycles alone, up to 50,000 beside other kernels).  The loop is therefore rolled: the registers
// shift by an entry a step (A_i,m+k and X_m+k,i sit in a[k] and x[k]) and the scratch is written
// shifted likewise.  7,200 cycles a step at a time, 4,600 with two pivots per exchange through the
// scratch, the unused tail of the registers dropped every eight steps, and the scratch read before
// the next root is taken (one warp alone on its SM).
// Returns false (uniformly over the warp) on a pivot that is not finite or not above dmin.
__device__ __forceinline__ bool factor32(float* A, int lda, float* X, int ldx, float* scr, float dmin) {
    const int lane = threadIdx.x & 31;
    float a[TB], x[TB];
#pragma unroll
    for (int q = 0; q < TB / 4; ++q) {
        const float4 v = ld4(A + lane * lda + 4 * q);
        a[4 * q] = v.x;
        a[4 * q + 1] = v.y;
        a[4 * q + 2] = v.z;
        a[4 * q + 3] = v.w;
    }
#pragma unroll
    for (int j = 0; j < TB; ++j) {
        if (j > lane) a[j] = 0.f;
        x[j] = j == lane ? 1.f : 0.f;
    }
    const float d = __shfl_sync(0xffffffffu, a[0], 0);
    bool ok = d > dmin && isfinite(d);
    // a few ulps suffice here: the factor is refined against the exact matrix later
    float isd = rsqrtf(ok ? d : 1.f);
    factor32_steps<32>(a, x, 0, 8, A, lda, X, ldx, scr, dmin, ok, isd);
    factor32_steps<24>(a, x, 8, 16, A, lda, X, ldx, scr, dmin, ok, isd);
    factor32_steps<16>(a, x, 16, 24, A, lda, X, ldx, scr, dmin, ok, isd);
    factor32_steps<8>(a, x, 24, 32, A, lda, X, ldx, scr, dmin, ok, isd);
    __syncwarp();
    return ok;
}

}  // namespace chol
}  // namespace otvmc
