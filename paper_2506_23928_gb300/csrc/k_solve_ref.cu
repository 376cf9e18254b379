// FP64 solve of (S + eps I) delta = D (the otVMC equation with the diagonal-shift regulariser) by
// an FP32 Cholesky factorization and iterative refinement to FP64: one cluster of CTAs per
// trajectory.
//
//   1. d_i = 2^-round(log2 sqrt(S_ii + eps)): the factored matrix is d A d, whose diagonal lies in
//      [1/2, 2] (powers of two: no rounding), so that rows of very different sizes (biases and the
//      tied sums of the homogeneous parameters) do not cost accuracy.
//   2. FP32 left-looking factorization in 32-wide block columns.  Per block column the CTAs of the
//      cluster take chunks of 256 rows of the update C = A - L L_b^T (SIMT, 4 x 4 per thread,
//      operands staged by asynchronous copies); one warp of CTA 0 factors and inverts the
//      diagonal tile (factor32); the CTAs multiply their rows of C by the inverse.
//   3. dx from the FP32 factor (CTA 0), x += dx in FP64, r -= A dx (rows over the warps of the cluster), from
//      x = 0 and r = D until the next correction, foretold from the last two, is below 2^-54 of x; the real
//      and the imaginary system separately (they may differ by any factor).  A dx is taken from whole
//      numbers: d S d in units of 2^-60 as three digits of 21 bits, dx / d rounded to 28 bits of its largest
//      entry (the rounded dx is the correction), their products summed exactly in 64-bit integers, so
//      that r is that of the sum of the corrections to about 2^-73 of D.  The solution is that sum rounded to
//      FP64.  All that is lost are the bits of d S d beyond 2^-60 in entries below 2^-8 (P = 399,
//      conditions 3e3 to 5e3: 2e-16 of the largest entry; with x in three digits and the six largest of
//      their nine products 1e-14; an FP64 Cholesky 2e-14 to 6e-14).
//
// Bound: the FP64 rate of these GPUs is 1/64 of the FP32 one.  The O(P^3) part runs in FP32; of the
// residuals' O(P^2), the integer form takes about 30 integer instructions an entry, less than half the
// time of two FP64 multiply-adds.
//
// 100 trajectories of P = 399: 0.75 ms (0.80 ms with the residual from all of x; 8.8 ms with the FP64
// factorization, one CTA per trajectory); 8 of P = 528: 0.80 ms (15 ms).  Below P = 48 the factor and its inverses do not fit
// the scratch that the FP64 factorization needs anyway.
//
// A trajectory is left to the FP64 factorization (flag 1) when a pivot of the FP32 one is not
// clear of the shift test's threshold by several times the FP32 rounding to be expected in it (so
// that the decision to raise the shift is FP64's; an estimate, not a bound: the worst case of a pivot's
// rounding grows as P, not sqrt(P)), when an entry is not finite, or when the refinement does not
// converge.  Such a call pays for the attempt as well: 9.1 ms for 8.8 ms at 100 trajectories of P = 399 on 300
// samples and a shift of 1e-6, whose pivots end near the shift (1.4 ms at a shift of 1e-4, which converges).
#include <cooperative_groups.h>

#include "chol_tile.cuh"
#include "common.cuh"

namespace cg = cooperative_groups;

namespace otvmc {
namespace solref {

using chol::factor32;
using chol::ld4;

constexpr int TB = 32;        // block column
constexpr int RC = 256;       // rows of one update chunk
constexpr int KC = 32;        // columns of L staged at a time
constexpr int THREADS = 512;
constexpr int WARPS = THREADS / 32;
constexpr int MAX_ITER = 12;

// Per-trajectory scratch in FP32: L (column-major, stride ld), the inverses of the diagonal
// tiles, then the residual's exchange buffers in FP64.
__host__ __device__ inline size_t ld_of(int P) { return (size_t)((P + 3) / 4) * 4; }

struct alignas(16) Smem {  // its size a multiple of 16: float4 vectors follow it
    float As[2][KC][RC];  // staged L; in the substitutions the next tile's inverse
    float Bs[2][KC][TB];
    float Dg[TB][TB + 4];
    float X[TB][TB + 4];
    float scr[4 * TB];
    float t[2][TB];
    uint32_t red[2][WARPS];
    int zex[2];  // CTA 0: exponents of the units of the corrections
    int flag;
};

__device__ __forceinline__ void cp16(void* dst, const void* src, bool ok) {
    const int n = ok ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(n));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// |v| as a whole number that orders like it to 2^-20: the upper half of its bits, at least 1 where v is not
// zero.  Infinities and NaN are the largest.  Maxima are taken of these: with maxima in FP64
// over the CTA, eight an iteration, 100 trajectories of P = 399 took 862 us; 771 us so.
__device__ __forceinline__ uint32_t mag_key(double v) {
    return ((uint32_t)__double2hiint(v) & 0x7FFFFFFFu) | (__double2loint(v) != 0 ? 1u : 0u);
}
__device__ __forceinline__ double key_value(uint32_t k) {
    return k >= 0x7FF00000u ? INFINITY : __hiloint2double((int)k, 0);
}
// e with 2^(e - 1) <= v < 2^e for the v of a finite key (-1022 for zero and below the normal range)
__device__ __forceinline__ int key_exponent(uint32_t k) { return max((int)(k >> 20), 0) - 1022; }
// 2^k, |k| < 1000
__device__ __forceinline__ double pow2(int k) { return __hiloint2double((1023 + k) << 20, 0); }

// the largest a and the largest b over the CTA
__device__ uint2 block_max2(uint32_t a, uint32_t b, uint32_t (*red)[WARPS]) {
    static_assert(WARPS == 16, "a warp's maximum to each of 16 lanes");
    a = __reduce_max_sync(0xffffffffu, a);
    b = __reduce_max_sync(0xffffffffu, b);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = a;
        red[1][threadIdx.x >> 5] = b;
    }
    __syncthreads();
    const uint32_t v = __reduce_max_sync(0xffffffffu, red[0][threadIdx.x & 15]);
    return make_uint2(v, __reduce_max_sync(0xffffffffu, red[1][threadIdx.x & 15]));
}

// The three 21-bit digits of s 2^(60 + sh), truncated towards zero, each with the sign of s: exact
// while |s 2^sh| >= 2^-8, an error below 2^-60 otherwise.  |s 2^sh| < 4 (larger values come out
// wrong: the refinement then fails).  32-bit integer instructions only: conversions from FP64 run
// at the FP64 rate.
__device__ __forceinline__ void digits_of(double s, int sh, int (&d)[3]) {
    const uint32_t hw = (uint32_t)__double2hiint(s), lw = (uint32_t)__double2loint(s);
    const int e = (int)((hw >> 20) & 0x7FFu);
    // mantissa left-justified in 64 bits, then shifted right: 2^52 at exponent 0 goes to 2^60, so
    // the top bit of the justified mantissa (2^63) moves right by 3 - exponent
    uint32_t hi = 0x80000000u | __funnelshift_l(lw, hw, 11) & 0x7FFFFFFFu, lo = lw << 11;
    const int r = 3 + 1023 - e - sh;
    if (e == 0 || r >= 64 || r < 0) hi = lo = 0u;
    if (r >= 32) {
        lo = hi;
        hi = 0u;
    }
    lo = __funnelshift_r(lo, hi, r & 31);
    hi >>= (r & 31);
    const int sg = (int)hw >> 31;  // 0 or -1
    d[2] = ((int)(lo & 0x1FFFFFu) ^ sg) - sg;
    d[1] = ((int)(__funnelshift_r(lo, hi, 21) & 0x1FFFFFu) ^ sg) - sg;
    d[0] = ((int)(hi >> 10) ^ sg) - sg;
}

// s 2^sh in FP32, rounded to nearest away from zero, without FP64 instructions (0 below the normal
// range, infinity above it).
__device__ __forceinline__ float scaled_float(double s, int sh) {
    const uint32_t hw = (uint32_t)__double2hiint(s), lw = (uint32_t)__double2loint(s);
    const int e = (int)((hw >> 20) & 0x7FFu) + sh - 1023 + 127;
    const uint32_t m = ((hw & 0xFFFFFu) << 3) | (lw >> 29);
    const uint32_t b = ((uint32_t)e << 23) + m + ((lw >> 28) & 1u);
    const uint32_t u = e <= 0 ? 0u : e >= 255 ? 0x7F800000u : b;
    return __uint_as_float(u | (hw & 0x80000000u));
}

// y (two right-hand sides in shared memory, stride PY) <- (L L^T)^-1 y, by CTA 0.  Each of the
// 2 P / 32 steps is two barriers around a 32 x 32 product and a rank-32 update of y; the tile of L
// that the update needs is loaded into registers before the product, the next inverse into shared
// memory by asynchronous copies, so that a step waits for global memory once.
__device__ void solve32(int P, int PY, size_t ld, const float* L, const float* Xi, float* y, Smem& sm) {
    const int tid = threadIdx.x;
    const int nblk = (P + TB - 1) / TB;
    float* xb = &sm.As[0][0][0];  // two inverses, [2][TB][TB + 4]
    constexpr int XS = TB * (TB + 4);
    auto fetch = [&](int b, int s) {
        if (tid < TB * TB / 4) {
            const int i = tid >> 3, c4 = 4 * (tid & 7);
            cp16(xb + s * XS + i * (TB + 4) + c4, Xi + (size_t)b * TB * TB + i * TB + c4, true);
        }
        cp_commit();
    };
    fetch(0, 0);
    // forward, right-looking: y_b = X_b y_b, then the rows below lose L y_b
    for (int b = 0; b < nblk; ++b) {
        const int jb = b * TB, i0 = jb + TB + tid;
        float l[TB];
        if (i0 < P) {
#pragma unroll
            for (int c = 0; c < TB; ++c) l[c] = L[(size_t)(jb + c) * ld + i0];
        }
        cp_wait<0>();
        __syncthreads();  // this inverse and the last update of y
        fetch(b + 1 < nblk ? b + 1 : b, (b + 1) & 1);
        if (tid < 2 * TB) {
            const int h = tid >> 5, i = tid & 31;
            const float* Xr = xb + (b & 1) * XS + i * (TB + 4);
            float s = 0.f;
#pragma unroll
            for (int q = 0; q < TB / 4; ++q) {
                const float4 v = ld4(Xr + 4 * q);
                const float4 w = ld4(y + h * PY + jb + 4 * q);
                s = fmaf(v.x, w.x, fmaf(v.y, w.y, fmaf(v.z, w.z, fmaf(v.w, w.w, s))));
            }
            sm.t[h][i] = s;
        }
        __syncthreads();
        if (tid < 2 * TB) y[(tid >> 5) * PY + jb + (tid & 31)] = sm.t[tid >> 5][tid & 31];
        for (int i = i0; i < P; i += THREADS) {
            if (i != i0) {
#pragma unroll
                for (int c = 0; c < TB; ++c) l[c] = L[(size_t)(jb + c) * ld + i];
            }
            float a = y[i], bq = y[PY + i];
#pragma unroll
            for (int c = 0; c < TB; ++c) {
                a = fmaf(-l[c], sm.t[0][c], a);
                bq = fmaf(-l[c], sm.t[1][c], bq);
            }
            y[i] = a;
            y[PY + i] = bq;
        }
    }
    // backward: x_b = X_b^T y_b, then the rows above lose L_b^T x_b.  (The last forward step fetched
    // the last inverse again, into the buffer of step nblk.)
    for (int q = 0; q < nblk; ++q) {
        const int b = nblk - 1 - q, jb = b * TB, nb = min(TB, P - jb);
        const int s_in = (nblk + q) & 1;
        float l[TB];
        auto load_l = [&](int j) {
            const float* Lj = L + (size_t)j * ld + jb;
#pragma unroll
            for (int k = 0; k < TB / 4; ++k) {
                // rows past P of the last block hold nothing
                const float4 v = 4 * k < nb ? ld4(Lj + 4 * k) : make_float4(0.f, 0.f, 0.f, 0.f);
                l[4 * k] = v.x;
                l[4 * k + 1] = 4 * k + 1 < nb ? v.y : 0.f;
                l[4 * k + 2] = 4 * k + 2 < nb ? v.z : 0.f;
                l[4 * k + 3] = 4 * k + 3 < nb ? v.w : 0.f;
            }
        };
        if (tid < jb) load_l(tid);
        cp_wait<0>();
        __syncthreads();
        if (b > 0) fetch(b - 1, (nblk + q + 1) & 1);
        if (tid < 2 * TB) {
            const int h = tid >> 5, i = tid & 31;
            const float* Xc = xb + s_in * XS + i;
            float s = 0.f;
#pragma unroll 8
            for (int k = 0; k < TB; ++k) s = fmaf(Xc[k * (TB + 4)], y[h * PY + jb + k], s);
            sm.t[h][i] = s;
        }
        __syncthreads();
        if (tid < 2 * TB) y[(tid >> 5) * PY + jb + (tid & 31)] = sm.t[tid >> 5][tid & 31];
        for (int j = tid; j < jb; j += THREADS) {
            if (j != tid) load_l(j);
            float a = y[j], bq = y[PY + j];
#pragma unroll
            for (int c = 0; c < TB; ++c) {
                a = fmaf(-l[c], sm.t[0][c], a);
                bq = fmaf(-l[c], sm.t[1][c], bq);
            }
            y[j] = a;
            y[PY + j] = bq;
        }
    }
    cp_wait<0>();
    __syncthreads();
}

__global__ void __launch_bounds__(THREADS, 1) solve_ref_kernel(int P, double eps, const double* __restrict__ S,
                                                               const double2* __restrict__ D,
                                                               double2* __restrict__ delta,
                                                               double* __restrict__ shift_used,
                                                               double* __restrict__ Lws, double* __restrict__ xws,
                                                               int* __restrict__ flags) {
    extern __shared__ __align__(16) unsigned char smraw[];
    Smem& sm = *reinterpret_cast<Smem*>(smraw);
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), cn = (int)cl.num_blocks();
    const int t = blockIdx.x / cn, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nblk = (P + TB - 1) / TB, PY = nblk * TB;
    const size_t ld = ld_of(P), PP = (size_t)P * P;
    float* dsc = reinterpret_cast<float*>(smraw + sizeof(Smem));  // [PY] scales
    float* y = dsc + PY;                                         // [2][PY] right-hand sides of the FP32 solve
    int2* zq = reinterpret_cast<int2*>(y + 2 * PY);              // [PY] the last correction over d, whole numbers
    int* dsh = reinterpret_cast<int*>(zq + PY);                  // [PY] log2 of the scales
    const double* St = S + (size_t)t * PP;
    const double2* Dt = D + (size_t)t * P;
    // an odd P leaves the trajectory's scratch at 8 bytes past a multiple of 16
    float* L = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(Lws + (size_t)t * PP) + 15) & ~(uintptr_t)15);
    float* Xi = L + (size_t)P * ld;          // [nblk][TB][TB]
    double* gx = xws + (size_t)t * 4 * P;    // [2][P] x (CTA 0), then [2][P] r, shared by the cluster
    double* gr = gx + 2 * P;

    // scales; a diagonal entry that is not a positive normal number goes to FP64
    int bad = 0;
    for (int i = tid; i < PY; i += THREADS) {
        float s = 1.f;
        int sh = 0;
        if (i < P) {
            const double v = St[(size_t)i * P + i] + eps;
            if (v > 1e-30 && v < 1e30) sh = -((ilogb(v) + 1) >> 1);
            else bad = 1;
            s = scalbnf(1.f, sh);
        }
        dsc[i] = s;
        dsh[i] = sh;
    }
    bad = __syncthreads_or(bad);
    // a pivot closer than this to the threshold could stand for one below it in FP64: several times
    // the rounding of a sum of P products of entries at most sqrt(2)
    const float guard = 5.9604645e-8f * (16.f + 8.f * sqrtf((float)P));
    if (tid == 0) sm.flag = bad;
    __syncthreads();

    for (int b = 0; b < nblk && !bad; ++b) {
        const int jb = b * TB, nb = min(TB, P - jb);
        // ---- update of this CTA's row chunks: C[i][c] = d_i d_c A_ic - sum_k L_ik L_(jb+c)k
        const int rg = tid >> 3, cgp = tid & 7;  // rows 4 rg .. + 3, columns 4 cgp .. + 3
        for (int r0 = jb + RC * rank; r0 < P; r0 += RC * cn) {
            float acc[4][4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) acc[u][v] = 0.f;
            const int nk = jb / KC;  // KC divides TB
            auto stage = [&](int s, int k0) {
                // KC columns x 256 rows (64 pieces of 16 bytes each), KC x 32 rows of the block
#pragma unroll
                for (int e = tid; e < KC * (RC / 4); e += THREADS) {
                    const int kk = e / (RC / 4), i4 = 4 * (e % (RC / 4));
                    const bool ok = r0 + i4 < P;  // the columns are padded to ld, a multiple of 4
                    cp16(&sm.As[s][kk][i4], L + (size_t)(k0 + kk) * ld + (ok ? r0 + i4 : 0), ok);
                }
                if (tid < KC * (TB / 4)) {
                    const int kk = tid / (TB / 4), c4 = 4 * (tid % (TB / 4));
                    const bool ok = jb + c4 < P;
                    cp16(&sm.Bs[s][kk][c4], L + (size_t)(k0 + kk) * ld + (ok ? jb + c4 : 0), ok);
                }
                cp_commit();
            };
            if (nk > 0) stage(0, 0);
            for (int kb = 0; kb < nk; ++kb) {
                if (kb + 1 < nk) {
                    stage((kb + 1) & 1, (kb + 1) * KC);
                    cp_wait<1>();
                } else {
                    cp_wait<0>();
                }
                __syncthreads();
#pragma unroll
                for (int kk = 0; kk < KC; ++kk) {
                    const float4 a = ld4(&sm.As[kb & 1][kk][4 * rg]), q = ld4(&sm.Bs[kb & 1][kk][4 * cgp]);
                    const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                    for (int u = 0; u < 4; ++u)
#pragma unroll
                        for (int v = 0; v < 4; ++v) acc[u][v] = fmaf(av[u], bv[v], acc[u][v]);
                }
                __syncthreads();
            }
            // S is symmetric: row jb + c of S read along i
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const int c = 4 * cgp + v, j = jb + c;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int i = r0 + 4 * rg + u;
                    if (i < P && j < P) {
                        float a = scaled_float(St[(size_t)j * P + i], dsh[i] + dsh[j]);
                        if (i == j) a = fmaf((float)eps * dsc[i], dsc[i], a);
                        const float x = a - acc[u][v];
                        if (r0 == jb && 4 * rg + u < TB) sm.Dg[4 * rg + u][c] = x;
                        L[(size_t)j * ld + i] = x;
                    } else if (r0 == jb && 4 * rg + u < TB) {
                        sm.Dg[4 * rg + u][c] = 4 * rg + u == c ? 1.f : 0.f;  // identity beyond P
                    }
                }
            }
        }
        __syncthreads();
        // ---- diagonal tile: factor and inverse by one warp of CTA 0
        if (rank == 0) {
            if (warp == 0) {
                // pivots: at least eps d^2 in exact arithmetic
                float dmin = 0.f;
                const int j = jb + lane;
                if (j < P) dmin = (float)(0.5 * eps) * dsc[j] * dsc[j];
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) dmin = fmaxf(dmin, __shfl_xor_sync(0xffffffffu, dmin, off));
                const bool ok = factor32(&sm.Dg[0][0], TB + 4, &sm.X[0][0], TB + 4, sm.scr, dmin + guard);
                if (lane == 0 && !ok) sm.flag = 1;
            }
            __syncthreads();
            for (int e = tid; e < TB * TB; e += THREADS) {
                const int i = e >> 5, c = e & 31;
                Xi[(size_t)b * TB * TB + e] = sm.X[i][c];
            }
            if (tid == 0) flags[t] = sm.flag;
        }
        __threadfence();
        cl.sync();
        if (*((volatile int*)flags + t)) {
            bad = 1;
            break;
        }
        // ---- panel: rows below the tile times the inverse (X from CTA 0), in place
        if (rank != 0)
            for (int e = tid; e < TB * TB; e += THREADS) sm.X[e >> 5][e & 31] = __ldcg(Xi + (size_t)b * TB * TB + e);
        __syncthreads();
        for (int r0 = jb + RC * rank; r0 < P; r0 += RC * cn) {
            const int i = r0 + (tid & (RC - 1)), half = tid / RC;  // 16 columns each
            float c[TB];
            if (i < P && i >= jb + nb) {
#pragma unroll
                for (int k = 0; k < TB; ++k) c[k] = L[(size_t)(jb + k) * ld + i];
            }
            __syncthreads();
            if (i < P && i >= jb + nb) {
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    const int cc = 16 * half + q;
                    float s = 0.f;
#pragma unroll
                    for (int k4 = 0; k4 < TB / 4; ++k4) {
                        const float4 v = ld4(&sm.X[cc][4 * k4]);
                        s = fmaf(c[4 * k4], v.x, s);
                        s = fmaf(c[4 * k4 + 1], v.y, s);
                        s = fmaf(c[4 * k4 + 2], v.z, s);
                        s = fmaf(c[4 * k4 + 3], v.w, s);
                    }
                    L[(size_t)(jb + cc) * ld + i] = s;
                }
            }
        }
        __threadfence();
        cl.sync();
    }

    if (bad) {
        if (rank == 0 && tid == 0) flags[t] = 1;
        return;  // uniform over the cluster
    }

    // ---- refinement
    if (rank == 0)
        for (int i = tid; i < 2 * P; i += THREADS) gx[i] = 0.0;
    // The two right-hand sides are systems of their own (they may differ by any factor): each has its
    // exponents, its last correction and its end.
    double prev[2] = {0.0, 0.0};  // CTA 0: the last correction's largest |x / d|
    int conv = 0;                 // CTA 0: bit h set once right-hand side h has converged
    bool done = false;
    for (int it = 0; it < MAX_ITER; ++it) {
        if (it == 0) {
            if (rank == 0)
                for (int i = tid; i < P; i += THREADS) {
                    gr[i] = Dt[i].x * (double)dsc[i];
                    gr[P + i] = Dt[i].y * (double)dsc[i];
                }
        } else {
            // r -= A dx, the correction from CTA 0
            const Smem* sm0 = cl.map_shared_rank(&sm, 0);
            const int ze[2] = {sm0->zex[0], sm0->zex[1]};
            if (rank != 0) {
                const int2* zq0 = cl.map_shared_rank(zq, 0);
                for (int i = tid; i < P; i += THREADS) zq[i] = zq0[i];
            }
            __syncthreads();
            for (int i = warp + WARPS * rank; i < P; i += WARPS * cn) {
                const double* Si = St + (size_t)i * P;
                const int shi = dsh[i];
                long long a[2][3];
#pragma unroll
                for (int h = 0; h < 2; ++h) a[h][0] = a[h][1] = a[h][2] = 0;
#pragma unroll 4
                for (int j = lane; j < P; j += 32) {
                    int sd[3];
                    digits_of(Si[j], shi + dsh[j], sd);
                    const int2 z = zq[j];
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        a[0][q] += (long long)sd[q] * z.x;
                        a[1][q] += (long long)sd[q] * z.y;
                    }
                }
#pragma unroll
                for (int off = 16; off > 0; off >>= 1)
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int q = 0; q < 3; ++q) a[h][q] += __shfl_xor_sync(0xffffffffu, a[h][q], off);
                if (lane < 2) {
                    // the sum, a whole number below 2^103, in two parts that convert exactly, largest first: the
                    // difference is small already
                    const int h = lane, zi = h ? zq[i].y : zq[i].x, zx = h ? ze[1] : ze[0];
                    const long long a0 = h ? a[1][0] : a[0][0], a1 = h ? a[1][1] : a[0][1], a2 = h ? a[1][2] : a[0][2];
                    const __int128 N = ((__int128)a0 << 42) + ((__int128)a1 << 21) + a2;
                    const long long hi = (long long)(N >> 53), lo = (long long)(N - ((__int128)hi << 53));
                    const double u = ldexp(1.0, zx), d = pow2(shi);
                    double r = fma(-(double)hi, u * 0x1.0p-7, __ldcg(gr + h * P + i));
                    r = fma(-(double)lo, u * 0x1.0p-60, r);
                    gr[h * P + i] = fma(-eps * d * d * u, (double)zi, r);
                }
            }
            __threadfence();
            cl.sync();
        }
        if (rank == 0) {
            int stop = 0;  // 1: converged, 2: left to FP64
            uint32_t km[2] = {0u, 0u};
            for (int i = tid; i < P; i += THREADS)
#pragma unroll
                for (int h = 0; h < 2; ++h) km[h] = max(km[h], mag_key(__ldcg(gr + h * P + i)));
            const uint2 kr = block_max2(km[0], km[1], sm.red);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const double rmax = key_value(h ? kr.y : kr.x);
                if (rmax == 0.0) conv |= 1 << h;
                // (the units of r, a 2^-167 of it at the end, stay normal numbers)
                else if (!(rmax < 0x1p800) || (it == 0 && rmax < 0x1p-800)) stop = 2;
            }
            if (stop == 0 && conv != 3) {
                int rex[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    rex[h] = key_exponent(h ? kr.y : kr.x);
                    const double up = conv & (1 << h) ? 0.0 : ldexp(1.0, -rex[h]);
                    for (int i = tid; i < PY; i += THREADS)
                        y[h * PY + i] = i < P ? (float)(__ldcg(gr + h * P + i) * up) : 0.f;
                }
                __syncthreads();
                solve32(P, PY, ld, L, Xi, y, sm);
                // the correction over d in units of 2^(ex - 27), 2^(ex - 1) <= its largest entry < 2^ex
                uint32_t kz[2] = {0u, 0u};  // (bits of a float's magnitude order like it)
                for (int i = tid; i < P; i += THREADS)
#pragma unroll
                    for (int h = 0; h < 2; ++h) kz[h] = max(kz[h], __float_as_uint(y[h * PY + i]) & 0x7FFFFFFFu);
                const uint2 kd = block_max2(kz[0], kz[1], sm.red);
                uint32_t kn[2] = {0u, 0u};
                double ndx[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint32_t k = h ? kd.y : kd.x;
                    const int ex = (int)(k >> 23) - 126;
                    const bool live = !(conv & (1 << h));
                    if (live && (ex < -60 || ex > 60)) stop = 2;  // (a correction of zeros, or not finite, among them)
                    const float up = live && stop == 0 ? __uint_as_float((uint32_t)(127 + 27 - ex) << 23) : 0.f;
                    const double unit = live ? ldexp(1.0, rex[h] + ex - 27) : 0.0;
                    ndx[h] = ldexp((double)__uint_as_float(k), rex[h]);
                    if (tid == 0) sm.zex[h] = rex[h] + ex - 27;
                    for (int i = tid; i < P; i += THREADS) {
                        const int z = __float2int_rn(y[h * PY + i] * up);
                        (h ? zq[i].y : zq[i].x) = z;
                        const double x = fma((double)z, unit * pow2(dsh[i]), __ldcg(gx + h * P + i));
                        kn[h] = max(kn[h], mag_key(x * pow2(-dsh[i])));
                        gx[h * P + i] = x;
                    }
                }
                const uint2 kx = block_max2(kn[0], kn[1], sm.red);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (conv & (1 << h)) continue;
                    const double nx = key_value(h ? kx.y : kx.x);  // largest |x / d|
                    // rate of the refinement from the last two corrections: what is left after this one is
                    // about rate * ndx.  Corrections at the rounding of x itself cannot shrink further.
                    if (!(ndx[h] < 1e300) || !(nx < 1e300) || (it > 0 && ndx[h] > 0.25 * prev[h] && ndx[h] > 1e-15 * nx))
                        stop = 2;
                    else if (it > 0 && (ndx[h] * fmax(ndx[h] / prev[h], 0x1.0p-22) <= 0x1.0p-54 * nx || ndx[h] <= 1e-15 * nx))
                        conv |= 1 << h;
                    prev[h] = ndx[h];
                }
            }
            if (stop == 0) stop = conv == 3 ? 1 : it == MAX_ITER - 1 ? 2 : 0;
            if (tid == 0) flags[t] = stop;
        }
        __threadfence();
        cl.sync();
        const int stop = *((volatile int*)flags + t);
        if (stop) {
            done = stop == 1;
            break;
        }
    }
    cl.sync();  // every CTA has read the flag
    if (rank != 0) return;
    if (tid == 0) flags[t] = done ? 0 : 1;
    if (!done) return;
    __syncthreads();
    for (int i = tid; i < P; i += THREADS) delta[(size_t)t * P + i] = make_double2(__ldcg(gx + i), __ldcg(gx + P + i));
    if (tid == 0 && shift_used) shift_used[t] = eps;
}

static_assert(sizeof(Smem) % 16 == 0, "the vectors behind Smem are read as float4");
static size_t smem_bytes(int P) {
    const size_t PY = (size_t)((P + TB - 1) / TB) * TB;
    return sizeof(Smem) + PY * 4 + 2 * PY * 4 + PY * 8 + PY * 4;
}

}  // namespace solref

// From where the FP32 factor and the tiles' inverses fit the P^2 doubles of scratch, to where the vectors of
// 40 bytes a parameter of its first form fitted a CTA's shared memory (those of now, 24 bytes, would up to about
// P = 5900: not measured).
bool solve_ref_ok(int P) { return P >= 48 && P <= 3520; }

// flags[t] = 0: solved; 1: left to the FP64 factorization.  Lws: P^2 doubles per trajectory, xws:
// 4 P doubles per trajectory.
cudaError_t launch_solve_ref(int ntraj, int P, double eps, const double* S, const double2* D, double2* delta,
                             double* shift_used, double* Lws, double* xws, int* flags, cudaStream_t s) {
    using namespace solref;
    const size_t smem = smem_bytes(P);
    cudaError_t e = cudaFuncSetAttribute(solve_ref_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // CTAs per trajectory: as many as the batch leaves SMs for, and no more than have a chunk
    int cn = 8;
    while (cn > 1 && (ntraj * cn > 152 || RC * (cn - 1) >= P)) cn /= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(ntraj * cn));
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cn;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, solve_ref_kernel, P, eps, S, D, delta, shift_used, Lws, xws, flags);
    if (e != cudaSuccess) return e;
    count_launch();
    return cudaGetLastError();
}

}  // namespace otvmc
