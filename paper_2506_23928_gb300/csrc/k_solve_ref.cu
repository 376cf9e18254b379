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
//   3. r = D - A x (rows over the warps of the cluster), dx from the FP32 factor (CTA 0), x += dx in
//      FP64, until the next correction, foretold from the last two, is below 2^-54 of x, for the real
//      and the imaginary system separately (a part 1e-8 of the other was left at 3e-11 of itself).  The
//      residual is taken from whole numbers: d S d and x / d as 63-bit fixed point in three signed
//      digits of 21 bits, the six leading digit products summed exactly in 64-bit integers.  Its
//      error is about 2^-61 |x|, below what an FP64 dot product leaves (2^-53 |S| |x|), so that the
//      solution is rounded from a value correct to a few 2^-53 wherever the refinement converges.
//
// Bound: the FP64 rate of these GPUs is 1/64 of the FP32 one.  The O(P^3) part runs in FP32; of the
// residuals' O(P^2), the integer form takes about 45 integer instructions an entry, half the time
// of two FP64 multiply-adds.
//
// 100 trajectories of P = 399: 0.80 ms (8.8 ms with the FP64 factorization, one CTA per
// trajectory); 8 of P = 528: 0.86 ms (15 ms).  Below P = 48 the factor and its inverses do not fit
// the scratch that the FP64 factorization needs anyway.
//
// A trajectory is left to the FP64 factorization (flag 1) when a pivot of the FP32 one is not
// clear of the shift test's threshold by the FP32 rounding (so that the decision to raise the
// shift is always taken in FP64), when an entry is not finite, or when the refinement does not
// converge.
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

// The three signed 21-bit digits of v (|v| < 2^62): v = d0 2^42 + d1 2^21 + d2.
__device__ __forceinline__ void digits(long long v, int (&d)[3]) {
    const int d2 = (int)((unsigned)v << 11) >> 11;
    v = (v - d2) >> 21;
    const int d1 = (int)((unsigned)v << 11) >> 11;
    d[2] = d2;
    d[1] = d1;
    d[0] = (int)((v - d1) >> 21);
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
    int* xd = reinterpret_cast<int*>(y + 2 * PY);                // [PY][2][3] digits of x / d
    int* dsh = xd + 6 * PY;                                      // [PY] log2 of the scales
    const double* St = S + (size_t)t * PP;
    const double2* Dt = D + (size_t)t * P;
    // an odd P leaves the trajectory's scratch at 8 bytes past a multiple of 16
    float* L = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(Lws + (size_t)t * PP) + 15) & ~(uintptr_t)15);
    float* Xi = L + (size_t)P * ld;          // [nblk][TB][TB]
    double* gx = xws + (size_t)t * 4 * P;    // [2][P] x, then [2][P] r, shared by the cluster
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
                // 16 columns x 256 rows (64 pieces of 16 bytes each), 16 x 32 rows of the block
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
            // digits of x / d in units of 2^(ex - 60), 2^(ex - 1) <= max |x / d| < 2^ex
            uint32_t km[2] = {0u, 0u};
            for (int i = tid; i < P; i += THREADS)
#pragma unroll
                for (int h = 0; h < 2; ++h) km[h] = max(km[h], mag_key(__ldcg(gx + h * P + i) * pow2(-dsh[i])));
            const uint2 kx = block_max2(km[0], km[1], sm.red);
            double unit[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int ex = key_exponent(h ? kx.y : kx.x);
                unit[h] = ldexp(1.0, ex - 120);
                for (int i = tid; i < PY; i += THREADS) {
                    int d[3] = {0, 0, 0};
                    if (i < P) digits(__double2ll_rn(ldexp(__ldcg(gx + h * P + i), 60 - ex - dsh[i])), d);
#pragma unroll
                    for (int q = 0; q < 3; ++q) xd[6 * i + 3 * h + q] = d[q];
                }
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
                    const int2* xj = reinterpret_cast<const int2*>(xd + 6 * j);
                    const int2 x0 = xj[0], x1 = xj[1], x2 = xj[2];
                    const int xv[2][3] = {{x0.x, x0.y, x1.x}, {x1.y, x2.x, x2.y}};
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        a[h][0] += (long long)sd[0] * xv[h][0];
                        a[h][1] += (long long)sd[0] * xv[h][1];
                        a[h][1] += (long long)sd[1] * xv[h][0];
                        a[h][2] += (long long)sd[0] * xv[h][2];
                        a[h][2] += (long long)sd[1] * xv[h][1];
                        a[h][2] += (long long)sd[2] * xv[h][0];
                    }
                }
#pragma unroll
                for (int off = 16; off > 0; off >>= 1)
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int q = 0; q < 3; ++q) a[h][q] += __shfl_xor_sync(0xffffffffu, a[h][q], off);
                if (lane < 2) {
                    // d_i r_i = d_i D_i - sum - eps d_i x_i, the largest terms first: the first
                    // difference is small already, and the digit sums (below 2^53) convert exactly
                    const int h = lane;
                    const double dd = (h ? Dt[i].y : Dt[i].x) * (double)dsc[i];
                    const long long a0 = h ? a[1][0] : a[0][0], a1 = h ? a[1][1] : a[0][1], a2 = h ? a[1][2] : a[0][2];
                    const double u = h ? unit[1] : unit[0];
                    double r = fma(-(double)a0, u * 0x1.0p84, dd);
                    r = fma(-eps * (double)dsc[i], __ldcg(gx + h * P + i), r);
                    r = fma(-(double)a1, u * 0x1.0p63, r);
                    gr[h * P + i] = fma(-(double)a2, u * 0x1.0p42, r);
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
                if (!(rmax < 1e300)) stop = 2;
            }
            if (stop == 0 && conv != 3) {
                double down[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int ex = key_exponent(h ? kr.y : kr.x);
                    const double up = conv & (1 << h) ? 0.0 : ldexp(1.0, -ex);
                    down[h] = ldexp(1.0, ex);
                    for (int i = tid; i < PY; i += THREADS)
                        y[h * PY + i] = i < P ? (float)(__ldcg(gr + h * P + i) * up) : 0.f;
                }
                __syncthreads();
                solve32(P, PY, ld, L, Xi, y, sm);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (conv & (1 << h)) continue;
                    uint32_t kd = 0u, kn = 0u;  // largest |dx / d| and |x / d|
                    for (int i = tid; i < P; i += THREADS) {
                        const double dx = (double)y[h * PY + i] * down[h];
                        const double x = fma(dx, pow2(dsh[i]), __ldcg(gx + h * P + i));
                        kd = max(kd, mag_key(dx));
                        kn = max(kn, mag_key(x * pow2(-dsh[i])));
                        gx[h * P + i] = x;
                    }
                    const uint2 k = block_max2(kd, kn, sm.red);
                    const double ndx = key_value(k.x), nx = key_value(k.y);
                    // rate of the refinement from the last two corrections: what is left after this one is
                    // about rate * ndx.  Corrections at the rounding of x itself cannot shrink further.
                    if (!(ndx < 1e300) || !(nx < 1e300) || (it > 0 && ndx > 0.25 * prev[h] && ndx > 1e-15 * nx))
                        stop = 2;
                    else if (it > 0 && (ndx * fmax(ndx / prev[h], 0x1.0p-22) <= 0x1.0p-54 * nx || ndx <= 1e-15 * nx))
                        conv |= 1 << h;
                    prev[h] = ndx;
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
    return sizeof(Smem) + PY * 4 + 2 * PY * 4 + 6 * PY * 4 + PY * 4;
}

}  // namespace solref

// P up to what the vectors of one trajectory leave of a CTA's shared memory (40 bytes a parameter),
// and from where the FP32 factor and the tiles' inverses fit the P^2 doubles of scratch.
bool solve_ref_ok(int P) { return P >= 48 && solref::smem_bytes(P) <= 220 * 1024; }

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
