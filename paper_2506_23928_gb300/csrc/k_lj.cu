// Partially inhomogeneous long-range Jastrow LJPHd / LJH (Eq. 12 and the paragraph after it).
//
// The two-body parameters are shared within groups of pairs: eta_jk = eta_g(j,k), every pair at
// distance <= d in a group of its own, all pairs at one larger distance in one group.  So
//     log psi = sum_i a_i s_i + sum_g eta_g sum_{(j,k) in g} s_j s_k,
//     O_{a_i} = s_i,   O_{eta_g} = sum_{(j,k) in g} s_j s_k   (an integer, |O| <= group size).
// Sampling, local estimators and observables only need the pair parameters eta_jk, so they run
// the full-Jastrow kernels on the expanded parameters theta_full (expand kernel).
//
// S and D come from one FP8 tensor-core Gram pass (k_gram_tc.cu), exactly.  A tied O reaches N in
// magnitude, more than E4M3 holds and more than FP32 sums of products hold exactly; it enters as two
// operand rows, O = 16 h + l with l in [-8, 7] and |h| <= 13 (N <= 200), so that every operand is a
// whole number of at most 16 and every sum of products stays below 2^24 up to LJ_TC_MAX_NS samples.
// A tied sum over all pairs at one distance D is (pairs) - 2 popcount(w xor (w shifted by D)), the
// rotation for a ring, so that no pair list is walked.  The digits of the quantised v and a row of
// ones ride along as in the full Jastrow's pass; S_ij = (ns G_ij - c_i c_j) / ns^2 and D are formed
// in 64- and 128-bit integers and rounded once.
// 100 trajectories of the 100-spin ring, P = 249, 4096 samples: 5.42 ms with the integer sums on the
// CUDA cores (full-Jastrow D folded over the groups, 16-bit O, integer Gram), which remain for more
// samples; 0.50 ms so (operand rows 0.28, Gram 0.09, S and D 0.10).
#include <algorithm>

#include "common.cuh"

namespace otvmc {
namespace lj {

constexpr int GT = 64;  // Gram tile (rows x columns)
constexpr int GK = 64;  // samples per chunk of the Gram kernel

// theta_full[t] = [a, eta_jk for j < k row-major] from theta[t] = [a, eta_g]
__global__ void expand_kernel(int n, int P, int Pf, const int* __restrict__ pair_grp,
                              const double2* __restrict__ theta, double2* __restrict__ theta_full) {
    const int t = blockIdx.y;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= Pf) return;
    const double2* th = theta + (size_t)t * P;
    theta_full[(size_t)t * Pf + k] = k < n ? th[k] : th[n + pair_grp[k - n]];
}

// obar[t][k] (and D, if given) of the tied parameters: the biases copied, each group the sum of
// its pairs' full-Jastrow values (in the fixed group order of grp_off / grp_pair).
__global__ void fold_kernel(int n, int P, int Pf, const int* __restrict__ grp_off, const int* __restrict__ grp_pair,
                            const double* __restrict__ obar_full, const double2* __restrict__ D_full,
                            double* __restrict__ obar, double2* __restrict__ D) {
    const int t = blockIdx.y;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= P) return;
    const double* of = obar_full + (size_t)t * Pf;
    const double2* df = D_full + (size_t)t * Pf;
    double o;
    double2 v;
    if (k < n) {
        o = of[k];
        v = df[k];
    } else {
        o = 0.0;
        v = make_double2(0.0, 0.0);
        for (int e = grp_off[k - n]; e < grp_off[k - n + 1]; ++e) {
            const int q = n + grp_pair[e];
            o += of[q];
            v.x += df[q].x;
            v.y += df[q].y;
        }
    }
    obar[(size_t)t * P + k] = o;
    if (D) D[(size_t)t * P + k] = v;
}

// O[t][k][x] as int16: s_k for k < n, sum over the group's pairs of s_j s_l for the rest.
// One thread per sample (coalesced stores along x), 16 rows per CTA row block.
__global__ void __launch_bounds__(256) obuild_kernel(int n, int W, int P, int ns, const int* __restrict__ grp_off,
                                                     const int* __restrict__ grp_pair, const int* __restrict__ pairs,
                                                     const uint64_t* __restrict__ spins, int16_t* __restrict__ O) {
    const int t = blockIdx.z, k0 = blockIdx.y * 16;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= ns) return;
    uint64_t w[4];
    const uint64_t* sp = spins + ((size_t)t * ns + x) * W;
#pragma unroll
    for (int q = 0; q < 4; ++q) w[q] = q < W ? sp[q] : 0ull;
    for (int k = k0; k < k0 + 16 && k < P; ++k) {
        int v;
        if (k < n) {
            v = ((w[k >> 6] >> (k & 63)) & 1ull) ? 1 : -1;
        } else {
            // s_j s_l = +1 when the bits agree; sum = size - 2 (number of disagreeing pairs)
            const int e0 = __ldg(grp_off + k - n), e1 = __ldg(grp_off + k - n + 1);
            int dis = 0;
            for (int e = e0; e < e1; ++e) {
                const int p = __ldg(grp_pair + e);
                const int j = __ldg(pairs + 2 * p), l = __ldg(pairs + 2 * p + 1);
                dis += (int)(((w[j >> 6] >> (j & 63)) ^ (w[l >> 6] >> (l & 63))) & 1ull);
            }
            v = (e1 - e0) - 2 * dis;
        }
        O[((size_t)t * P + k) * ns + x] = (int16_t)v;
    }
}

// Upper tiles I <= J (64 x 64) of G[t] = sum_x O_k(x) O_l(x) in int64: per chunk of 64 samples
// the products (|O| <= 256) are summed exactly in int32, then added to int64.  Thread (ty, tx)
// owns rows 4 ty .. 4 ty + 3 and columns 4 tx .. 4 tx + 3; the chunks sit in shared memory
// transposed (sample-major), so that a thread's four rows are one 8-byte load.
__global__ void __launch_bounds__(256) gram_int_kernel(int P, int ns, const int16_t* __restrict__ O,
                                                       long long* __restrict__ G) {
    const int t = blockIdx.y;
    int J = (int)((sqrtf(8.f * (float)blockIdx.x + 1.f) - 1.f) * 0.5f);
    while ((J + 1) * (J + 2) / 2 <= (int)blockIdx.x) ++J;
    while (J * (J + 1) / 2 > (int)blockIdx.x) --J;
    const int I = blockIdx.x - J * (J + 1) / 2;
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    __shared__ __align__(16) int16_t As[GK][GT + 4];
    __shared__ __align__(16) int16_t Bs[GK][GT + 4];
    const int16_t* Ot = O + (size_t)t * P * ns;
    const int r0 = I * GT, c0 = J * GT;
    long long acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0;
    for (int x0 = 0; x0 < ns; x0 += GK) {
        __syncthreads();
        for (int e = tid; e < GT * GK; e += 256) {
            const int r = e / GK, xs = e - r * GK, x = x0 + xs;
            As[xs][r] = (r0 + r < P && x < ns) ? Ot[(size_t)(r0 + r) * ns + x] : (int16_t)0;
            Bs[xs][r] = (c0 + r < P && x < ns) ? Ot[(size_t)(c0 + r) * ns + x] : (int16_t)0;
        }
        __syncthreads();
        int s[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) s[a][b] = 0;
#pragma unroll 8
        for (int xs = 0; xs < GK; ++xs) {
            const short4 av = *reinterpret_cast<const short4*>(&As[xs][4 * ty]);
            const short4 bv = *reinterpret_cast<const short4*>(&Bs[xs][4 * tx]);
            const int ar[4] = {av.x, av.y, av.z, av.w}, bc[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) s[a][b] += ar[a] * bc[b];
        }
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] += s[a][b];
    }
    long long* Gt = G + (size_t)t * P * P;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const int i = r0 + 4 * ty + a;
        if (i >= P) continue;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int j = c0 + 4 * tx + b;
            if (j < P && j >= i) Gt[(size_t)i * P + j] = acc[a][b];
        }
    }
}

// S[t] full symmetric FP64: S_ij = G_ij / ns - obar_i obar_j (G upper triangle)
__global__ void S_kernel(int P, int ns, const long long* __restrict__ G, const double* __restrict__ obar,
                         double* __restrict__ S) {
    const int t = blockIdx.y;
    const double inv = 1.0 / ns;
    const long long* Gt = G + (size_t)t * P * P;
    const double* ob = obar + (size_t)t * P;
    double* St = S + (size_t)t * P * P;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < (size_t)P * P;
         e += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(e / P), j = (int)(e - (size_t)i * P);
        const long long g = i <= j ? Gt[(size_t)i * P + j] : Gt[(size_t)j * P + i];
        St[e] = (double)g * inv - ob[i] * ob[j];
    }
}

// Largest |h| is 13: 13 * 13 * ns < 2^24
constexpr int LJ_TC_MAX_NS = 99200;
constexpr int OB = 32;  // rows of O per batch

// w, a string of 64 NW bits, shifted down (or UP) by D >= 0, zeros in
template <int NW, bool UP>
__device__ __forceinline__ void shift_bits(const uint64_t (&w)[NW], int D, uint64_t (&o)[NW]) {
    const int q = D >> 6, r = D & 63;
#pragma unroll
    for (int i = 0; i < NW; ++i) {
        uint64_t a = 0ull, b = 0ull;  // the word that lands on i, and the one whose bits come in
#pragma unroll
        for (int k = 0; k < NW; ++k) {
            if (k == (UP ? i - q : i + q)) a = w[k];
            if (k == (UP ? i - q - 1 : i + q + 1)) b = w[k];
        }
        if (r) o[i] = UP ? (a << r) | (b >> (64 - r)) : (a >> r) | (b << (64 - r));
        else o[i] = a;
    }
}
// E4M3 code of a whole number |d| <= 16
__device__ __forceinline__ uint32_t e4m3_int(int d) {
    if (d == 0) return 0u;
    const int a = d < 0 ? -d : d, e = 31 - __clz(a);
    return (d < 0 ? 0x80u : 0u) | ((uint32_t)(e + 7) << 3) | (uint32_t)(e <= 3 ? (a << (3 - e)) - 8 : (a >> (e - 3)) - 8);
}

// Operand rows of one trajectory: s_k (n), the free pairs (nf), then h and l of every tied distance
// (2 nt, interleaved), then the D_XROWS extra rows (digits of q, ones); K-major, pitch bytes a row,
// samples from ns on zero.  One thread per sample; OB rows at a time go through shared memory so
// that the stores are 16 bytes of consecutive samples.  Bound: about 20 instructions per tied sum.
template <int W>
__global__ void __launch_bounds__(256) obuild8_kernel(int n, int nf, int nt, int d, int pbc, int ns, int pitch,
                                                      const int* __restrict__ grp_pair, const int* __restrict__ pairs,
                                                      const uint64_t* __restrict__ spins,
                                                      const long long* __restrict__ qv, uint8_t* __restrict__ O) {
    __shared__ __align__(16) uint8_t tile[OB][256];
    const int t = blockIdx.y, tid = threadIdx.x, x = blockIdx.x * 256 + tid;
    const int PO = n + nf + 2 * nt, R = PO + D_XROWS;
    const bool live = x < ns;
    uint64_t w[W];
#pragma unroll
    for (int q = 0; q < W; ++q) w[q] = live ? spins[((size_t)t * ns + x) * W + q] : 0ull;
    // digit p of q + 8 (1 + 16 + ...) in base 16, less 8: the balanced digits
    constexpr unsigned long long BIAS = 0x8888888888888888ull;
    const unsigned long long q0 = live ? (unsigned long long)qv[((size_t)t * ns + x) * 2] + BIAS : BIAS;
    const unsigned long long q1 = live ? (unsigned long long)qv[((size_t)t * ns + x) * 2 + 1] + BIAS : BIAS;
    auto bit = [&](int j) -> uint32_t {
        uint64_t v = w[0];
#pragma unroll
        for (int q = 1; q < W; ++q) v = (j >> 6) == q ? w[q] : v;
        return (uint32_t)(v >> (j & 63)) & 1u;
    };
    uint8_t* Ot = O + (size_t)t * R * pitch;
    for (int b = blockIdx.z; b * OB < R; b += gridDim.z) {
        int val = 0;
        for (int r = 0; r < OB; ++r) {
            const int row = b * OB + r;  // uniform over the CTA
            uint32_t code = 0u;
            if (row < n) {
                code = bit(row) ? 0x38u : 0xB8u;
            } else if (row < n + nf) {
                const int p = __ldg(grp_pair + row - n);
                code = bit(__ldg(pairs + 2 * p)) == bit(__ldg(pairs + 2 * p + 1)) ? 0x38u : 0xB8u;
            } else if (row < PO) {
                const int g = (row - n - nf) >> 1, D = d + 1 + g;
                const bool low = (row - n - nf) & 1;
                if (!low || r == 0) {
                    // pairs (j, j + D), and for a ring (j, j + D - n): disagreeing bits
                    uint64_t u[W], v[W];
                    shift_bits<W, false>(w, D, u);
                    if (pbc) {
                        shift_bits<W, true>(w, n - D, v);
#pragma unroll
                        for (int q = 0; q < W; ++q) u[q] |= v[q];
                    }
                    const int m = pbc ? n : n - D;
                    int dis = 0;
#pragma unroll
                    for (int q = 0; q < W; ++q) {
                        const int left = m - 64 * q;
                        const uint64_t mask = left >= 64 ? ~0ull : left > 0 ? (1ull << left) - 1ull : 0ull;
                        dis += __popcll((w[q] ^ u[q]) & mask);
                    }
                    // half way round an even ring every pair is met twice
                    const bool twice = pbc && 2 * D == n;
                    val = twice ? m / 2 - dis : m - 2 * dis;
                }
                const int l = ((val + 8) & 15) - 8;
                code = e4m3_int(low ? l : (val - l) >> 4);
            } else if (row < R) {
                const int p = row - PO;
                code = p == 32 ? 0x38u : e4m3_int((int)(((p < 16 ? q0 : q1) >> (4 * (p & 15))) & 15ull) - 8);
            }
            tile[r][tid] = live ? (uint8_t)code : (uint8_t)0;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int r = (tid >> 4) + 16 * k, row = b * OB + r, xs = blockIdx.x * 256 + 16 * (tid & 15);
            if (row < R && xs < pitch)
                *reinterpret_cast<uint4*>(Ot + (size_t)row * pitch + xs) =
                    *reinterpret_cast<const uint4*>(&tile[r][16 * (tid & 15)]);
        }
        __syncthreads();
    }
}

// Operand row (the h row of a tied sum) of parameter k, and whether it is tied.
__device__ __forceinline__ int orow(int k, int nu, bool& tied) {
    tied = k >= nu;
    return tied ? nu + 2 * (k - nu) : k;
}
__device__ __forceinline__ long long count_of(const float* Xt, int row, bool tied) {
    const long long a = (long long)Xt[(size_t)row * D_XROWS + 32];
    return tied ? 16 * a + (long long)Xt[(size_t)(row + 1) * D_XROWS + 32] : a;
}

// obar and D from the side output of the Gram pass, X[t][row][D_XROWS]: sums over the samples of O
// against the digits of q and the ones.
__global__ void __launch_bounds__(128) D_kernel(int nu, int P, int PO, int ns, const float* __restrict__ X,
                                                const double* __restrict__ vinfo, const long long* __restrict__ qsum,
                                                double* __restrict__ obar, double2* __restrict__ D) {
    const int t = blockIdx.y, k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= P) return;
    const float* Xt = X + (size_t)t * PO * D_XROWS;
    bool tied;
    const int row = orow(k, nu, tied);
    const long long c = count_of(Xt, row, tied);
    double out[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        // sum_x O q, exactly (at most 200 2^60), then ns sum - c Q
        __int128 sum = 0;
#pragma unroll
        for (int p = 15; p >= 0; --p) {
            long long a = (long long)Xt[(size_t)row * D_XROWS + 16 * h + p];
            if (tied) a = 16 * a + (long long)Xt[(size_t)(row + 1) * D_XROWS + 16 * h + p];
            sum = sum * 16 + a;
        }
        const __int128 num = sum * ns - (__int128)c * qsum[2 * t + h];
        // in two parts of 64 bits: one rounding
        const long long hi = (long long)(num >> 53), lo = (long long)(num - ((__int128)hi << 53));
        out[h] = fma((double)hi, 9007199254740992.0, (double)lo);
    }
    const double inv = vinfo[4 * t + 2] / ((double)ns * (double)ns);
    obar[(size_t)t * P + k] = (double)c / ns;
    D[(size_t)t * P + k] = make_double2(out[0] * inv, out[1] * inv);
}

// S (full, FP64) from the Gram counts of the operand rows (upper triangle, FP32): one 32 x 32 tile
// of the upper triangle per CTA, mirrored through shared memory.
__global__ void __launch_bounds__(256) S8_kernel(int nu, int P, int PO, int ns, const float* __restrict__ G,
                                                 const float* __restrict__ X, double* __restrict__ S) {
    constexpr int B = 32;
    __shared__ double tile[B][B + 1];
    __shared__ long long ci[B], cj[B];
    const int t = blockIdx.y;
    int J = (int)((sqrtf(8.f * (float)blockIdx.x + 1.f) - 1.f) * 0.5f);
    while ((J + 1) * (J + 2) / 2 <= (int)blockIdx.x) ++J;
    while (J * (J + 1) / 2 > (int)blockIdx.x) --J;
    const int I = blockIdx.x - J * (J + 1) / 2;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const float* Xt = X + (size_t)t * PO * D_XROWS;
    if (threadIdx.x < 2 * B) {
        const int k = (threadIdx.x < B ? I : J) * B + tx;
        bool tied;
        const int row = orow(k, nu, tied);
        (threadIdx.x < B ? ci : cj)[tx] = k < P ? count_of(Xt, row, tied) : 0ll;
    }
    __syncthreads();
    const float* Gt = G + (size_t)t * PO * PO;
    double* St = S + (size_t)t * P * P;
    const double den = (double)ns * (double)ns;
#pragma unroll
    for (int r = ty; r < B; r += 8) {
        const int i = I * B + r, j = J * B + tx;
        double v = 0.0;
        if (i < P && j < P && i <= j) {
            bool ti, tj;
            const int a = orow(i, nu, ti), b = orow(j, nu, tj);
            const float* g = Gt + (size_t)a * PO + b;
            long long s = (long long)g[0];
            if (tj) s = 16 * s + (long long)g[1];
            if (ti) {
                // the l row of i against b and b + 1; on the diagonal (l, h) is (h, l)
                const long long lo = i == j ? (long long)g[1] : (long long)g[PO];
                s = 16 * s + (tj ? 16 * lo + (long long)g[PO + 1] : lo);
            }
            v = (double)(s * ns - ci[r] * cj[tx]) / den;
            St[(size_t)i * P + j] = v;
        }
        tile[r][tx] = v;
    }
    __syncthreads();
#pragma unroll
    for (int r = ty; r < B; r += 8) {
        const int j = J * B + r, i = I * B + tx;
        if (i < P && j < P && i < j) St[(size_t)j * P + i] = tile[tx][r];
    }
}

static size_t rup(size_t b) { return (b + 255) & ~(size_t)255; }
static int operand_rows(const otvmc_ansatz* a) { return a->n + a->nfree + 2 * (a->ngroups - a->nfree); }

}  // namespace lj

int lj_operand_rows(const otvmc_ansatz* a) { return lj::operand_rows(a); }

cudaError_t launch_lj_expand(const otvmc_ansatz* a, int ntraj, const double2* theta, double2* theta_full,
                             cudaStream_t s) {
    const int Pf = (int)a->full->P;
    ProfScope prof_(OTVMC_K_PREP, s);
    lj::expand_kernel<<<dim3((Pf + 255) / 256, ntraj), 256, 0, s>>>(a->n, (int)a->P, Pf, a->pair_grp_d, theta,
                                                                     theta_full);
    count_launch();
    return cudaGetLastError();
}

size_t lj_build_bytes(const otvmc_ansatz* a, int ntraj, int ns) {
    using lj::rup;
    const size_t T = (size_t)ntraj, P = (size_t)a->P, Pf = (size_t)a->full->P, PO = (size_t)lj::operand_rows(a);
    if (ns <= lj::LJ_TC_MAX_NS)
        return rup(T * (PO + D_XROWS) * o_pitch(ns)) + rup(T * PO * PO * 4) + rup(T * PO * D_XROWS * 4) + 256;
    return rup(T * Pf * 8) + rup(T * Pf * 16) + rup(T * P * ns * 2) + rup(T * P * P * 8) + 256;
}

static cudaError_t lj_build_tc(const otvmc_ansatz* a, const uint64_t* spins, int ntraj, int ns, const EvalBufs& b,
                               void* ws, double* S, double* obar, double2* D, int* status, cudaStream_t s) {
    using lj::rup;
    const int n = a->n, W = (n + 63) / 64, P = (int)a->P, nu = n + a->nfree, PO = lj::operand_rows(a);
    const int pitch = o_pitch(ns), R = PO + D_XROWS;
    uint8_t* O = (uint8_t*)ws;
    float* G = (float*)((char*)ws + rup((size_t)ntraj * R * pitch));
    float* X = (float*)((char*)G + rup((size_t)ntraj * PO * PO * 4));
    {
        ProfScope prof_(OTVMC_K_OBUILD, s);
        // the row batches over gridDim.z while the batch leaves SMs without work
        const int gx = (pitch + 255) / 256, nb = (R + lj::OB - 1) / lj::OB;
        const int gz = std::max(1, std::min(nb, (8 * 152 + gx * ntraj - 1) / (gx * ntraj)));
        const auto fn = W == 1 ? lj::obuild8_kernel<1> : W == 2 ? lj::obuild8_kernel<2>
                        : W == 3 ? lj::obuild8_kernel<3> : lj::obuild8_kernel<4>;
        fn<<<dim3(gx, ntraj, gz), 256, 0, s>>>(n, a->nfree, a->ngroups - a->nfree, a->lj_d, a->lj_pbc, ns, pitch,
                                               a->grp_pair_d, a->full->pairs_d, spins, b.qv, O);
        count_launch();
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    const cudaError_t e = launch_gram_tc(ntraj, PO, R, ns, pitch, O, a->tiles_d, a->ntiles, G, X, status, s);
    if (e != cudaSuccess) return e;
    ProfScope prof_(OTVMC_K_D, s);
    const int nt = (P + 31) / 32;
    lj::D_kernel<<<dim3((P + 127) / 128, ntraj), 128, 0, s>>>(nu, P, PO, ns, X, b.vinfo, b.qsum, obar, D);
    lj::S8_kernel<<<dim3(nt * (nt + 1) / 2, ntraj), 256, 0, s>>>(nu, P, PO, ns, G, X, S);
    count_launch(2);
    return cudaGetLastError();
}

// S (full FP64), obar and D of the tied parameters from the samples and the quantised v in b
// (vpart / vquant already run on b).  Beyond LJ_TC_MAX_NS samples on the CUDA cores: D and obar of the
// full Jastrow by the exact integer sums, folded over the groups; S from the exact integer Gram
// matrix of the tied O.
cudaError_t launch_lj_build(const otvmc_ansatz* a, const uint64_t* spins, int ntraj, int ns, const EvalBufs& b,
                            void* ws, double* S, double* obar, double2* D, int* status, cudaStream_t s) {
    using lj::rup;
    if (ns <= lj::LJ_TC_MAX_NS) return lj_build_tc(a, spins, ntraj, ns, b, ws, S, obar, D, status, s);
    const otvmc_ansatz* f = a->full;
    const int n = a->n, P = (int)a->P, Pf = (int)f->P, W = (n + 63) / 64;
    char* q = (char*)ws;
    auto take = [&](size_t bytes) {
        char* r = q;
        q += rup(bytes);
        return (void*)r;
    };
    double* obar_f = (double*)take((size_t)ntraj * Pf * 8);
    double2* D_f = (double2*)take((size_t)ntraj * Pf * 16);
    int16_t* O = (int16_t*)take((size_t)ntraj * P * ns * 2);
    long long* G = (long long*)take((size_t)ntraj * P * P * 8);
    cudaError_t e = launch_D_fixed_jastrow(f, spins, ntraj, ns, b, obar_f, D_f, s);
    if (e != cudaSuccess) return e;
    {
        ProfScope prof_(OTVMC_K_D, s);
        lj::fold_kernel<<<dim3((P + 255) / 256, ntraj), 256, 0, s>>>(n, P, Pf, a->grp_off_d, a->grp_pair_d, obar_f,
                                                                     D_f, obar, D);
        count_launch();
    }
    {
        ProfScope prof_(OTVMC_K_OBUILD, s);
        lj::obuild_kernel<<<dim3((ns + 255) / 256, (P + 15) / 16, ntraj), 256, 0, s>>>(
            n, W, P, ns, a->grp_off_d, a->grp_pair_d, f->pairs_d, spins, O);
        count_launch();
    }
    {
        ProfScope prof_(OTVMC_K_GRAM, s);
        const int nt = (P + lj::GT - 1) / lj::GT;
        lj::gram_int_kernel<<<dim3(nt * (nt + 1) / 2, ntraj), 256, 0, s>>>(P, ns, O, G);
        lj::S_kernel<<<dim3(256, ntraj), 256, 0, s>>>(P, ns, G, obar, S);
        count_launch(2);
    }
    return cudaGetLastError();
}

}  // namespace otvmc
