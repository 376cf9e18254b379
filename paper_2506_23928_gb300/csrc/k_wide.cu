// Wide Jastrow chains on the mixed path: local estimators beyond 128 sites and pair moments beyond
// 64, where the tensor-core kernels end.  Both are sums over k of one coupling record per (k, j),
// taken in the same order and precision as est1_jastrow_kernel<true> and
// observables_kernel<float2, float, .>, so that every result is the same bit for bit.
//
// Bound: instruction issue and shared memory.  The kernels they replace were
// bound by the tables instead: eight samples a CTA read all N^2 entries of three 64-bit tables
// (0.6 MB at N = 160) from L2, and the observables read one 8-byte table entry from shared memory
// per term with one CTA of eight warps on an SM.  Here a CTA takes as many samples as its threads
// hold, records of 16 bytes (converted once per trajectory) arrive in chunks of 16 rows by
// asynchronous copies one chunk ahead, and a record in registers serves several samples.
// Estimators of 100 x 4096 samples of 160 sites: 8.7 -> 4.04 ms; observables of 64 x 8192 samples of
// 100 sites: 11.9 -> 4.43 ms (16.5 instructions a term of 32 lanes, padding among them, 72 % of the issue slots).
#include "common.cuh"

namespace otvmc {
namespace wide {

constexpr int KC = 16;             // rows of a staged chunk
constexpr int EST_Q = EST_SAMPLES_PER_THREAD;
constexpr int EST_G = KC / 4;      // groups of eight samples per CTA, each building one group's table
constexpr int OBS_Q = 4;           // samples of a thread at a time
constexpr int OBS_VB = 2;          // blocks of 256 threads (in the partials' layout) per CTA

// The estimators' records lie in the half of b.r that FP32 ratios leave free (16-byte aligned), the
// observables' where the FP64 path keeps exp(+-4 eta): no workspace grows.
inline size_t r_bytes(int ntraj, int ns, int n) { return ((size_t)ntraj * ns * n * 8 + 15) & ~(size_t)15; }

__device__ __forceinline__ void cp16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src));
}
__device__ __forceinline__ void cp8(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;"); }
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// ------------------------------------------------------------------------------- estimators
// FP32 copies of Re eta and J, a record per (k, j).
__global__ void __launch_bounds__(256) est_rec_kernel(int n, const long long* __restrict__ Qre,
                                                      const long long* __restrict__ QJ, float2* __restrict__ rec) {
    const int t = blockIdx.y, i = blockIdx.x * 256 + threadIdx.x;
    if (i >= n * n) return;
    const size_t o = (size_t)t * n * n + i;
    rec[o] = make_float2(fx_to_float(Qre[o]), fx_to_float(QJ[i]));
}

struct EstSmem {  // byte offsets
    int rec, ms, offs, sw, total;
    __host__ __device__ EstSmem(int n, int W, int S) {  // S samples
        const int nc = (n + KC - 1) / KC;
        rec = 4 * 16 * n * 8;                 // after the table [4][16][n], later the E_H partials
        ms = rec + 2 * KC * n * 8;            // records [2][KC][n]
        offs = ms + S * nc * KC * 4;          // sigma_k = +1 as 1.f or 0.f, [S][nc KC]
        sw = offs + S * nc * 16;              // table offsets of a chunk's four groups, [S][nc]
        total = sw + S * W * 8;               // spin words
    }
};

// Groups of NT threads, thread j of a group owning site j of the group's eight samples: the block of
// eight samples is est1_jastrow_kernel's CTA beyond 128 sites, with its partial of the site sums.
// The real and J fields take every k in order, fma(0 or 1, entry, sum); the imaginary field, whole
// numbers, takes four k at a time from a table of their 16 partial sums, built per chunk and shared
// by the CTA's samples.  7.0 instructions a term of 32 lanes in all (predicated additions: 10.5, bound by
// the half-rate integer pipe).
template <int MAXT>
__global__ void __launch_bounds__(MAXT, 1) est1_wide_kernel(
    int n, int W, int ns, int nblk, double h, const uint64_t* __restrict__ spins, const float2* __restrict__ rec,
    const long long* __restrict__ Qim, const long long* __restrict__ base_re, const long long* __restrict__ base_im,
    const long long* __restrict__ baseJ, float2* __restrict__ r_out, double2* __restrict__ EH_out,
    double2* __restrict__ part_r, double* __restrict__ part_s) {
    const int NT = ((n + 31) / 32) * 32, t = blockIdx.y;
    constexpr int G = EST_G;
    const int g = threadIdx.x / NT, j = threadIdx.x % NT, blk = blockIdx.x * G + g;
    const bool active = j < n && blk < nblk;
    const int nc = (n + KC - 1) / KC, S = G * EST_Q;
    const EstSmem lay(n, W, S);
    extern __shared__ __align__(16) unsigned char smraw[];
    long long* tab = reinterpret_cast<long long*>(smraw);
    float2* recs = reinterpret_cast<float2*>(smraw + lay.rec);
    float* ms = reinterpret_cast<float*>(smraw + lay.ms);
    int* offs = reinterpret_cast<int*>(smraw + lay.offs);
    uint64_t* sw = reinterpret_cast<uint64_t*>(smraw + lay.sw);
    double2* ered = reinterpret_cast<double2*>(smraw);  // [S][NT / 32]
    const int s_first = blockIdx.x * S;
    const float2* rt = rec + (size_t)t * n * n;
    const long long* qt = Qim + (size_t)t * n * n + j;
    auto stage = [&](int c) {
        float2* dst = recs + (c & 1) * KC * n;
        const int cnt = min(KC, n - c * KC) * n;
        for (int i = threadIdx.x; i < KC * n; i += blockDim.x) {
            if (i < cnt) cp8(dst + i, rt + (size_t)c * KC * n + i);
            else dst[i] = make_float2(0.f, 0.f);
        }
        cp_commit();
    };
    long long q4[4] = {0, 0, 0, 0};  // Im of four rows of the next chunk
    auto fetch = [&](int c) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int k = c * KC + 4 * g + u;
            q4[u] = k < n ? qt[(size_t)k * n] : 0;
        }
    };
    const bool builds = j < n;
    stage(0);
    if (builds) fetch(0);
    for (int i = threadIdx.x; i < S * W; i += blockDim.x) {
        const int s = s_first + i / W;
        sw[i] = s < ns ? spins[((size_t)t * ns + s) * W + i % W] : 0ull;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < S * nc * KC; i += blockDim.x) {
        const int s = i / (nc * KC), k = i % (nc * KC);
        ms[i] = k < n && (sw[s * W + (k >> 6)] >> (k & 63)) & 1ull ? 1.f : 0.f;
    }
    for (int i = threadIdx.x; i < S * nc * 4; i += blockDim.x) {
        const int s = i / (nc * 4), c = i / 4 % nc, q = i & 3;
        offs[i] = (16 * q + ((int)(sw[s * W + (c >> 2)] >> (KC * (c & 3) + 4 * q)) & 15)) * n * 8;
    }
    float ar[EST_Q], aj[EST_Q];
    long long ai[EST_Q];
#pragma unroll
    for (int q = 0; q < EST_Q; ++q) {
        ar[q] = aj[q] = 0.f;
        ai[q] = 0;
    }
    const uint64_t* sg = sw + g * EST_Q * W;
    const float* mg = ms + g * EST_Q * nc * KC;
    const int4* og = reinterpret_cast<const int4*>(offs) + g * EST_Q * nc;
    const unsigned char* tj = smraw + 8 * j;
    for (int c = 0; c < nc; ++c) {
        cp_wait_all();
        __syncthreads();  // the records are here; the table and the other buffer have been read
        if (builds) {
            long long* tb = tab + (size_t)16 * g * n + j;
            const long long s01 = q4[0] + q4[1], s23 = q4[2] + q4[3];
#pragma unroll
            for (int p = 0; p < 16; ++p) {
                const long long lo = (p & 3) == 3 ? s01 : (p & 1) ? q4[0] : (p & 2) ? q4[1] : 0;
                const long long hi = (p & 12) == 12 ? s23 : (p & 4) ? q4[2] : (p & 8) ? q4[3] : 0;
                tb[p * n] = lo + hi;
            }
            if (c + 1 < nc) fetch(c + 1);
        }
        if (c + 1 < nc) stage(c + 1);
        __syncthreads();
        if (!active) continue;
#pragma unroll
        for (int q = 0; q < EST_Q; ++q) {
            const int4 o = og[q * nc + c];
            ai[q] += (*reinterpret_cast<const long long*>(tj + o.x) + *reinterpret_cast<const long long*>(tj + o.y)) +
                     (*reinterpret_cast<const long long*>(tj + o.z) + *reinterpret_cast<const long long*>(tj + o.w));
        }
        const float2* rc = recs + (c & 1) * KC * n + j;
        const float* mc = mg + c * KC;
#pragma unroll
        for (int k4 = 0; k4 < KC; k4 += 4) {
            float2 e[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) e[u] = rc[(k4 + u) * n];
#pragma unroll
            for (int q = 0; q < EST_Q; ++q) {
                const float4 m = *reinterpret_cast<const float4*>(mc + q * nc * KC + k4);
                const float mv[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    ar[q] = fmaf(mv[u], e[u].x, ar[q]);
                    aj[q] = fmaf(mv[u], e[u].y, aj[q]);
                }
            }
        }
    }
    __syncthreads();  // the table has been read
    const int lane = threadIdx.x & 31, nw = NT / 32;
    float2 pr = make_float2(0.f, 0.f);
    int ps = 0;
    const float bre = active ? fx_to_float(base_re[(size_t)t * n + j]) : 0.f;
    const float bj = active ? fx_to_float(baseJ[j]) : 0.f;
    const long long bim = active ? base_im[(size_t)t * n + j] : 0;
#pragma unroll
    for (int q = 0; q < EST_Q; ++q) {
        const int s = blk * EST_Q + q;
        float hrx = 0.f, hry = 0.f, fsg = 0.f;
        if (active && s < ns) {
            const bool up = (sg[q * W + (j >> 6)] >> (j & 63)) & 1ull;
            const float fre = fmaf(2.f, ar[q], bre);
            const long long fim = bim + 2 * ai[q];
            const float fj = fmaf(2.f, aj[q], bj);
            // log r_j = -2 sigma_j f_j
            const long long lim = up ? -2 * fim : 2 * fim;
            const float e = expf(up ? -2.f * fre : 2.f * fre);
            const int kq = __float2int_rn(fx_to_float(lim) * 0.15915494309189535f);
            const long long red = lim - (long long)kq * FX_TWO_PI;
            float sn, cs;
            sincosf(fx_to_float(red), &sn, &cs);
            const float2 r = make_float2(e * cs, e * sn);
            r_out[((size_t)t * ns + s) * n + j] = r;
            hrx = r.x;
            hry = r.y;
            fsg = up ? fj : -fj;  // sigma_j f^J_j
            pr.x += r.x;
            pr.y += r.y;
            ps += up ? 1 : -1;
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            hrx += __shfl_xor_sync(0xffffffffu, hrx, off);
            hry += __shfl_xor_sync(0xffffffffu, hry, off);
            fsg += __shfl_xor_sync(0xffffffffu, fsg, off);
        }
        if (lane == 0)
            ered[(g * EST_Q + q) * nw + j / 32] = make_double2(0.5 * (double)fsg + h * (double)hrx, h * (double)hry);
    }
    if (active) {
        const size_t o = ((size_t)t * nblk + blk) * n + j;
        part_r[o] = make_double2((double)pr.x, (double)pr.y);
        part_s[o] = (double)ps;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < G * EST_Q; i += blockDim.x) {
        const int s = s_first + i;
        if (s >= ns) break;
        double2 e = make_double2(0.0, 0.0);
        for (int w = 0; w < nw; ++w) {
            e.x += ered[i * nw + w].x;
            e.y += ered[i * nw + w].y;
        }
        EH_out[(size_t)t * ns + s] = e;
    }
}

// ------------------------------------------------------------------------------ observables
// {exp(4 eta_jk), exp(-4 eta_jk)} rounded to FP32 from FP64, (1, 1) on the diagonal.  A thread per
// pair j < k: rows j and n - 1 - j together hold n - 1 pairs.
__global__ void __launch_bounds__(128) obs_rec_kernel(const double2* __restrict__ theta, int P, int n,
                                                      float4* __restrict__ rec) {
    const int t = blockIdx.y;
    const double2* th = theta + (size_t)t * P + n;
    float4* out = rec + (size_t)t * n * n;
    const int i = blockIdx.x * 128 + threadIdx.x;
    if (i < n) out[i * n + i] = make_float4(1.f, 0.f, 1.f, 0.f);
    const int row = i / (n - 1), m = i % (n - 1);
    if (row >= (n + 1) / 2) return;
    const bool first = m < n - 1 - row;
    const int j = first ? row : n - 1 - row, k = j + 1 + (first ? m : m - (n - 1 - row));
    if (k >= n) return;
    const double2 e = th[j * n - j * (j + 1) / 2 + (k - j - 1)];
    double s, c;
    sincos(4.0 * e.y, &s, &c);
    const double ep = exp(4.0 * e.x), em = exp(-4.0 * e.x);
    const float4 v = make_float4((float)(ep * c), (float)(ep * s), (float)(em * c), (float)(em * -s));
    out[j * n + k] = v;
    out[k * n + j] = v;
}

// (x + i y) e with the roundings of the SIMT kernel's expression as the compiler contracts it there
__device__ __forceinline__ float2 cmul_fma(float x, float y, float2 e) {
    return make_float2(__fmaf_rn(x, e.x, -__fmul_rn(y, e.y)), __fmaf_rn(x, e.y, __fmul_rn(y, e.x)));
}

struct ObsPtrs {
    const uint64_t* spins;
    const float2* r;
    const float4* rec;
    double* part;
};

// Thread (block vb, group g, site j) takes the samples of observables_kernel's thread (g, j) of that
// block in the same order, four at a time; the partials are that kernel's.
__global__ void __launch_bounds__(256 * OBS_VB, 2) obs_wide_kernel(int n, int W, int ns, int spt, int nblk, ObsPtrs b) {
    const int NT = ((n + 31) / 32) * 32, SPP = 256 / NT, SB = SPP * spt;
    const int t = blockIdx.y, vb = threadIdx.x >> 8, lt = threadIdx.x & 255;
    const int j = lt % NT, g = lt / NT, blk = blockIdx.x * OBS_VB + vb;
    const bool in_group = g < SPP, active = in_group && j < n;
    const int gi = vb * SPP + g;
    extern __shared__ __align__(16) unsigned char smraw[];
    float4* tab = reinterpret_cast<float4*>(smraw);                        // [2][KC][n]
    float4* rs = tab + 2 * KC * n;                                         // [VB * SPP][OBS_Q][n]: r, sigma
    uint64_t* sw = reinterpret_cast<uint64_t*>(rs + OBS_VB * SPP * OBS_Q * n);  // [VB * SPP][OBS_Q][W]
    double* red = reinterpret_cast<double*>(smraw);                        // [VB][256][9] at the end
    const float4* rt = b.rec + (size_t)t * n * n;
    const int nc = (n + KC - 1) / KC;
    auto stage = [&](int c) {
        const int cnt = min(KC, n - c * KC) * n;
        for (int i = threadIdx.x; i < cnt; i += blockDim.x)
            cp16(tab + (c & 1) * KC * n + i, rt + (size_t)c * KC * n + i);
        cp_commit();
    };
    float acc[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) acc[i] = 0.f;
    float4* rg = rs + gi * OBS_Q * n;
    uint64_t* sg = sw + gi * OBS_Q * W;
    for (int q0 = 0; q0 < spt; q0 += OBS_Q) {
        const int s0 = blk * SB + g + q0 * SPP;  // samples s0 + i SPP
        __syncthreads();
        stage(0);
        if (active) {
#pragma unroll
            for (int i = 0; i < OBS_Q; ++i) {
                const int s = s0 + i * SPP;
                float4 v = make_float4(0.f, 0.f, 1.f, 0.f);
                if (s < ns) {
                    const float2 x = b.r[((size_t)t * ns + s) * n + j];
                    const bool up = (b.spins[((size_t)t * ns + s) * W + (j >> 6)] >> (j & 63)) & 1ull;
                    v = make_float4(x.x, x.y, up ? 1.f : -1.f, 0.f);
                }
                rg[i * n + j] = v;
            }
            if (j < OBS_Q * W) {
                const int s = s0 + j / W * SPP;
                sg[j] = s < ns ? b.spins[((size_t)t * ns + s) * W + j % W] : 0ull;
            }
        }
        float2 a2[OBS_Q], b2[OBS_Q];
        float sj[OBS_Q];  // s_j
#pragma unroll
        for (int i = 0; i < OBS_Q; ++i) a2[i] = b2[i] = make_float2(sj[i] = 0.f, 0.f);
        for (int c = 0; c < nc; ++c) {
            cp_wait_all();
            __syncthreads();  // chunk c (and the samples) are here, the other buffer has been read
            if (c + 1 < nc) stage(c + 1);
            if (!active) continue;
            if (c == 0)
#pragma unroll
                for (int i = 0; i < OBS_Q; ++i) sj[i] = rg[i * n + j].z;
            const float4* tc = tab + (c & 1) * KC * n + j;
            const float4* rc = rg + c * KC;
            auto term = [&](int kk) {
                const float4 E = tc[kk * n];
#pragma unroll
                for (int i = 0; i < OBS_Q; ++i) {
                    const float4 rk = rc[i * n + kk];
                    const bool same = rk.z == sj[i];
                    const float2 e = make_float2(same ? E.x : E.z, same ? E.y : E.w);
                    const float2 p = cmul_fma(rk.x, rk.y, e);
                    a2[i].x += p.x;
                    a2[i].y += p.y;
                    b2[i].x = fma(rk.z, p.x, b2[i].x);
                    b2[i].y = fma(rk.z, p.y, b2[i].y);
                }
            };
            const int rows = min(KC, n - c * KC);
            if (rows == KC) {
#pragma unroll
                for (int kk = 0; kk < KC; ++kk) term(kk);
            } else {
                for (int kk = 0; kk < rows; ++kk) term(kk);
            }
        }
        if (!active) continue;
#pragma unroll
        for (int i = 0; i < OBS_Q; ++i) {
            if (s0 + i * SPP >= ns) continue;
            int S = 0;
            for (int ww = 0; ww < W; ++ww) S += 2 * __popcll(sg[i * W + ww]);
            S -= n;
            const float4 rv = rg[i * n + j];
            const float2 rj = make_float2(rv.x, rv.y);
            float2 a = a2[i], bb = b2[i];
            // the diagonal's term r_j (and sigma_j r_j) taken out again
            a.x -= rj.x;
            a.y -= rj.y;
            bb.x -= sj[i] * rj.x;
            bb.y -= sj[i] * rj.y;
            const float rax = cmul_fma(rj.x, rj.y, a).x;
            const float2 rb = cmul_fma(rj.x, rj.y, bb);
            const float fs = sj[i], fS = (float)S - fs;
            acc[0] += rj.x;
            acc[1] += fs * rj.y;
            acc[2] += fs;
            acc[3] += rax;
            acc[4] -= fs * rb.x;
            if (j == 0) acc[5] += (float)(S * S - n);
            acc[6] += rb.y;
            acc[7] += rj.x * fS;
            acc[8] += fs * rj.y * fS;
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 9; ++i) red[threadIdx.x * 9 + i] = (double)acc[i];
    __syncthreads();
    if (blk < nblk) obs_block_sum(red + vb * 256 * 9, lt >> 5, 8, b.part + ((size_t)t * nblk + blk) * 9);
}

}  // namespace wide

bool est_wide_ok(const otvmc_ansatz* a, bool fp32, int ntraj, int ns) {
    if (!fp32 || a->kind != OTVMC_JASTROW || a->n <= ETC_MAX_N) return false;
    const size_t n = a->n;
    return wide::r_bytes(ntraj, ns, a->n) + (size_t)ntraj * n * n * 8 <= (size_t)ntraj * ns * n * 16;
}

cudaError_t launch_est1_wide(const otvmc_ansatz* a, const uint64_t* spins, int ntraj, int ns, const EvalBufs& b,
                             cudaStream_t s) {
    using namespace wide;
    ProfScope prof_(OTVMC_K_EST1, s);
    const int n = a->n, W = (n + 63) / 64, NT = ((n + 31) / 32) * 32, nblk = est_blocks(n, ns);
    const otvmc_model* m = a->model;
    float2* rec = reinterpret_cast<float2*>(reinterpret_cast<char*>(b.r) + r_bytes(ntraj, ns, n));
    est_rec_kernel<<<dim3((n * n + 255) / 256, ntraj), 256, 0, s>>>(n, b.Qre, m->QJ_d, rec);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    auto kern = NT <= 160 ? est1_wide_kernel<640> : NT <= 192 ? est1_wide_kernel<768> : est1_wide_kernel<896>;
    const size_t smem = EstSmem(n, W, EST_G * EST_Q).total;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<dim3((nblk + EST_G - 1) / EST_G, ntraj), EST_G * NT, smem, s>>>(
        n, W, ns, nblk, m->h, spins, rec, b.Qim, b.base_re, b.base_im, m->baseJ_d, reinterpret_cast<float2*>(b.r), b.EH,
        b.part_r, b.part_s);
    count_launch(2);
    return cudaGetLastError();
}

cudaError_t launch_obs_prep_wide(const otvmc_ansatz* a, const double2* theta, int ntraj, const EvalBufs& b,
                                 cudaStream_t s) {
    const int n = a->n, items = (n + 1) / 2 * (n - 1);
    wide::obs_rec_kernel<<<dim3((items + 127) / 128, ntraj), 128, 0, s>>>(theta, (int)a->P, n,
                                                                          reinterpret_cast<float4*>(b.Epm));
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_obs_wide(const otvmc_ansatz* a, const uint64_t* spins, int ntraj, int ns, const EvalBufs& b,
                            double* moments, cudaStream_t s) {
    using namespace wide;
    ProfScope prof_(OTVMC_K_OBS, s);
    const int n = a->n, W = (n + 63) / 64, NT = ((n + 31) / 32) * 32, SPP = 256 / NT, nblk = obs_blocks(n, ns);
    const size_t work = (size_t)2 * KC * n * 16 + (size_t)OBS_VB * SPP * OBS_Q * (n * 16 + W * 8);
    const size_t red = (size_t)OBS_VB * 256 * 9 * 8, smem = work > red ? work : red;
    cudaError_t e = cudaFuncSetAttribute(obs_wide_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const ObsPtrs p{spins, reinterpret_cast<const float2*>(b.r), reinterpret_cast<const float4*>(b.Epm), b.part_obs};
    obs_wide_kernel<<<dim3((nblk + OBS_VB - 1) / OBS_VB, ntraj), 256 * OBS_VB, smem, s>>>(
        n, W, ns, obs_samples_per_thread(), nblk, p);
    count_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_obs_final_n(n, ns, ntraj, nblk, b, moments, s);
}

}  // namespace otvmc
