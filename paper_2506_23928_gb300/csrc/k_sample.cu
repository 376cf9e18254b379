// Metropolis sampling of |psi_theta(x)|^2 for the long-range Jastrow ansatz (Eq. 12),
// one thread per Markov chain (otVMC procedure paragraph: configurations are drawn by the
// Metropolis algorithm from the normalised |psi|^2).
//
// Proposal p of a chain flips the site drawn from Philox; it is accepted iff
// u < |psi(x')/psi(x)|^2 = exp(ell), ell = -4 sigma_j Re f_j, f_j = a_j + sum_k eta_jk sigma_k.
//
// A chain keeps only its spins.  The field of the proposed site is looked up: the sites are cut
// into groups of B consecutive ones, and a table in shared memory holds for every site j, group
// g and spin pattern m of the group the sum of Re eta_jk sigma_k over the group, as a 16-bit
// integer in units of sc_j = (largest sum of |Re eta_jk| over a group) / 32767.  A proposal adds
// L = ceil(N / B) of them (exactly, in int32): N / B reads, where fields kept per chain
// cost N reads of Re eta, N of the fields and N stores per accepted flip, with the lanes that
// rejected idle.  The looked-up ell is off by at most
//     4 (0.51 L sc_j + 12 2^-24 R_j),   R_j = |Re a_j| + sum_k |Re eta_jk|
// (rounding of each table entry to a unit, FP32 rounding of its terms and of the final
// conversion), so a guard band above that bound (plus the error of the FP32 logarithm: 2^-21.4
// absolute or 3 ulp) decides every proposal as FP64 would; proposals inside the band recompute
// ell in FP64 from theta.  Parameters that are not finite make the band NaN or infinite: FP64.
//
// Bound: the bank conflicts of the lookups (32 lanes at random sites: about 3.5 wavefronts per
// read) and the ~5 instructions per lookup.  B is the largest of 6, 5, 4, 3 whose table fits the
// 227 KB of shared memory (N <= 102, 133, 168, 200), because the reads per proposal fall as
// 1 / B; the sites' tables are skewed by one bank each so that polarised configurations (equal
// patterns, different sites) spread over the banks as well.  Measured: 128 x 8192 chains of 100
// sites, 2 sweeps, 1.90 ms (fields per chain in shared memory: 19.8 ms); 256 x 4096 chains of 64
// sites, 1.0 ms (fields in registers: 2.36 ms).
#include "common.cuh"

namespace otvmc {

__host__ __device__ __forceinline__ int pair_index(int lo, int hi, int n) {
    return lo * n - lo * (lo + 1) / 2 + (hi - lo - 1);
}

// The table of one site: L groups of 2^B entries of 16 bits, and one spare word, which skews the
// banks of the sites (a group's row is a multiple of four words long).
__host__ __device__ constexpr int samp_row(int B) { return 2 << B; }
__host__ __device__ constexpr int samp_site(int B, int L) { return L * samp_row(B) + 4; }
__host__ __device__ constexpr int samp_gpr(int B) { return 32 / B; }  // groups per 32-bit register
inline size_t samp_smem(int B, int n) {
    return (size_t)n * samp_site(B, (n + B - 1) / B) + 3 * (size_t)n * sizeof(float);
}
constexpr int SAMP_SMEM_MAX = 232448;  // 227 KB
constexpr int SAMP_THREADS = 1024;

// NF: registers whose groups are all in use; one more holds the last L - NF * (groups per
// register) groups (rem < groups per register, possibly none).
template <int B, int NF>
__global__ void __launch_bounds__(SAMP_THREADS, 1) sample_jastrow_kernel(
    const double2* __restrict__ theta, int P, int n, int W, int ns, int n_sweep, uint32_t k0, uint32_t k1,
    uint32_t evtag, int traj0, uint64_t* __restrict__ spins, unsigned long long* __restrict__ accepted) {
    constexpr int GP = samp_gpr(B), RB = GP * B, NR = NF + 1, ROW = samp_row(B), M = 1 << B;
    extern __shared__ __align__(16) unsigned char smp[];
    const int t = blockIdx.y, TPB = blockDim.x;
    const int L = (n + B - 1) / B;
    float* ca = reinterpret_cast<float*>(smp);  // [n] Re a_j
    float* csc = ca + n;                        // [n] unit of the table's entries of site j
    float* cg = csc + n;                        // [n] guard band, without the logarithm's part
    unsigned char* tab = smp + 3 * (size_t)n * sizeof(float);  // [n][L] rows
    const double2* th = theta + (size_t)t * P;

    // per site: largest group sum of |Re eta|, R_j (a thread per site and group)
    const int L1 = L * n;
    for (int j = threadIdx.x; j < n; j += TPB) csc[j] = cg[j] = 0.f;
    __syncthreads();
#pragma unroll 2
    for (int e = threadIdx.x; e < L1; e += TPB) {
        const int g = e / n, j = e - g * n;
        float q = 0.f;
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const int k = g * B + b;
            if (k < n && k != j) q += fabsf((float)th[n + pair_index(min(j, k), max(j, k), n)].x);
        }
        // (non-negative floats order as their bits; a NaN is the largest of them)
        atomicMax(reinterpret_cast<int*>(csc + j), __float_as_int(q));
        atomicAdd(cg + j, q);
    }
    __syncthreads();
    for (int j = threadIdx.x; j < n; j += TPB) {
        const float a = (float)th[j].x, mx = csc[j];
        const float sc = mx * (1.000001f / 32767.f), R = (cg[j] + fabsf(a)) * 1.00001f;
        const bool bad = !isfinite(R);
        ca[j] = a;
        csc[j] = bad ? 0.f : sc;
        // 4.4 = 4 with a tenth to spare; 12 2^-24 R_j: the FP32 roundings
        cg[j] = bad ? INFINITY : 4.4f * (0.52f * (float)L * sc + 7.2e-7f * R) + 1e-6f;
    }
    __syncthreads();
    // the table, a (group, site) row per thread: 2^B sums out of two halves
    const int JS = samp_site(B, L);
    for (int e = threadIdx.x; e < L1; e += TPB) {
        const int g = e / n, j = e - g * n;
        float q[B];
        const float inv = csc[j] > 0.f ? 1.f / csc[j] : 0.f;
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const int k = g * B + b;
            q[b] = k < n && k != j ? (float)th[n + pair_index(min(j, k), max(j, k), n)].x : 0.f;
        }
        constexpr int BL = B / 2, BH = B - BL;
        float lo[1 << BL], hi[1 << BH];
#pragma unroll
        for (int m = 0; m < (1 << BL); ++m) {
            float s = 0.f;
#pragma unroll
            for (int b = 0; b < BL; ++b) s += ((m >> b) & 1) ? q[b] : -q[b];
            lo[m] = s;
        }
#pragma unroll
        for (int m = 0; m < (1 << BH); ++m) {
            float s = 0.f;
#pragma unroll
            for (int b = 0; b < BH; ++b) s += ((m >> b) & 1) ? q[BL + b] : -q[BL + b];
            hi[m] = s;
        }
        uint32_t* row = reinterpret_cast<uint32_t*>(tab + j * JS + g * ROW);
#pragma unroll
        for (int m = 0; m < M; m += 2) {
            const int x = __float2int_rn((lo[m & ((1 << BL) - 1)] + hi[m >> BL]) * inv);
            const int y = __float2int_rn((lo[(m + 1) & ((1 << BL) - 1)] + hi[(m + 1) >> BL]) * inv);
            row[m >> 1] = ((uint32_t)x & 0xFFFFu) | ((uint32_t)y << 16);
        }
    }
    __syncthreads();

    const int chain = blockIdx.x * TPB + threadIdx.x;
    if (chain >= ns) return;
    uint64_t* sp = spins + ((size_t)t * ns + chain) * W;
    // the spins, RB consecutive sites to a register (groups never straddle registers)
    uint32_t w[NR];
    {
        uint64_t wd[5];
#pragma unroll
        for (int i = 0; i < 4; ++i) wd[i] = i < W ? sp[i] : 0ull;
        wd[4] = 0ull;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const int o = r * RB, i = o >> 6, s = o & 63;
            uint64_t x = i < 4 ? wd[i < 4 ? i : 4] >> s : 0ull;
            if (s + RB > 64 && i < 3) x |= wd[i + 1] << (64 - s);
            w[r] = (uint32_t)x & (RB == 32 ? 0xFFFFFFFFu : (1u << RB) - 1u);
        }
    }
    const int rem = L - NF * GP;
    const int nprop = n_sweep * n;
    int m = 0;
    u32x4 draw = {0u, 0u, 0u, 0u};
    for (int p = 0; p < nprop; ++p) {
        if ((p & 1) == 0) draw = philox(u32x4{(uint32_t)(p / 2), (uint32_t)chain, (uint32_t)(traj0 + t), evtag}, k0, k1);
        const uint32_t wsite = (p & 1) ? draw.z : draw.x;
        const uint32_t wu = (p & 1) ? draw.w : draw.y;
        const int j = (int)__umulhi(wsite, (uint32_t)n);
        const unsigned char* row = tab + j * JS;
        int acc = 0;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
#pragma unroll
            for (int q = 0; q < GP; ++q)
                if (r < NF || q < rem)
                    acc += *reinterpret_cast<const int16_t*>(row + 2u * ((w[r] >> (q * B)) & (uint32_t)(M - 1)) +
                                                             (r * GP + q) * ROW);
        }
        const int jr = j / RB;
        const uint32_t bit = 1u << (j - jr * RB);
        uint32_t ws = w[0];
#pragma unroll
        for (int r = 1; r < NR; ++r) ws = jr == r ? w[r] : ws;
        const bool up = (ws & bit) != 0u;
        const float fj = fmaf((float)acc, csc[j], ca[j]);
        const float l32 = up ? -4.f * fj : 4.f * fj;
        // u = (wu + 1/2) 2^-32 in FP32 (relative error <= 2^-23, inside the guard band)
        const float lu = __logf(fmaf((float)wu, 0x1.0p-32f, 0x1.0p-33f));
        const float guard = fmaf(5e-7f, fabsf(lu), cg[j]);
        const float d = l32 - lu;
        bool take;
        if (d > guard) {
            take = true;
        } else if (d < -guard) {
            take = false;
        } else {
            double part = 0.0;
            for (int k = 0; k < n; ++k) {
                if (k == j) continue;
                const int kr = k / RB;
                uint32_t wk = w[0];
#pragma unroll
                for (int r = 1; r < NR; ++r) wk = kr == r ? w[r] : wk;
                const double x = th[n + pair_index(min(j, k), max(j, k), n)].x;
                part += ((wk >> (k - kr * RB)) & 1u) ? x : -x;
            }
            const double f = th[j].x + part;
            take = u01(wu) < exp(up ? -4.0 * f : 4.0 * f);
        }
        if (take) {
#pragma unroll
            for (int r = 0; r < NR; ++r) w[r] ^= jr == r ? bit : 0u;
            ++m;
        }
    }
    {
        uint64_t wd[5] = {0ull, 0ull, 0ull, 0ull, 0ull};
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const int o = r * RB, i = o >> 6, s = o & 63;
            if (i < 4) wd[i < 4 ? i : 4] |= (uint64_t)w[r] << s;
            if (s + RB > 64 && i < 3) wd[i + 1] |= (uint64_t)w[r] >> (64 - s);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (i < W) sp[i] = wd[i];
    }
    if (accepted != nullptr && m) atomicAdd(accepted + t, (unsigned long long)m);
}

using SampleFn = void (*)(const double2*, int, int, int, int, int, uint32_t, uint32_t, uint32_t, int, uint64_t*,
                          unsigned long long*);

// The kernel of table width B for L groups.
static SampleFn sample_fn(int B, int L) {
    const int nf = L / samp_gpr(B);
    if (B == 6) {
        constexpr SampleFn f[4] = {sample_jastrow_kernel<6, 0>, sample_jastrow_kernel<6, 1>,
                                   sample_jastrow_kernel<6, 2>, sample_jastrow_kernel<6, 3>};
        return f[nf];
    }
    if (B == 5) return nf == 3 ? sample_jastrow_kernel<5, 3> : sample_jastrow_kernel<5, 4>;
    if (B == 4) return nf == 4 ? sample_jastrow_kernel<4, 4> : sample_jastrow_kernel<4, 5>;
    return nf == 5 ? sample_jastrow_kernel<3, 5> : sample_jastrow_kernel<3, 6>;
}

cudaError_t launch_sample_jastrow(const otvmc_ansatz* an, const double2* theta, int ntraj, int traj0, int ns,
                                  int n_sweep, uint64_t seed, int64_t eval, uint64_t* spins,
                                  unsigned long long* accepted, int* status, cudaStream_t s) {
    ProfScope prof_(OTVMC_K_SAMPLE, s);
    (void)status;
    const int n = an->n, W = (n + 63) / 64;
    const uint32_t evtag = (TAG_SAMPLE << 28) | ((uint32_t)eval & 0x0FFFFFFFu);
    int B = 6;
    while (B > 3 && samp_smem(B, n) > SAMP_SMEM_MAX) --B;
    const size_t smem = samp_smem(B, n);
    const SampleFn fn = sample_fn(B, (n + B - 1) / B);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // 32 warps per SM: one CTA where the table takes more than half of the shared memory, else
    // two of 512; smaller CTAs while the batch leaves SMs without one
    int tpb = smem > 113 * 1024 ? 1024 : 512;
    while (tpb > 64 && (tpb / 2 >= ns || (tpb > 128 && (long long)ntraj * ((ns + tpb - 1) / tpb) < 152)))
        tpb /= 2;
    fn<<<dim3((ns + tpb - 1) / tpb, ntraj), tpb, smem, s>>>(theta, (int)an->P, n, W, ns, n_sweep, (uint32_t)seed,
                                                            (uint32_t)(seed >> 32), evtag, traj0, spins, accepted);
    count_launch();
    return cudaGetLastError();
}

}  // namespace otvmc
