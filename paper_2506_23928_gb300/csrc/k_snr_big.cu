// SNR-regularised solve in the eigenbasis of S (otVMC procedure paragraph) for P beyond the
// shared-memory Jacobi of k_snr.cu: the same filter,
//     S = V diag(lambda) V^T,  rho = V^T D,  Q_k(x) = (V^T O_c(x))_k v_c(x),
//     SNR_k = |rho_k| / sqrt(Var_x Q_k / ns),
//     f_k = 1 / (1 + (thr / SNR_k)^6) * 1 / (1 + (eps_svd lambda_max / lambda_k)^6),
//     delta = V diag(f_k / lambda_k) rho   (lambda_k <= 0 dropped),
// in five launches, all in FP64 or exact integers:
//   tri    Householder tridiagonalisation of a copy A of S: T = Q^T A Q, Q = H_0 H_1 ... H_{P-3},
//          H_k = I - tau_k v_k v_k^T acting on indices k+1 .. P-1 (v_k kept in column k of A); then
//          Q^T explicitly, as X = H_{P-3}, X <- X H_k for k = P-4 .. 0, each step touching only the
//          trailing block that H_k acts on.  One CTA per trajectory.
//   ql     the implicit QL iteration with the shift from the leading 2 x 2 block on T (d, e), every
//          plane rotation applied to the rows of X, so that at the end row k of X is the eigenvector
//          of eigenvalue d_k (X = V^T); eigenvalues to an absolute accuracy of a few eps ||S||, as a
//          dense symmetric eigensolver gives them.  One CTA per trajectory: one warp runs the scalar
//          recurrence of a sweep while eight apply the rotations of the sweep before.
//   mean   the means of O along the eigenvectors and of v.
//   pass   Q_k of every sample from whole numbers, summed with |Q_k|^2: P^2 products per sample in two 32-bit
//          digits of the eigenvectors, which run at 16 times the FP64 rate.
//   final  rho, the filter and the back-projection.
// Bound: FP64 at 2 multiply-adds per cycle and SM (tri: about 5/3 P^3 of them, ql: 2 per rotation and
// column, about 3 P^3), and in ql the chain of the recurrence (about 0.85 P^2 rotations).
// 100 trajectories of P = 249, 4096 samples, in one kernel with FP64 projections of every sample
// and the recurrence between the rotations: 321 ms; now 69.5 ms (tri
// 12, ql 47, mean and pass 9.9; ql at 1,700 cycles a rotation of its recurrence, 730 of its columns).
// A and X live in the caller's workspace (2 P^2 doubles per trajectory); the tridiagonal and then the eigenvalues
// pass from launch to launch in A's last rows (SnrScratch), the sample pass's sums in its first (PassScratch).
#include "common.cuh"
#include "rsqrt_pos.cuh"

namespace otvmc {

constexpr int SNRB_THREADS = 512;
constexpr int SNRB_WARPS = SNRB_THREADS / 32;
constexpr int SNRB_MAX_ITER = 60;        // QL iterations per eigenvalue before giving up
constexpr int SNRB_SMEM_BUDGET = 216 * 1024;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// Sums over the 32 lanes of eight values per lane in 9 additions (each step halves the values a lane
// keeps; additions are what an FP64 reduction costs); every lane gets all eight totals.
__device__ __forceinline__ void warp_sum8(double (&v)[8]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int h = 4, off = 16; h >= 1; h >>= 1, off >>= 1) {
        const bool up = lane & off;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (u < h) {
                const double send = up ? v[u] : v[u + h], keep = up ? v[u + h] : v[u];
                v[u] = keep + __shfl_xor_sync(0xffffffffu, send, off);
            }
    }
    double s = v[0];
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    // lane bits 4, 3, 2 hold the index of its total
#pragma unroll
    for (int u = 0; u < 8; ++u)
        v[u] = __shfl_sync(0xffffffffu, s, ((u >> 2) & 1) * 16 + ((u >> 1) & 1) * 8 + (u & 1) * 4);
}

__device__ __forceinline__ double pick8(const double (&v)[8], int i) {
    double r = v[0];
#pragma unroll
    for (int u = 1; u < 8; ++u) r = i == u ? v[u] : r;
    return r;
}

// Sum over a CTA of NW warps (every thread calls it; red holds NW doubles).
template <int NW>
__device__ double block_sum(double v, double* red) {
    v = warp_sum(v);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < NW; ++i) s += red[i];
    return s;
}

// d_k (then the eigenvalue) and e_k in the strict lower triangle of A, once the reflectors there are no
// longer needed: rows P - 1 and P - 2, what does not fit in row P - 3.
struct SnrScratch {
    double* A;
    int P;
    __device__ double& d(int k) const { return k < P - 1 ? A[(size_t)(P - 1) * P + k] : A[(size_t)(P - 3) * P]; }
    __device__ double& e(int k) const {
        return k < P - 2 ? A[(size_t)(P - 2) * P + k] : A[(size_t)(P - 3) * P + 1 + (k - (P - 2))];
    }
};

// ------------------------------------------------------------------- tridiagonalisation
__global__ void __launch_bounds__(SNRB_THREADS, 1) snr_tri_kernel(int P, const double* __restrict__ S,
                                                                  double* __restrict__ Aws, double* __restrict__ Xws) {
    const int t = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    extern __shared__ __align__(16) double sm[];
    double* d = sm;            // [P] diagonal
    double* e = d + P;         // [P] subdiagonal (e[i] couples i and i + 1)
    double* tau = e + P;       // [P]
    double* vb = tau + P;      // [P] reflector
    double* pb = vb + P;       // [P] p, then w
    double* red = pb + P;      // [SNRB_WARPS]
    const size_t PP = (size_t)P * P;
    double* A = Aws + (size_t)t * PP;
    double* X = Xws + (size_t)t * PP;
    const double* St = S + (size_t)t * PP;
    for (size_t i = tid; i < PP; i += blockDim.x) A[i] = St[i];
    __syncthreads();

    for (int k = 0; k + 2 < P; ++k) {
        const int m = P - 1 - k;
        double s2 = 0.0;
        for (int i = tid; i < m; i += blockDim.x) {
            const double x = A[(size_t)(k + 1 + i) * P + k];
            vb[i] = x;
            s2 += x * x;
        }
        const double nrm2 = block_sum<SNRB_WARPS>(s2, red);
        const double x0 = vb[0];
        const double alpha = nrm2 > 0.0 ? -copysign(sqrt(nrm2), x0) : 0.0;
        const double vtv = nrm2 - 2.0 * alpha * x0 + alpha * alpha;
        const double tk = vtv > 0.0 ? 2.0 / vtv : 0.0;
        __syncthreads();
        if (tid == 0) {
            vb[0] = x0 - alpha;
            d[k] = A[(size_t)k * P + k];
            e[k] = alpha;
            tau[k] = tk;
        }
        __syncthreads();
        if (tk != 0.0) {
            // p = tau B v (B the trailing block), eight rows per warp
            for (int i0 = 8 * warp; i0 < m; i0 += 8 * SNRB_WARPS) {
                const double* Bi = A + (size_t)(k + 1 + i0) * P + k + 1;
                const int nr = min(8, m - i0);
                double s[8] = {};
                for (int j = lane; j < m; j += 32) {
                    const double vj = vb[j];
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                        if (u < nr) s[u] = fma(Bi[(size_t)u * P + j], vj, s[u]);
                }
                warp_sum8(s);
                if (lane < nr) pb[i0 + lane] = tk * pick8(s, lane);
            }
            __syncthreads();
            double pv = 0.0;
            for (int i = tid; i < m; i += blockDim.x) pv += pb[i] * vb[i];
            const double K = 0.5 * tk * block_sum<SNRB_WARPS>(pv, red);
            for (int i = tid; i < m; i += blockDim.x) pb[i] -= K * vb[i];  // w = p - K v
            __syncthreads();
            // B -= v w^T + w v^T
            for (int i0 = 8 * warp; i0 < m; i0 += 8 * SNRB_WARPS) {
                double* Bi = A + (size_t)(k + 1 + i0) * P + k + 1;
                const int nr = min(8, m - i0);
                double vi[8], wi[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    vi[u] = u < nr ? -vb[i0 + u] : 0.0;
                    wi[u] = u < nr ? -pb[i0 + u] : 0.0;
                }
                for (int j = lane; j < m; j += 32) {
                    const double pj = pb[j], vj = vb[j];
                    double x[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) x[u] = u < nr ? Bi[(size_t)u * P + j] : 0.0;
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                        if (u < nr) Bi[(size_t)u * P + j] = fma(vi[u], pj, fma(wi[u], vj, x[u]));
                }
            }
        }
        __syncthreads();
        for (int i = tid; i < m; i += blockDim.x) A[(size_t)(k + 1 + i) * P + k] = vb[i];
        __syncthreads();
    }
    if (tid == 0) {
        if (P >= 2) {
            d[P - 2] = A[(size_t)(P - 2) * P + P - 2];
            e[P - 2] = A[(size_t)(P - 1) * P + P - 2];
        }
        d[P - 1] = A[(size_t)(P - 1) * P + P - 1];
        e[P - 1] = 0.0;
    }
    __syncthreads();

    // X = Q^T = H_{P-3} ... H_0, formed as X <- X H_k from the identity, k descending
    for (size_t i = tid; i < PP; i += blockDim.x) X[i] = (i / P == i % P) ? 1.0 : 0.0;
    __syncthreads();
    for (int k = P - 3; k >= 0; --k) {
        const double tk = tau[k];
        if (tk == 0.0) continue;  // uniform
        const int m = P - 1 - k;
        for (int i = tid; i < m; i += blockDim.x) vb[i] = A[(size_t)(k + 1 + i) * P + k];
        __syncthreads();
        // rows r >= k + 1 of X are the only ones with entries in columns k + 1 .. (X is the
        // identity elsewhere): u_r = (X v)_r, then X[r][k+1+b] -= tau u_r v_b, eight rows per warp
        for (int r0 = 8 * warp; r0 < m; r0 += 8 * SNRB_WARPS) {
            double* Xr = X + (size_t)(k + 1 + r0) * P + k + 1;
            const int nr = min(8, m - r0);
            double s[8] = {};
            for (int b = lane; b < m; b += 32) {
                const double v = vb[b];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (u < nr) s[u] = fma(Xr[(size_t)u * P + b], v, s[u]);
            }
            warp_sum8(s);
#pragma unroll
            for (int u = 0; u < 8; ++u) s[u] *= -tk;
            for (int b = lane; b < m; b += 32) {
                const double v = vb[b];
                double x[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) x[u] = u < nr ? Xr[(size_t)u * P + b] : 0.0;
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (u < nr) Xr[(size_t)u * P + b] = fma(s[u], v, x[u]);
            }
        }
        __syncthreads();
    }
    const SnrScratch sc{A, P};
    for (int i = tid; i < P; i += blockDim.x) {
        sc.d(i) = d[i];
        sc.e(i) = e[i];
    }
}

// --------------------------------------------------------------------------- QL iteration
// Twelve warps, of which warp 0 runs the recurrence and the nine that do not share its scheduler apply
// rotations, a column of X per thread: an FP64 instruction holds a scheduler's FP64 unit for 64
// cycles whatever the number of its lanes, so the recurrence costs what it counts in FP64
// instructions (19 a rotation, with comparisons, doublings and the first approximation of the
// reciprocal root in integers and FP32).
constexpr int QL_THREADS = 384;
constexpr int QL_APPLY = 288;

// 2 x for a normal x, and 0 for 0
__device__ __forceinline__ double twice(double x) {
    const int hw = __double2hiint(x);
    return (hw & 0x7FF00000) ? __hiloint2double(hw + 0x100000, __double2loint(x)) : x;
}

__global__ void __launch_bounds__(QL_THREADS, 1) snr_ql_kernel(int P, double* __restrict__ Aws,
                                                                  double* __restrict__ Xws, int* status) {
    const int t = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    extern __shared__ __align__(16) double sm[];
    double* d = sm;          // [P] diagonal, becoming the eigenvalues
    double* e = d + P;       // [P] subdiagonal
    double* cs2 = e + P;     // [2][P] rotations of two sweeps
    double* ss2 = cs2 + 2 * P;
    __shared__ int sm_m[2], sm_lo[2], sm_done[2], sm_fail;
    double* X = Xws + (size_t)t * P * P;
    const SnrScratch sc{Aws + (size_t)t * P * P, P};
    for (int i = tid; i < P; i += blockDim.x) {
        d[i] = sc.d(i);
        e[i] = sc.e(i);
    }
    if (tid == 0) sm_fail = 0;
    __syncthreads();
    // deflation: |e_m| below eps of the neighbouring diagonal entries, or below eps of the norm of
    // T (the accuracy the decomposition has anyway; without it a block of eigenvalues at the
    // rounding level of a rank-deficient S, where e stays at that level, never deflates)
    constexpr double EPS = 2.220446049250313e-16;
    double tol_abs = 0.0;
    int l = 0, iter = 0;
    if (warp == 0) {
        double tn = 0.0;
        for (int i = lane; i < P; i += 32) tn = fmax(tn, fabs(d[i]) + fabs(e[i]) + (i > 0 ? fabs(e[i - 1]) : 0.0));
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) tn = fmax(tn, __shfl_xor_sync(0xffffffffu, tn, off));
        tol_abs = EPS * tn;
    }
    for (int step = 0;; ++step) {
        if (warp == 0) {
            // the next unreduced block from l on, found by the warp; then one QL sweep by its lane 0
            const int buf = step & 1;
            double *cs = cs2 + buf * P, *ss = ss2 + buf * P;
            int m = l, done = 0, fail = 0;
            while (true) {
                if (l >= P) {
                    done = 1;
                    break;
                }
                for (m = l;; m += 32) {
                    const int i = m + lane;
                    bool small = i >= P - 1;
                    if (i < P - 1) small = fabs(e[i]) <= tol_abs || fabs(e[i]) <= EPS * (fabs(d[i]) + fabs(d[i + 1]));
                    const unsigned hit = __ballot_sync(0xffffffffu, small);
                    if (hit) {
                        m += __ffs((int)hit) - 1;
                        break;
                    }
                }
                if (m > l) break;
                ++l;  // d[l] converged
                iter = 0;
            }
            if (!done && ++iter > SNRB_MAX_ITER) done = fail = 1;
            int lo = m;
            if (!done && lane == 0) {
                double g = (d[l + 1] - d[l]) / (2.0 * e[l]);
                double r = hypot(g, 1.0);
                g = d[m] - d[l] + e[l] / (g + copysign(r, g));
                double s = 1.0, c = 1.0, p = 0.0;
                double ei = e[m - 1], di = d[m - 1], dn = d[m];  // e[i], d[i], d[i + 1]
                bool underflow = false;
                int i = m - 1;
                for (; i >= l; --i) {
                    const int ip = i > l ? i - 1 : l;
                    const double en = e[ip], dp = d[ip];  // ahead of the stores below
                    const double f = s * ei, b = c * ei;
                    const double h2 = fma(f, f, g * g);
                    double ir;
                    const int ex = __double2hiint(h2) >> 20;
                    if (ex > 64 && ex < 2000) {
                        ir = rsqrt_pos(h2);
                        r = h2 * ir;
                    } else {  // squares near or below the normal range (or not finite)
                        r = hypot(f, g);
                        ir = r > 0.0 ? 1.0 / r : 0.0;
                        if (r == 0.0) {  // deflation inside the sweep
                            e[i + 1] = 0.0;
                            d[i + 1] = dn - p;
                            e[m] = 0.0;
                            underflow = true;
                            break;
                        }
                    }
                    e[i + 1] = r;
                    s = f * ir;
                    c = g * ir;
                    g = dn - p;
                    r = fma(twice(c), b, (di - g) * s);
                    p = s * r;
                    d[i + 1] = g + p;
                    g = fma(c, r, -b);
                    cs[i] = c;
                    ss[i] = s;
                    ei = en;
                    dn = di;
                    di = dp;
                }
                lo = i + 1;  // rotations recorded for i = m - 1 .. lo
                if (!underflow) {
                    d[l] -= p;
                    e[l] = g;
                    e[m] = 0.0;
                }
            }
            if (lane == 0) {
                sm_m[buf] = m;
                sm_lo[buf] = lo;
                sm_done[buf] = done;
                if (fail) sm_fail = 1;
            }
            __syncwarp();
        } else if (step > 0 && (warp & 3) != 0) {
            // rotations i = m - 1 down to lo of the sweep before, on rows i and i + 1 of every column
            const int buf = (step - 1) & 1, m = sm_m[buf], lo = sm_lo[buf];
            const double *cs = cs2 + buf * P, *ss = ss2 + buf * P;
            if (m - 1 >= lo)
                for (int col = 32 * (3 * (warp >> 2) + (warp & 3) - 1) + lane; col < P; col += QL_APPLY) {
                    double zi1 = X[(size_t)m * P + col];  // row i + 1 for i = m - 1
                    // rows are loaded ahead of the rotations that use them (each row is stored only
                    // after it has been loaded)
                    constexpr int U = 16;
                    for (int i = m - 1; i >= lo; i -= U) {
                        const int nb = min(U, i - lo + 1);
                        double z[U];
#pragma unroll
                        for (int u = 0; u < U; ++u)
                            if (u < nb) z[u] = X[(size_t)(i - u) * P + col];
#pragma unroll
                        for (int u = 0; u < U; ++u)
                            if (u < nb) {
                                const double c = cs[i - u], s = ss[i - u];
                                X[(size_t)(i - u + 1) * P + col] = fma(s, z[u], c * zi1);
                                zi1 = fma(c, z[u], -s * zi1);
                            }
                    }
                    X[(size_t)lo * P + col] = zi1;
                }
        }
        // (the step that finds nothing left to do still applies the sweep before it; its flag is not
        // written again before the barrier of the next step but one)
        __syncthreads();
        if (sm_done[step & 1]) break;
    }
    if (sm_fail && tid == 0) record_error(status, OTVMC_ERR_NONFINITE, t);
    // eigenvalues; NaN marks a decomposition that did not converge
    for (int i = tid; i < P; i += blockDim.x) sc.d(i) = sm_fail ? NAN : d[i];
}

// ------------------------------------------------------------------------- sample pass
// y_k(x) = sum_i X_ki (O_i(x) - obar_i) for every eigenvector and sample, then the sums over x of Q_k = y_k v_c
// and |Q_k|^2.  O is a small whole number and X goes in as one (units of 2^-60, two digits of 30 bits), so
// that y is a sum of whole numbers, exact but for the rounding of X to 2^-61; the mean, subtracted from
// it in 128 bits, leaves what is small next to O as exact as the rest (directions of small variance, polarised
// samples), and the one rounding to FP64 comes after it.  The squares are summed as they are: a
// quadratic form v_k^T M v_k with M = sum_x |v_c|^2 O_c O_c^T takes half the products and, with P^3 FP64
// ones after them, 11.2 ms where this takes 9.9 (100 trajectories of P = 249, 4096 samples); it cancels as
// lambda_max / lambda_k, and its sums end at some 1e5 samples (ns^3 2^46 |O|^2 in 128 bits).
constexpr int WG = 64;         // tile of eigenvectors and of samples
constexpr int WK = 32;         // parameters per chunk
constexpr int WGP = WG + 4;    // row of the transposed digits
constexpr int NSPLIT_MAX = 16; // CTAs that share a tile's samples

// O_k of a sample with spin words word(0 .. W - 1): s_k, s_j s_l, or the sum over a tied group.
struct OShape {
    int n, W, P, nu;      // nu: parameters that are single spins or pairs
    int d, pbc;           // tied distances d + 1 + (k - nu)
    const int* pairs;     // pairs of the full Jastrow
    const int* grp_pair;  // tied ansatz: the free groups' pairs (nullptr: parameter n + q is pair q)
};
template <class Words>
__device__ __forceinline__ int o_value(const OShape& o, Words word, int k) {
    auto bit = [&](int j) { return (int)((word(j >> 6) >> (j & 63)) & 1ull); };
    if (k < o.n) return 2 * bit(k) - 1;
    if (k < o.nu) {
        const int p = o.grp_pair ? __ldg(o.grp_pair + k - o.n) : k - o.n;
        const int2 jl = __ldg(reinterpret_cast<const int2*>(o.pairs) + p);
        return 1 - 2 * (bit(jl.x) ^ bit(jl.y));
    }
    // all pairs at distance D: (pairs) - 2 (disagreeing ones), from the string shifted by D (rotated
    // for a ring, where each pair half way round is met twice)
    const int D = o.d + 1 + k - o.nu, m = o.pbc ? o.n : o.n - D;
    int dis = 0;
    for (int q = 0; q < o.W; ++q) {
        const int left = m - 64 * q;
        if (left <= 0) break;
        uint64_t u = 0ull;
        {
            const int b = 64 * q + D, i = b >> 6, r = b & 63;
            if (i < o.W) u = word(i) >> r;
            if (r && i + 1 < o.W) u |= word(i + 1) << (64 - r);
        }
        if (o.pbc) {  // bits n - D and up take the string's first bits
            const int b = 64 * q - (o.n - D), i = b >> 6, r = b & 63;  // (arithmetic shift: b may be negative)
            if (i >= 0 && i < o.W) u |= word(i) >> r;
            if (i + 1 >= 0 && i + 1 < o.W && r) u |= word(i + 1) << (64 - r);
        }
        const uint64_t mask = left >= 64 ? ~0ull : (1ull << left) - 1ull;
        dis += __popcll((word(q) ^ u) & mask);
    }
    return o.pbc && 2 * D == o.n ? m / 2 - dis : m - 2 * dis;
}

// x 2^60 to nearest, |x| < 2 (0 for what is not), in 64-bit integers
__device__ __forceinline__ long long fix60(double x) {
    const long long b = __double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7FF), sh = 1014 - e;  // mantissa 2^(e - 1075) 2^61
    const unsigned long long m = ((unsigned long long)b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
    unsigned long long v = sh >= 64 || sh < -9 ? 0ull : sh > 0 ? m >> sh : m << -sh;
    v = (v + 1) >> 1;
    return b < 0 ? -(long long)v : (long long)v;
}

__device__ __forceinline__ double to_double(__int128 v) {  // |v| < 2^116
    const long long hi = (long long)(v >> 53), lo = (long long)(v - ((__int128)hi << 53));
    // (hi may take more than 53 bits: then its conversion is the one rounding that counts)
    return fma((double)hi, 9007199254740992.0, (double)lo);
}

// What the sample pass takes from the kernel before it and leaves for the one after it, in A's place (the
// eigenvalues stay in its last rows): 4 P + 2 + 3 P NSPLIT_MAX of its (P - 3) P first doubles.
struct PassScratch {
    double* A;
    int P;
    __device__ long long* mean_lo() const { return reinterpret_cast<long long*>(A); }          // sum_i X_ki (obar_i -
    __device__ long long* mean_hi() const { return reinterpret_cast<long long*>(A) + P; }      // o_i) in 2^-60, 128 bits
    __device__ double* mean_f() const { return A + 2 * P; }                                    // the part of wild obar
    __device__ long long* o() const { return reinterpret_cast<long long*>(A) + 3 * P; }        // o_i
    __device__ double* vbar() const { return A + 4 * P; }
    __device__ double* part(int split) const { return A + 4 * P + 2 + (size_t)split * 3 * P; }  // [3][P]
};

// Means for the sample pass, 32 eigenvectors per CTA: o_i, the whole number nearest to obar_i (the pass sums
// O_i - o_i), and the rest of the mean along each eigenvector, from c_i / ns where obar_i = c_i / ns.
__global__ void __launch_bounds__(256) snr_mean_kernel(int P, int ns, const double2* __restrict__ v,
                                                       const double* __restrict__ obar, const double* __restrict__ Xws,
                                                       double* Aws) {
    const int t = blockIdx.x, k0 = blockIdx.y * 32, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    extern __shared__ __align__(16) double sm[];
    long long* rf = reinterpret_cast<long long*>(sm);  // [P] obar_i - o_i in units of 2^-60
    __shared__ double red[8];
    const PassScratch ps{Aws + (size_t)t * P * P, P};
    const double* ob = obar + (size_t)t * P;
    const double* X = Xws + (size_t)t * P * P;
    int wild = 0;
    for (int i = tid; i < P; i += 256) {
        const double b = ob[i];
        long long o = 0, r = 0;
        if (fabs(b) <= 256.0) {
            o = __double2ll_rn(b);
            const double c = rint(b * ns);
            // (c / ns rounded, times ns rounded, is within two roundings of c)
            const double f = fabs(b * ns - c) <= 0x1p-51 * fabs(c) ? (c - (double)o * ns) / ns : b - (double)o;
            r = __double2ll_rn(f * 0x1p60);
        } else {
            wild = 1;
        }
        rf[i] = r;
        if (k0 == 0) ps.o()[i] = o;
    }
    wild = __syncthreads_or(wild);
    for (int k = k0 + warp; k < min(P, k0 + 32); k += 8) {
        const double* Xk = X + (size_t)k * P;
        __int128 s = 0;
        double f = 0.0;
        for (int i = lane; i < P; i += 32) {
            s += (__int128)fix60(Xk[i]) * rf[i];
            if (wild && !(fabs(ob[i]) <= 256.0)) f = fma(Xk[i], ob[i], f);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const unsigned long long lo = __shfl_xor_sync(0xffffffffu, (unsigned long long)s, off);
            const long long hi = __shfl_xor_sync(0xffffffffu, (long long)(s >> 64), off);
            s += ((__int128)hi << 64) + lo;
            f += __shfl_xor_sync(0xffffffffu, f, off);
        }
        s = (s + ((__int128)1 << 59)) >> 60;
        if (lane == 0) {
            ps.mean_lo()[k] = (long long)s;
            ps.mean_hi()[k] = (long long)(s >> 64);
            ps.mean_f()[k] = f;
        }
    }
    if (k0 > 0) return;
    const double2* vt = v + (size_t)t * ns;
    double sx = 0.0, sy = 0.0;
    for (int x = tid; x < ns; x += 256) {
        sx += vt[x].x;
        sy += vt[x].y;
    }
    sx = block_sum<8>(sx, red);
    sy = block_sum<8>(sy, red);
    if (tid == 0) {
        ps.vbar()[0] = sx / ns;
        ps.vbar()[1] = sy / ns;
    }
}

// 64 eigenvectors by every nsplit-th tile of 64 samples per CTA, a thread 4 x 4 of a tile.
__global__ void __launch_bounds__(256, 2) snr_pass_kernel(OShape o, int ns, int nk, int nsplit,
                                                         const uint64_t* __restrict__ spins,
                                                         const double2* __restrict__ v,
                                                         const double* __restrict__ Xws, double* Aws) {
    const int t = blockIdx.x, k0 = (int)blockIdx.y % nk * WG, split = (int)blockIdx.y / nk;
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15, P = o.P, W = o.W;
    __shared__ __align__(16) int X1[WK][WGP], X0[WK][WGP];  // the digits of X, transposed
    __shared__ __align__(16) int Os[WK][WG];                // O - o
    __shared__ uint64_t sw[4][WG];
    __shared__ double vs[3][WG];                            // v_c and its square
    __shared__ long long ml[WG], mh[WG];
    __shared__ double mf[WG];
    const PassScratch ps{Aws + (size_t)t * P * P, P};
    const double* X = Xws + (size_t)t * P * P;
    const double2* vt = v + (size_t)t * ns;
    const uint64_t* sp = spins + (size_t)t * ns * W;
    if (tid < WG) {
        const int k = k0 + tid;
        ml[tid] = k < P ? ps.mean_lo()[k] : 0;
        mh[tid] = k < P ? ps.mean_hi()[k] : 0;
        mf[tid] = k < P ? ps.mean_f()[k] * 0x1p60 : 0.0;
    }
    const double vbx = ps.vbar()[0], vby = ps.vbar()[1];
    double q2[4] = {}, qx[4] = {}, qy[4] = {};
    for (int x0 = WG * split; x0 < ns; x0 += WG * nsplit) {
        __syncthreads();
        for (int e = tid; e < WG * W; e += 256) {
            const int x = e / W, q = e - x * W;
            sw[q][x] = x0 + x < ns ? sp[(size_t)(x0 + x) * W + q] : 0ull;
        }
        if (tid < WG) {
            const bool in = x0 + tid < ns;
            const double a = in ? vt[x0 + tid].x - vbx : 0.0, b = in ? vt[x0 + tid].y - vby : 0.0;
            vs[0][tid] = a;
            vs[1][tid] = b;
            vs[2][tid] = fma(a, a, b * b);
        }
        long long a1[4][4], a0[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) a1[a][b] = a0[a][b] = 0;
        for (int i0 = 0; i0 < P; i0 += WK) {
            __syncthreads();
#pragma unroll 2
            for (int e = tid; e < WK * WG; e += 256) {
                const int i = e & (WK - 1), r = e / WK;
                const long long q = k0 + r < P && i0 + i < P ? fix60(X[(size_t)(k0 + r) * P + i0 + i]) : 0ll;
                X1[i][r] = (int)(q >> 30);
                X0[i][r] = (int)(q & 0x3FFFFFFF);
            }
#pragma unroll 2
            for (int e = tid; e < WK * WG; e += 256) {
                const int x = e & (WG - 1), i = e / WG;  // a warp has one parameter
                int val = 0;
                if (i0 + i < P)
                    val = o_value(o, [&](int q) { return sw[q][x]; }, i0 + i) - (int)ps.o()[i0 + i];
                Os[i][x] = val;
            }
            __syncthreads();
#pragma unroll 4
            for (int i = 0; i < WK; ++i) {
                const int4 u1 = *reinterpret_cast<const int4*>(&X1[i][4 * ty]), u0 = *reinterpret_cast<const int4*>(&X0[i][4 * ty]);
                const int4 ov = *reinterpret_cast<const int4*>(&Os[i][4 * tx]);
                const int xr[4] = {u1.x, u1.y, u1.z, u1.w}, xl[4] = {u0.x, u0.y, u0.z, u0.w}, oc[4] = {ov.x, ov.y, ov.z, ov.w};
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        a1[a][b] += (long long)xr[a] * oc[b];
                        a0[a][b] += (long long)xl[a] * oc[b];
                    }
            }
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int r = 4 * ty + a;
            const __int128 mean = ((__int128)mh[r] << 64) + (unsigned long long)ml[r];
            const double f = mf[r];
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int x = 4 * tx + b;
                double y = to_double(((__int128)a1[a][b] << 30) + a0[a][b] - mean);  // in units of 2^-60
                if (f != 0.0) y -= f;
                qx[a] = fma(y, vs[0][x], qx[a]);
                qy[a] = fma(y, vs[1][x], qy[a]);
                q2[a] = fma(y * y, vs[2][x], q2[a]);
            }
        }
    }
    double* part = ps.part(split);
#pragma unroll
    for (int a = 0; a < 4; ++a) {
#pragma unroll
        for (int off = 8; off > 0; off >>= 1) {
            q2[a] += __shfl_xor_sync(0xffffffffu, q2[a], off);
            qx[a] += __shfl_xor_sync(0xffffffffu, qx[a], off);
            qy[a] += __shfl_xor_sync(0xffffffffu, qy[a], off);
        }
        const int k = k0 + 4 * ty + a;
        if (tx == 0 && k < P) {
            part[k] = q2[a] * 0x1p-120;
            part[P + k] = qx[a] * 0x1p-60;
            part[2 * P + k] = qy[a] * 0x1p-60;
        }
    }
}

// ------------------------------------------------------------------------------ the solution
__global__ void __launch_bounds__(256) snr_final_kernel(int P, int ns, int nsplit, const double2* __restrict__ D, double thr,
                                                        double eps_svd, double* Aws, const double* __restrict__ Xws,
                                                        double2* __restrict__ delta, double* __restrict__ lam_out) {
    const int t = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    extern __shared__ __align__(16) double sm[];
    double2* cf = reinterpret_cast<double2*>(sm);  // [P] filtered coefficients
    __shared__ double red[8];
    const double* X = Xws + (size_t)t * P * P;
    const SnrScratch sc{Aws + (size_t)t * P * P, P};  // eigenvalues
    const PassScratch ps{Aws + (size_t)t * P * P, P};
    double2* xt = delta + (size_t)t * P;
    const double2* Dt = D + (size_t)t * P;
    double lm = -INFINITY;
    int bad = 0;
    for (int k = tid; k < P; k += 256) {
        lm = fmax(lm, sc.d(k));
        bad |= isnan(sc.d(k));
    }
    bad = __syncthreads_or(bad);
    if (bad) {
        for (int k = tid; k < P; k += 256) xt[k] = make_double2(0.0, 0.0);
        return;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) lm = fmax(lm, __shfl_xor_sync(0xffffffffu, lm, off));
    if (lane == 0) red[warp] = lm;
    __syncthreads();
    lm = red[0];
    for (int i = 1; i < 8; ++i) lm = fmax(lm, red[i]);
    for (int k = warp; k < P; k += 8) {
        const double* Xk = X + (size_t)k * P;
        double ax = 0.0, ay = 0.0;
#pragma unroll 4
        for (int i = lane; i < P; i += 32) {
            ax += Xk[i] * Dt[i].x;
            ay += Xk[i] * Dt[i].y;
        }
        ax = warp_sum(ax);  // rho_k
        ay = warp_sum(ay);
        if (lane == 0) {
            double q2 = 0.0, qx = 0.0, qy = 0.0;
            for (int p = 0; p < nsplit; ++p) {
                const double* part = ps.part(p) + k;
                q2 += part[0];
                qx += part[P];
                qy += part[2 * P];
            }
            qx /= ns;
            qy /= ns;
            const double lam = sc.d(k);
            const double var = fmax(q2 / ns - (qx * qx + qy * qy), 0.0);
            const double snr = sqrt(ax * ax + ay * ay) / sqrt(var / ns + 1e-300);
            const double f_snr = 1.0 / (1.0 + pow(thr / snr, 6.0));
            const double f_svd = 1.0 / (1.0 + pow(eps_svd * lm / fmax(lam, 1e-300), 6.0));
            const double inv = lam > 0.0 ? f_snr * f_svd / fmax(lam, 1e-300) : 0.0;
            cf[k] = make_double2(inv * ax, inv * ay);
            if (lam_out) lam_out[(size_t)t * P + k] = lam;
        }
    }
    __syncthreads();
    for (int i = tid; i < P; i += 256) {
        double ax = 0.0, ay = 0.0;
#pragma unroll 4
        for (int k = 0; k < P; ++k) {
            const double xki = X[(size_t)k * P + i];
            ax += xki * cf[k].x;
            ay += xki * cf[k].y;
        }
        xt[i] = make_double2(ax, ay);
    }
}

size_t snr_big_ws_bytes(int ntraj, int P) {
    return (size_t)ntraj * 2 * (size_t)P * P * sizeof(double) + 256;
}

// (the bound of the one-kernel form, kept: about P = 3000)
bool snr_big_fits(int P) { return (SNRB_SMEM_BUDGET / 8 - 7 * P - 33) / P >= 2; }

cudaError_t launch_snr_big(const otvmc_ansatz* a, int ntraj, int ns, const uint64_t* spins, const double* S,
                           const double* obar, const double2* v, const double2* D, double thr, double eps_svd,
                           double2* delta, double* lam, void* ws, int* status, cudaStream_t s) {
    ProfScope prof_(OTVMC_K_SOLVE, s);
    const int P = (int)a->P, n = a->n;
    double* Aws = (double*)ws;
    double* Xws = Aws + (size_t)ntraj * P * P;
    const bool tied = a->kind == OTVMC_LJ;
    const OShape o{n, (n + 63) / 64, P, tied ? n + a->nfree : P, tied ? a->lj_d : 0, tied ? a->lj_pbc : 0,
                   tied ? a->full->pairs_d : a->pairs_d, tied ? a->grp_pair_d : nullptr};
    const int smem_tri = (5 * P + SNRB_WARPS) * (int)sizeof(double), smem_ql = 6 * P * (int)sizeof(double);
    cudaError_t e = cudaFuncSetAttribute(snr_tri_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_tri);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(snr_ql_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_ql);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(snr_final_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * P * (int)sizeof(double));
    if (e != cudaSuccess) return e;
    // (the trajectories along x: a grid's other dimensions end at 65535.)  The split of the samples does not
    // depend on the batch, so that neither do the sums.
    const int nk = (P + WG - 1) / WG, nx = (ns + WG - 1) / WG, nsplit = nx < NSPLIT_MAX ? nx : NSPLIT_MAX;
    snr_tri_kernel<<<ntraj, SNRB_THREADS, smem_tri, s>>>(P, S, Aws, Xws);
    snr_ql_kernel<<<ntraj, QL_THREADS, smem_ql, s>>>(P, Aws, Xws, status);
    snr_mean_kernel<<<dim3(ntraj, (P + 31) / 32), 256, P * (int)sizeof(long long), s>>>(P, ns, v, obar, Xws, Aws);
    snr_pass_kernel<<<dim3(ntraj, nk * nsplit), 256, 0, s>>>(o, ns, nk, nsplit, spins, v, Xws, Aws);
    snr_final_kernel<<<ntraj, 256, 2 * P * (int)sizeof(double), s>>>(P, ns, nsplit, D, thr, eps_svd, Aws, Xws, delta, lam);
    count_launch(5);
    return cudaGetLastError();
}

}  // namespace otvmc
