// Ritz pairs and thermal sums on the GPU (Section 2.2, Eqs. 5-7 with the Eq. 14 weights):
// device code shared by the entry points that run them.
#pragma once

#include <cooperative_groups.h>
#include <float.h>
#include <math.h>

#include <algorithm>

#include "common.cuh"

namespace ftlm {

constexpr int kThermoThreads = 256;

// ---------------------------------------------------------------- tridiagonal eigensolve (implicit QL, FP64)
//
// One thread per chain.  An FP64 instruction occupies its scheduler's FP64 pipe for about 64 cycles
// whether one lane or all 32 are active (measured: a warp of 1 to 32 chains takes the same time), so
// the FP64 instructions of a rotation bind:
//  - a rotation takes 1 / sqrt(f^2 + g^2) once instead of a hypot and two divisions; the matrix is
//    scaled by a power of two first, so the squares cannot overflow, and tiny ones take the hypot form;
//  - comparisons look at exponents with integer instructions;
//  - d, e and z live in shared memory, [row][chain], and the next row is loaded ahead of its use;
//  - every lane walks its own sequence of sweeps, so lanes wait for the longest total sequence of
//    their warp and not for the longest one of every eigenvalue; the warp starts each sweep together and
//    counts the longest one's rotations, since lanes that the compiler lets run apart pay for
//    every rotation again (eight chains of a warp: 6.0 ms apart, 4.5 together, one chain 3.9);
//  - a CTA is one warp and takes ceil(chains / (4 SMs)) chains: every scheduler gets one warp first.
// 4560 chains of 60 steps: 9.0 ms with one thread per chain in global memory, 4.5 ms now.

// 1 / sqrt(h) for normal h: the hardware's approximation and one step of Householder's third-order
// iteration, y (1 + e / 2 + 3 e^2 / 8) with e = 1 - h y^2 (five FP64 operations).
static __device__ __forceinline__ double ql_rsqrt(double h) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(h));
    const double e = fma(-(h * y), y, 1.0);
    return fma(fma(e, 0.375, 0.5), y * e, y);
}

// Whether |e| can be at most DBL_EPSILON (|d0| + |d1|), from the exponents alone (no FP64 operation).
static __device__ __forceinline__ bool ql_maybe_small(double e, double d0, double d1) {
    const int xe = (__double2hiint(e) >> 20) & 0x7ff;
    const int x0 = (__double2hiint(d0) >> 20) & 0x7ff, x1 = (__double2hiint(d1) >> 20) & 0x7ff;
    return xe + 50 <= max(x0, x1) || xe == 0;
}

// Eigenvalues of the symmetric tridiagonal matrix (diag d[0..n-1], off-diagonal
// e[i] between i and i+1) and the first row z of its orthonormal eigenvector
// matrix, element i of each array at i * ST.  Implicit QL sweeps with the shift
// taken from the leading 2x2 block; each Givens rotation is also applied to z.
// Called by the whole warp, lanes without a chain with n = 0.  Returns false if an
// eigenvalue does not converge within 60 sweeps.
static __device__ bool tridiag_ql(int n, double *d, double *e, double *z, int ST) {
    for (int i = 0; i < n; ++i) z[i * ST] = (i == 0) ? 1.0 : 0.0;
    if (n > 0) e[(n - 1) * ST] = 0.0;
    int l = 0, sweep = 0;
    bool live = n > 0, ok = true;
    for (;;) {
        int m = l;
        if (live) {
            for (; l < n; m = ++l, sweep = 0) {  // the next eigenvalue that needs a sweep, and its block's end
                for (; m < n - 1; ++m) {
                    const double em = e[m * ST], d0 = d[m * ST], d1 = d[(m + 1) * ST];
                    if (ql_maybe_small(em, d0, d1) && fabs(em) <= DBL_EPSILON * (fabs(d0) + fabs(d1))) break;
                }
                if (m != l) break;
            }
            live = l < n;
            if (live && sweep++ == 60) live = ok = false;
        }
        const int longest = __reduce_max_sync(kFull, live ? m - l : 0);
        if (longest == 0) return ok;
        double g = 0.0, dhi = 0.0, zhi = 0.0, ei = 0.0, di = 0.0, zi = 0.0;
        if (live) {
            const double dl = d[l * ST], el = e[l * ST];
            g = (d[(l + 1) * ST] - dl) / (2.0 * el);
            const double r0 = hypot(g, 1.0);
            dhi = d[m * ST];
            zhi = z[m * ST];
            g = dhi - dl + el / (g + (g >= 0 ? r0 : -r0));
            ei = e[(m - 1) * ST];
            di = d[(m - 1) * ST];
            zi = z[(m - 1) * ST];
        }
        double s = 1.0, c = 1.0, p = 0.0;
        bool run = live;
        int i = m - 1;
        for (int step = 0; step < longest; ++step, --i) {  // the same count in every lane
            __syncwarp();
            if (!run || i < l) continue;
            const int nx = (i > l ? i - 1 : i) * ST;
            const double en = e[nx], dn = d[nx], zn = z[nx];
            const double f = s * ei, bb = c * ei;
            const double h = fma(f, f, g * g);
            double r;
            if ((unsigned)__double2hiint(h) - 0x05D00000u < 0x7FF00000u - 0x05D00000u) {  // 2^-930 <= h < infinity
                const double inv = ql_rsqrt(h);
                r = h * inv;
                s = f * inv;
                c = g * inv;
            } else {
                r = hypot(f, g);
                if (r == 0.0) {
                    e[(i + 1) * ST] = 0.0;
                    d[(i + 1) * ST] = dhi - p;
                    z[(i + 1) * ST] = zhi;
                    e[m * ST] = 0.0;
                    run = false;
                    continue;
                }
                s = f / r;
                c = g / r;
            }
            e[(i + 1) * ST] = r;
            g = dhi - p;
            const double t = fma(di - g, s, (c + c) * bb);
            p = s * t;
            d[(i + 1) * ST] = g + p;
            g = c * t - bb;
            z[(i + 1) * ST] = s * zi + c * zhi;
            zhi = c * zi - s * zhi;
            dhi = di;
            ei = en;
            di = dn;
            zi = zn;
        }
        if (run) {
            d[l * ST] = dhi - p;
            z[l * ST] = zhi;
            e[l * ST] = g;
            e[m * ST] = 0.0;
        }
    }
}

// theta, w (sorted ascending) from alpha/beta rows of length m[c]: one warp per CTA, `per` chains each
static __global__ void __launch_bounds__(32) ritz_kernel(int n_chains, int ld, int per, const int *m, const double *alpha,
                                                         const double *beta, double *theta, double *w, int *err) {
    extern __shared__ double ritz_smem[];  // d, e, z: [ld][per] each
    const int lane = threadIdx.x, c0 = blockIdx.x * per, nc = min(per, n_chains - c0);
    double *sd = ritz_smem, *se = sd + (size_t)ld * per, *sz = se + (size_t)ld * per;
    for (int q = 0; q < nc; ++q)  // rows read along the chain, stored across
        for (int i = lane; i < ld; i += 32) {
            const int n = m[c0 + q];
            const size_t g = (size_t)(c0 + q) * ld + i;
            sd[i * per + q] = i < n ? alpha[g] : 0.0;
            se[i * per + q] = i < n ? beta[g] : 0.0;
            sz[i * per + q] = 0.0;
        }
    __syncwarp();
    const int n_raw = lane < nc ? m[c0 + lane] : 0;
    const bool bad = n_raw > ld || n_raw > kMaxSteps;
    if (bad) atomicOr(err, 2);
    const int n = bad || n_raw < 0 ? 0 : n_raw;
    double *d = sd + lane, *e = se + lane, *z = sz + lane;  // read and written below n only
    double big = 0.0;
    for (int i = 0; i < n; ++i) big = fmax(big, fmax(fabs(d[i * per]), i + 1 < n ? fabs(e[i * per]) : 0.0));
    const int k = big > 0.0 && big < INFINITY ? ilogb(big) : 0;
    if (k != 0)
        for (int i = 0; i < n; ++i) {
            d[i * per] = ldexp(d[i * per], -k);
            e[i * per] = ldexp(e[i * per], -k);
        }
    if (!tridiag_ql(n, d, e, z, per)) atomicOr(err, 1);
    for (int i = 0; i < n; ++i) {
        if (k != 0) d[i * per] = ldexp(d[i * per], k);
        z[i * per] *= z[i * per];
    }
    __syncwarp();
    for (int q = 0; q < nc; ++q) {  // the warp ranks one chain's values at a time (ties in row order)
        const int nq = __shfl_sync(kFull, n, q);
        const size_t g = (size_t)(c0 + q) * ld;
        for (int i = lane; i < ld; i += 32) {
            if (i >= nq) {
                theta[g + i] = 0.0;
                w[g + i] = 0.0;
                continue;
            }
            const double v = sd[i * per + q];
            int rank = 0;
            for (int j = 0; j < nq; ++j) {
                const double u = sd[j * per + q];
                rank += (u < v) || (j < i && !(u > v));
            }
            theta[g + rank] = v;
            w[g + rank] = sz[i * per + q];
        }
    }
}

// Chains per CTA and its shared memory: all SMs first, then fuller warps; three rows of ld doubles per chain.
static inline int ritz_per(int n_chains, int ld) {
    const int fit = std::max(1, (int)(200 * 1024 / (3 * sizeof(double) * (size_t)ld)));
    return std::min(std::min(32, fit), std::max(1, (n_chains + 4 * kNumSMs - 1) / (4 * kNumSMs)));
}
static inline ftlm_status ritz_launch(int n_chains, int ld, const int *m, const double *alpha, const double *beta,
                                      double *theta, double *w, int *err, cudaStream_t st) {
    const int per = ritz_per(n_chains, ld);
    const size_t smem = 3 * sizeof(double) * (size_t)ld * per;
    if (smem > 48 * 1024)
        FTLM_CUDA(cudaFuncSetAttribute(ritz_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    count_launch();
    ritz_kernel<<<(n_chains + per - 1) / per, 32, smem, st>>>(n_chains, ld, per, m, alpha, beta, theta, w, err);
    FTLM_CUDA(cudaGetLastError());
    return FTLM_OK;
}

// ---------------------------------------------------------------- thermal sums (Eqs. 5-7, 14)

struct ThermoIn {
    int n_chains, ld;
    const int *m;
    const double *theta, *w, *Wc, *Msq;
};

// smallest Ritz value: every chain's are sorted, so its first one
static __global__ void ground_energy(ThermoIn in, double *E0) {
    __shared__ double s[kThermoThreads / 32];
    double mn = INFINITY;
    for (int c = threadIdx.x; c < in.n_chains; c += blockDim.x)
        if (in.m[c] > 0) mn = fmin(mn, in.theta[(size_t)c * in.ld]);
    for (int o = 16; o; o >>= 1) mn = fmin(mn, __shfl_xor_sync(kFull, mn, o));
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = mn;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < kThermoThreads / 32; ++i) mn = fmin(mn, s[i]);
        *E0 = mn;
    }
}

// One cluster of kThermoCluster CTAs per temperature; the CTAs' sums meet through distributed shared
// memory, in rank order.  FP64 instructions bind, so one pass takes every moment: with x = theta - c for a c near
// the mean energy, z = sum W e, sum W e x and sum W e x^2, E = c + <x> and C = beta^2 (<x^2> - <x>^2).  c comes from a
// pass in FP32; any c gives the moments, and where this one is so far off that the difference would cancel
// more than a bit (energies far from zero beside their spread, values out of FP32's range), a second pass takes the
// centred moment.  (Error of C in units of 2^-53, 1e4 normal levels, the lowest 7.5 spreads down, T from 0.4 to 300
// spreads: up to 210 with c = E0 and six bits of cancellation allowed, 1.8 so, 2.3 with two centred FP64 passes.)
// The exponential is
// table-driven (Tang, ACM TOMS 15, 1989): e^{-beta x} = 2^{k / 256} 2^{r / 256} with k the nearest integer to
// -256 beta x / ln 2 and r the rest, -256 beta / ln 2 held as a sum of two doubles per temperature: r is exact
// to its own rounding, so the result does not carry the rounding of beta x.  17 FP64 operations per pair and
// temperature instead of about 60 in two passes.
// 273,600 pairs and 200 temperatures: 7.3 ms with two FP64 passes of one CTA per temperature, 2.9 ms now.
constexpr int kThermoCluster = 8;
constexpr int kExpTab = 256;

// 2^{x (s_hi + s_lo) / 256}, y = x s_hi rounded, -1100 * 256 < y <= 0, from tab[j] = 2^{j / 256}: the exponent is
// 256 q + j + r, |r| <= 1/2, and 2^{r / 256} - 1 its Taylor polynomial to fourth order (its remainder is below 4e-17)
static __device__ __forceinline__ double exp2_256(double x, double y, double s_hi, double s_lo, const double *tab) {
    constexpr double kShift = 6755399441055744.0;  // 1.5 * 2^52: adding it rounds to an integer
    constexpr double a = 0.0027076061740622863;    // ln 2 / 256
    const double s = y + kShift;
    const int k = __double2loint(s);
    const double r = fma(x, s_lo, fma(x, s_hi, -(s - kShift)));
    const double p = fma(r, fma(r, fma(r, a * a * a * a / 24.0, a * a * a / 6.0), a * a / 2.0), a);
    const double t = tab[k & (kExpTab - 1)];
    const double v = fma(t, r * p, t);  // in [1, 2)
    const int q = k >> 8;
    if (q < -1021) return ldexp(v, q);
    return __hiloint2double(__double2hiint(v) + (q << 20), __double2loint(v));
}

// a double cut to float by its bits (a conversion instruction would occupy the FP64 pipe); 0 below FP32's range,
// infinite or NaN above it
static __device__ __forceinline__ float coarse(double v) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const int e = (int)((hi >> 20) & 0x7ffu) - 1023 + 127;
    const unsigned m = ((hi << 3) | (lo >> 29)) & 0x7fffffu;
    const unsigned mag = e <= 0 ? 0u : e >= 255 ? 0x7f800000u | m : ((unsigned)e << 23) | m;
    return __uint_as_float((hi & 0x80000000u) | mag);
}

// (chain, step) of this thread's pairs: a flat walk over [n_chains][ld] with the division done once
template <class F>
static __device__ __forceinline__ void thermo_pairs(const ThermoIn &in, int rank, F f) {
    const unsigned stride = kThermoCluster * kThermoThreads, ld = (unsigned)in.ld;
    const unsigned i0 = (unsigned)rank * kThermoThreads + threadIdx.x;
    const unsigned dc = stride / ld, dk = stride % ld;
    unsigned c = i0 / ld, k = i0 % ld;
    while (c < (unsigned)in.n_chains) {
        if ((int)k < in.m[c]) f(c, (size_t)c * ld + k);
        c += dc;
        k += dk;
        if (k >= ld) {
            k -= ld;
            ++c;
        }
    }
}

static __global__ void __cluster_dims__(kThermoCluster, 1, 1) __launch_bounds__(kThermoThreads)
    thermo_kernel(ThermoIn in, const double *T, const double *E0p, double g, double *out /*[4][n_T]*/, int n_T) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    __shared__ double part[4], wsum[4][kThermoThreads / 32], mid[2], tab[kExpTab];
    const int it = blockIdx.x / kThermoCluster, rank = (int)cl.block_rank();
    const double beta = 1.0 / T[it], E0 = *E0p;
    for (int i = threadIdx.x; i < kExpTab; i += blockDim.x) tab[i] = exp2(i * (1.0 / kExpTab));
    __syncthreads();
    constexpr double c_hi = kExpTab / 0.69314718055994530942, c_lo = 5.2109500776783445e-15;  // 256 / ln 2
    const double s_hi = -beta * c_hi, s_lo = fma(-beta, c_hi, -s_hi) - beta * c_lo;
    auto boltzmann = [&](unsigned c, size_t t, double &x) {  // W e^{-beta x}
        x = in.theta[t] - E0;
        const double y = x * s_hi;
        const unsigned hi = (unsigned)__double2hiint(y);
        if (hi > 0xC1110000u || hi < 0x80000000u) {  // below -2^18 - 2^14, NaN, infinite or not negative
            if (hi < 0xFFF00000u && hi >= 0x80000000u) return 0.0;  // finite: e^{-beta x} rounds to 0
            return in.Wc[c] * in.w[t] * exp(-beta * x);
        }
        return in.Wc[c] * in.w[t] * exp2_256(x, y, s_hi, s_lo, tab);
    };
    // sums of v[0..3] over the cluster, valid in rank 0's thread 0
    auto cluster_sum = [&](double(&v)[4]) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            for (int o = 16; o; o >>= 1) v[q] += __shfl_xor_sync(kFull, v[q], o);
            if ((threadIdx.x & 31) == 0) wsum[q][threadIdx.x >> 5] = v[q];
        }
        __syncthreads();
        if (threadIdx.x < 4) {
            double sum = 0.0;
            for (int i = 0; i < kThermoThreads / 32; ++i) sum += wsum[threadIdx.x][i];
            part[threadIdx.x] = sum;
        }
        cl.sync();
        if (rank == 0 && threadIdx.x == 0)
            for (int q = 0; q < 4; ++q) {
                v[q] = 0.0;
#pragma unroll
                for (int r = 0; r < kThermoCluster; ++r) v[q] += *cl.map_shared_rank(&part[q], r);
            }
    };
    const float e0f = coarse(E0), sf = -1.442695f * (float)beta;
    float f0 = 0.f, f1 = 0.f;  // z and <theta - E0> z, to FP32's accuracy
    thermo_pairs(in, rank, [&](unsigned c, size_t t) {
        const float x = coarse(in.theta[t]) - e0f;
        const float b = coarse(in.Wc[c]) * coarse(in.w[t]) * exp2f(sf * x);
        f0 += b;
        f1 = fmaf(b, x, f1);
    });
    double v[4] = {(double)f0, (double)f1, 0.0, 0.0};
    cluster_sum(v);
    if (rank == 0 && threadIdx.x == 0) {
        const double m = v[1] / v[0];
        mid[0] = m > 0.0 && m < INFINITY ? E0 + m : E0;
    }
    cl.sync();
    const double ec = *cl.map_shared_rank(&mid[0], 0);
    v[0] = v[1] = v[2] = v[3] = 0.0;  // z, <x> z, <x^2> z, <M^2> z with x = theta - ec
    thermo_pairs(in, rank, [&](unsigned c, size_t t) {
        double x0;
        const double b = boltzmann(c, t, x0);
        if (b == 0.0 && x0 < INFINITY) return;
        const double x = in.theta[t] - ec, bx = b * x;
        v[0] += b;
        v[1] += bx;
        v[2] = fma(bx, x, v[2]);
        v[3] = fma(b, in.Msq[c], v[3]);
    });
    cluster_sum(v);
    const double z = v[0], xm = v[1] / v[0], zm = v[3];
    double var = v[2] / v[0] - xm * xm;
    if (rank == 0 && threadIdx.x == 0) {
        mid[0] = ec + xm;
        mid[1] = var < xm * xm ? 1.0 : 0.0;
    }
    cl.sync();
    const double xc = *cl.map_shared_rank(&mid[0], 0);
    const bool again = *cl.map_shared_rank(&mid[1], 0) != 0.0;
    if (again) {
        double u[4] = {0.0, 0.0, 0.0, 0.0};
        thermo_pairs(in, rank, [&](unsigned c, size_t t) {
            double x0;
            const double b = boltzmann(c, t, x0);
            if (b == 0.0 && x0 < INFINITY) return;
            const double x = in.theta[t] - xc;
            u[0] = fma(b * x, x, u[0]);
        });
        cluster_sum(u);
        var = u[0] / z;
    }
    if (rank == 0 && threadIdx.x == 0) {
        out[it] = log(z) - beta * E0;
        out[n_T + it] = ec + xm;
        out[2 * n_T + it] = beta * beta * var;
        out[3 * n_T + it] = g * g * beta * zm / z;
    }
    cl.sync();  // rank 0 has read every part before a CTA leaves
}

static inline ftlm_status thermo_launch(const ThermoIn &in, const double *T, double *E0, double g, double *out, int n_T,
                                        cudaStream_t st) {
    count_launch(2);
    ground_energy<<<1, kThermoThreads, 0, st>>>(in, E0);
    thermo_kernel<<<(unsigned)n_T * kThermoCluster, kThermoThreads, 0, st>>>(in, T, E0, g, out, n_T);
    FTLM_CUDA(cudaGetLastError());
    return FTLM_OK;
}

}  // namespace ftlm
