// fl_laplace.cu -- Algorithm 1 of Kunis & Melzer (Section 3): the real discrete
// Laplace transform f_j = sum_k c_k exp(-s_j t_k) through the hierarchical
// factorisation K~ = diag(L^{Y_m}) (K^{Y_m,Omega_l}) diag(L^{Omega_l})^T plus the
// cumulative sums g_m (Definition 3.2, Theorem A.3):
//
//   g_M = sum_{t_k in Omega_M} c_k,  g_m = g_{m+1} + sum_{t_k in Omega_m} c_k
//   v^{Omega_l}_r = sum_{t_k in Omega_l} L_r^{Omega_l}(t_k) c_k         (moments)
//   h^{Y_m}_s = sum_{l=l_m}^{L_m} sum_r K^{Y_m,Omega_l}_{s r} v^{Omega_l}_r (coupling)
//   f~_j = sum_s L_s^{Y_m}(s_j) h^{Y_m}_s + g_{L_m+1}  (s_j in Y_m),  g_1 (s_j in Y_M)
//
// Kernels of a planned transform: k_lap_minmax (interval ends y_1 = max s,
// xi_1 = max t, validity), k_lap_band (band of every t_k and s_j), and per
// execute k_lap_moments_cheb, k_lap_reduce_items, k_lap_couple_cheb and
// k_lap_eval_cheb, which carry the moments and the band functions as Chebyshev
// sums (the same interpolants, see the note at k_lap_kcheb).  The
// allocation-free call keeps the barycentric form (k_lap_moments, k_lap_reduce,
// k_lap_couple, k_lap_eval): it has no plan to hold the tables.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <string>
#include <vector>

#include "fl_plan.cuh"

namespace fl {

constexpr int kLapWarps = 8;          // warps per moment block
constexpr int kLapMaxBlocks = 128;    // moment blocks (fixed: partial-sum order)

__device__ __forceinline__ int lap_band(double v, double v1, int levels) {
    if (levels <= 1) return 1;
    if (v > ldexp(v1, -1)) return 1;
    if (!(v > ldexp(v1, -(levels - 1)))) return levels;
    int b = (int)floor(log2(v1 / v)) + 1;
    b = max(1, min(b, levels - 1));
    while (b > 1 && v > ldexp(v1, -(b - 1))) --b;
    while (b < levels - 1 && !(v > ldexp(v1, -b))) ++b;
    return b;
}

// max over non-negative doubles by their bit patterns (monotone for x >= 0);
// flag bit 1: a t_k or s_j is negative or not finite.
__global__ void k_lap_minmax(int64_t N, const double* __restrict__ t, int64_t M,
                             const double* __restrict__ s, unsigned long long* __restrict__ mx,
                             int* __restrict__ flag) {
    unsigned long long mt = 0, ms = 0;
    int bad = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += stride) {
        const double v = t[i];
        if (!(v >= 0.0) || !isfinite(v)) bad = 1;
        else mt = max(mt, (unsigned long long)__double_as_longlong(v));
    }
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < M; i += stride) {
        const double v = s[i];
        if (!(v >= 0.0) || !isfinite(v)) bad = 1;
        else ms = max(ms, (unsigned long long)__double_as_longlong(v));
    }
    if (bad) atomicOr(flag, 1);
    atomicMax(&mx[0], mt);
    atomicMax(&mx[1], ms);
}

__global__ void k_lap_band(int64_t n, const double* __restrict__ v, double v1, int levels,
                           uint8_t* __restrict__ band) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) band[i] = (uint8_t)lap_band(v[i], v1, levels);
}

// Moments and band sums.  Table row l (1..levels) holds v^{Omega_l}_0..q-1 and,
// in column q, the band sum sum_{t_k in Omega_l} c_k.  Each warp owns a table;
// for every 32 consecutive t_k it takes, lanes are grouped by band
// (match_any) and each group's sum is formed in lane order and added by the
// group's lowest lane, so the result does not depend on scheduling.
template <typename T>
__global__ void k_lap_moments(int64_t N, const double* __restrict__ t, const T* __restrict__ c,
                              int levels, int q, double xi1, const double* __restrict__ cheb,
                              T* __restrict__ partial) {
    extern __shared__ unsigned char smem_raw[];
    T* tab = reinterpret_cast<T*>(smem_raw);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nw = blockDim.x >> 5;   // warps (tables) per block
    const int row = q + 1;
    const int entries = (levels + 1) * row;
    for (int i = threadIdx.x; i < nw * entries; i += blockDim.x) tab[i] = (T)0;
    __syncthreads();
    T* mytab = tab + w * entries;
    const int64_t nchunk = (N + 31) / 32;
    for (int64_t ch = (int64_t)blockIdx.x * nw + w; ch < nchunk; ch += (int64_t)gridDim.x * nw) {
        const int64_t k = ch * 32 + lane;
        const bool valid = k < N;
        const int l = valid ? lap_band(t[k], xi1, levels) : 255;
        const double cv = valid ? (double)c[k] : 0.0;
        // barycentric denominator on Omega_l (only for interpolated bands)
        double tau = 0.0, inv_den = 1.0;
        int hit = -1;
        const bool interp = valid && l < levels;
        if (interp) {
            const double a = ldexp(xi1, -l);
            tau = (t[k] - 1.5 * a) / (0.5 * a);
            double den = 0.0;
            for (int r = 0; r < q; ++r) {
                const double d = tau - cheb[r];
                if (d == 0.0) hit = r;
                den += cheb[q + r] / d;
            }
            inv_den = 1.0 / den;
        }
        const unsigned peers = __match_any_sync(0xffffffffu, l);
        const bool leader = (peers & ((1u << lane) - 1u)) == 0u;
        for (int r = 0; r <= q; ++r) {
            T val = (T)0;
            if (r == q) {
                val = (T)cv;
            } else if (interp) {
                const double Lr = (hit >= 0) ? (r == hit ? 1.0 : 0.0)
                                             : (cheb[q + r] / (tau - cheb[r])) * inv_den;
                val = (T)(Lr * cv);
            }
            T acc = (T)0;
            for (int src = 0; src < 32; ++src) {
                const T x = __shfl_sync(0xffffffffu, val, src);
                if ((peers >> src) & 1u) acc += x;
            }
            if (valid && leader) mytab[l * row + r] += acc;
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < entries; i += blockDim.x) {
        T s = (T)0;
        for (int ww = 0; ww < nw; ++ww) s += tab[ww * entries + i];
        partial[(int64_t)blockIdx.x * entries + i] = s;
    }
}

// Barycentric weights w_r = lambda_r / (tau - t_r), r < q, with one division:
// Montgomery's batch inversion (prefix products of d_r = tau - t_r, one
// reciprocal, a backward sweep), about 3q ulps instead of 1/2 ulp per weight.
// Returns false and leaves hit = r when some d_r is exactly zero.
__device__ __forceinline__ bool bary_batch(double tau, int q, const double* __restrict__ cheb,
                                           double* w, int* hit) {
    double pre = 1.0;
    for (int r = 0; r < q; ++r) {
        const double d = tau - cheb[r];
        if (d == 0.0) {
            *hit = r;
            return false;
        }
        w[r] = pre;                      // product of d_0 .. d_{r-1}
        pre *= d;
    }
    double inv = 1.0 / pre;              // 1 / (d_0 ... d_{q-1})
    for (int r = q - 1; r >= 0; --r) {
        const double d = tau - cheb[r];
        const double ir = inv * w[r];    // 1 / d_r
        inv *= d;
        w[r] = cheb[q + r] * ir;
    }
    return true;
}

// vS[i] = sum over blocks of partial[b][i]: one warp per entry, lane l summing
// the blocks l, l + 32, ... and a fixed shuffle tree combining the lanes.
template <typename T>
__global__ void k_lap_reduce(int nblocks, int entries, const T* __restrict__ partial,
                             double* __restrict__ vS) {
    const int i = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (i >= entries) return;                    // uniform across the warp
    double s = 0.0;
    for (int b = lane; b < nblocks; b += 32) s += (double)partial[(int64_t)b * entries + i];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) vS[i] = s;
}

// h^{Y_m}_s for m = blockIdx.x + 1 (threads over s) with
// K^{Y_m,Omega_l}_{s r} = exp(-y_s xi_r) formed on the fly; block 0 also forms
// the cumulative sums g_l = sum_{l' >= l} S_{l'}, g_{levels+1} = 0.
__global__ void k_lap_couple(int levels, int q, double y1, double xi1,
                             const int* __restrict__ ell, const double* __restrict__ cheb,
                             const double* __restrict__ vS, double* __restrict__ h,
                             double* __restrict__ g) {
    const int m = blockIdx.x + 1;
    const int row = q + 1;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        g[levels + 1] = 0.0;
        for (int l = levels; l >= 1; --l) g[l] = g[l + 1] + vS[l * row + q];
    }
    if (m >= levels) return;
    const int s = threadIdx.x;
    if (s >= q) return;
    const double ay = ldexp(y1, -m);
    const double ys = 1.5 * ay + 0.5 * ay * cheb[s];
    double acc = 0.0;
    for (int l = ell[m]; l <= levels - m; ++l) {
        const double ax = ldexp(xi1, -l);
        for (int r = 0; r < q; ++r) {
            const double xr = 1.5 * ax + 0.5 * ax * cheb[r];
            acc += exp(-ys * xr) * vS[l * row + r];
        }
    }
    h[m * q + s] = acc;
}

// Plan-time table of the coupling blocks: Kt[koff[m] + ((l - l_m) q + s) q + r]
// = exp(-y_s^{Y_m} xi_r^{Omega_l}), the same expression k_lap_couple evaluates.
__global__ void k_lap_ktable(int levels, int q, double y1, double xi1, const int* __restrict__ ell,
                             const int64_t* __restrict__ koff, const double* __restrict__ cheb,
                             double* __restrict__ Kt) {
    const int m = blockIdx.x + 1;
    if (m >= levels) return;
    const int nl = levels - m - ell[m] + 1;
    const double ay = ldexp(y1, -m);
    for (int i = threadIdx.x; i < nl * q * q; i += blockDim.x) {
        const int r = i % q, s = (i / q) % q, l = ell[m] + i / (q * q);
        const double ys = 1.5 * ay + 0.5 * ay * cheb[s];
        const double ax = ldexp(xi1, -l);
        const double xr = 1.5 * ax + 0.5 * ax * cheb[r];
        Kt[koff[m] + i] = exp(-ys * xr);
    }
}

// Chebyshev form of a planned transform.  On Omega_l the Lagrange weights of
// the q Chebyshev points are L_r(t) = sum_j C_j(r) T_j(tau), C_j(r) =
// (2 - [j = 0]) / q T_j(t_r) (discrete orthogonality of the T_j, j < q), and
// likewise on Y_m, so with
//   u^{Omega_l}_j = sum_{t_k in Omega_l} T_j(tau_k) c_k   (u_0: the band sum S_l)
//   K''_{ij} = sum_s sum_r C_i(s) K^{Y_m,Omega_l}_{s r} C_j(r)   (plan time; stored as rows
//              over (l, j) per (m, i), so that a sum reads consecutive entries)
//   a^{Y_m}_i = sum_l sum_j K''_{ij} u^{Omega_l}_j
// the same interpolant is f~_j = sum_i T_i(sigma_j) a_i + g_{L_m+1}.  An element
// costs three operations per degree instead of the weights' products, their
// inversion and a scan over the warp: no division, no exact-hit case.
__global__ void k_lap_kcheb(int levels, int q, const int* __restrict__ ell, const int64_t* __restrict__ koff,
                            const double* __restrict__ Kt, double* __restrict__ Kc) {
    extern __shared__ double ksm[];                 // C (q x q), K (q x q), K C^T (q x q)
    double *C = ksm, *K = ksm + q * q, *X = ksm + 2 * q * q;
    const int m = blockIdx.x + 1, li = blockIdx.y;
    const int nl = ell ? levels - m - ell[m] + 1 : levels - 1;
    if (li >= nl) return;
    const int64_t base = ell ? koff[m] : (int64_t)(m - 1) * nl * q * q;
    const double* src = Kt + base + (int64_t)li * q * q;
    double* out = Kc + base + (int64_t)li * q;
    for (int i = threadIdx.x; i < q * q; i += blockDim.x) {
        const int j = i / q, r = i % q;
        C[i] = cospi((double)(j * (2 * r + 1) % (4 * q)) / (2.0 * q)) * ((j ? 2.0 : 1.0) / q);
        K[i] = src[i];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < q * q; i += blockDim.x) {
        const int s = i / q, j = i % q;
        double a = 0.0;
        for (int r = 0; r < q; ++r) a += K[s * q + r] * C[j * q + r];
        X[i] = a;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < q * q; i += blockDim.x) {
        const int ii = i / q, j = i % q;
        double a = 0.0;
        for (int s = 0; s < q; ++s) a += C[ii * q + s] * X[s * q + j];
        out[(int64_t)ii * nl * q + j] = a;
    }
}

// tau_k = (t_k - 3/2 a) / (a/2), a = v1 / 2^band, of every value (0 in the last
// band): double, or a float pair for the FP32 form, so that an execute needs no
// FP64 arithmetic per element there.
template <typename T> struct lap_tau { using type = double; };
template <> struct lap_tau<float> { using type = ff; };
template <typename T> using LapTau = typename lap_tau<T>::type;

template <typename T>
__global__ void k_lap_tau(int64_t n, const double* __restrict__ v, const uint8_t* __restrict__ band,
                          double v1, int levels, LapTau<T>* __restrict__ tau) {
    __shared__ double inv[FL_MAX_LEVELS + 1];            // 2 / a of every band
    for (int l = threadIdx.x; l < levels; l += blockDim.x) inv[l] = 1.0 / (0.5 * ldexp(v1, -l));
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int l = band[i];
    double x = 0.0;
    if (l < levels) {   // the quotient by its reciprocal, corrected once
        const double a = ldexp(v1, -l), h = 0.5 * a, d = v[i] - 1.5 * a, r = inv[l], q = d * r;
        x = r > 1e-280 && r < 1e280 ? fma(fma(-q, h, d), r, q) : d / h;
    }
    tau[i] = LapTau<T>(x);
}

// first[l] = first position of band l among the n bands in ascending order,
// l = 0 .. levels + 1.
__global__ void k_lap_starts(int64_t n, const uint8_t* __restrict__ band, int levels, int64_t* __restrict__ first) {
    const int l = threadIdx.x;
    if (l > levels + 1) return;
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (band[mid] < l) lo = mid + 1;
        else hi = mid;
    }
    first[l] = lo;
}

// The recurrences of T_j(tau), j < q.  Doubles step the differences
// d_{j+1} = T_{j+1} - T_j = d_j + 2 (|tau| - 1) T_j (with T_j(-x) = (-1)^j T_j(x)),
// whose rounding grows with j where the three-term recurrence's grows with j^2
// near the ends of the interval: three operations per degree.  Up to rank
// kLapPlain the three-term recurrence, of two, stays within the 3 q units that
// the barycentric weights' products had (16^2 / 2 units at the very ends, a few
// elsewhere); in float pairs j^2 2^-48 is far below the FP32 form's rounding.
constexpr int kLapPlain = 16;
__device__ __forceinline__ float ff_round(ff a) { return a.hi + a.lo; }

// What the moments are summed in: double, or (FP32 form) a float with the
// rounding of all its sums beside it, so that a moment reaches the coupling sums
// in more than FP32 accuracy -- the band functions' Chebyshev coefficients are as
// large as the function at its larger end, and moments rounded to float were
// off by up to 1.8 times what the float sums over Lagrange weights are (K_1/2 at 4431 x
// 35414: 7.9e-8 against 4.5e-8; 2^-24 = 6e-8).  An overflow stays in hi.
struct LapSum32 {
    float hi, lo;
    __device__ __forceinline__ LapSum32() : hi(0.f), lo(0.f) {}
    __device__ __forceinline__ LapSum32(float h, float l) : hi(h), lo(l) {}
    // exact sum of the high parts and their rounding
    __device__ __forceinline__ LapSum32 operator+(LapSum32 b) const {
        const float s = hi + b.hi, z = s - hi;
        return LapSum32(s, lo + b.lo + ((hi - (s - z)) + (b.hi - z)));
    }
};
template <typename T> struct lap_sum { using type = double; };
template <> struct lap_sum<float> { using type = LapSum32; };
template <typename T> using LapSum = typename lap_sum<T>::type;
__device__ __forceinline__ double lap_total(double v) { return v; }
__device__ __forceinline__ double lap_total(LapSum32 v) {
    return isfinite(v.hi) ? (double)v.hi + (double)v.lo : (double)v.hi;
}

// acc[j] += c T_j(tau), j < q <= P.
template <int P>
__device__ __forceinline__ void cheb_moments(double tau, double c, int q, double* acc) {
    if constexpr (P <= kLapPlain) {
        const double x2 = tau + tau;
        double t0 = 1.0, t1 = tau;
        acc[0] += c;
#pragma unroll
        for (int j = 1; j < P; ++j) {
            if (j < q) {
                if (j > 1) {
                    const double t2 = fma(x2, t1, -t0);
                    t0 = t1;
                    t1 = t2;
                }
                acc[j] = fma(c, t1, acc[j]);
            }
        }
        return;
    }
    const double e = fabs(tau) - 1.0, e2 = 2.0 * e, co = tau < 0.0 ? -c : c;
    double t = 1.0, d = e;
    acc[0] += c;
#pragma unroll
    for (int j = 1; j < P; ++j) {
        if (j < q) {
            if (j > 1) d = fma(e2, t, d);
            t += d;
            acc[j] = fma(j & 1 ? co : c, t, acc[j]);
        }
    }
}
template <int P>
__device__ __forceinline__ void cheb_moments(ff tau, float c, int q, LapSum32* acc) {
    const ff x2 = ff(2.f * tau.hi, 2.f * tau.lo);
    ff t0 = ff(1.f), t1 = tau;
    acc[0] = acc[0] + LapSum32(c, 0.f);
#pragma unroll
    for (int j = 1; j < P; ++j) {
        if (j < q) {
            if (j > 1) {
                const ff t2 = x2 * t1 - t0;
                t0 = t1;
                t1 = t2;
            }
            const float p = c * t1.hi;
            acc[j] = acc[j] + LapSum32(p, fmaf(c, t1.lo, fmaf(c, t1.hi, -p)));
        }
    }
}

// sum_i T_i(tau) a_i, i < q.
__device__ __forceinline__ double cheb_sum(double tau, const double* a, int q) {
    if (q <= kLapPlain) {
        const double x2 = tau + tau;
        double t0 = 1.0, t1 = tau, s = a[0];
        for (int i = 1; i < q; ++i) {
            s = fma(a[i], t1, s);
            const double t2 = fma(x2, t1, -t0);
            t0 = t1;
            t1 = t2;
        }
        return s;
    }
    const double e = fabs(tau) - 1.0, e2 = 2.0 * e;
    double t = 1.0, d = e, even = a[0], odd = 0.0;
    for (int i = 1; i < q; i += 2) {
        if (i > 1) d = fma(e2, t, d);
        t += d;
        odd = fma(a[i], t, odd);
        if (i + 1 < q) {
            d = fma(e2, t, d);
            t += d;
            even = fma(a[i + 1], t, even);
        }
    }
    return tau < 0.0 ? even - odd : even + odd;
}
__device__ __forceinline__ ff cheb_sum(ff tau, const ff* a, int q) {
    const ff x2 = ff(2.f * tau.hi, 2.f * tau.lo);
    ff t0 = ff(1.f), t1 = tau, s = a[0];
    for (int i = 1; i < q; ++i) {
        s += a[i] * t1;
        const ff t2 = x2 * t1 - t0;
        t0 = t1;
        t1 = t2;
    }
    return s;
}

// Work items of the moments: runs of consecutive elements of one band.
constexpr int kLapThreads = 256;
constexpr int kLapMaxPer = 16;     // elements per thread of an item, at most
struct LapItem {
    int64_t k0;
    int count;
    int band;
};

__device__ __forceinline__ float lap_shfl(float v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ double lap_shfl(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ LapSum32 lap_shfl(LapSum32 v, int o) { return LapSum32(lap_shfl(v.hi, o), lap_shfl(v.lo, o)); }

// Sums v[0 .. 7] over the lanes of a warp: halving steps (a lane keeps one half of
// its values and takes its partner's sums of that half), then two full ones; lane
// l ends with the sum of entry 4 [l & 16] + 2 [l & 8] + [l & 4] in v[0].  Nine
// exchanges for eight values instead of 40.
template <typename T> __device__ __forceinline__ void sum8(T* v, int lane) {
#pragma unroll
    for (int h = 4, off = 16; h > 0; h >>= 1, off >>= 1) {
        const bool up = lane & off;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const T give = up ? v[i] : v[i + h];
            const T keep = up ? v[i + h] : v[i];
            v[i] = keep + lap_shfl(give, off);
        }
    }
    v[0] = v[0] + lap_shfl(v[0], 2);
    v[0] = v[0] + lap_shfl(v[0], 1);
}

// Moments u_j of one item, j < q <= P: each thread sums its elements over the
// degrees in registers, exchanges sum the warp, shared memory the warps, all in a
// fixed order.  P is q rounded up to 8 (64 accumulators at q = 34 left one CTA
// per SM: 42 us at N = 2^16).  Bound by the FP64 pipe in the FP64 form (2 or 3
// operations per element and degree, 0.53e12 per second); the barycentric
// weights and a scan per degree took 38.7 us at N = 2^16, q = 11, and 354 us at
// N = 10^6 in the FP32 form, whose recurrence and sums run in float pairs (23
// operations per element and degree; with plain float sums the whole call at 10^6
// x 7 10^5 took 31.7 us, with pairs 37.0).
template <typename T, int P>
__global__ void __launch_bounds__(kLapThreads, P <= 40 ? 2 : 1)
    k_lap_moments_cheb(const LapItem* __restrict__ items, const LapTau<T>* __restrict__ tau,
                       const int32_t* __restrict__ tperm, const T* __restrict__ c, int levels, int q,
                       double* __restrict__ partial) {
    using S = LapSum<T>;
    __shared__ double red[kLapThreads / 32][P];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const LapItem it = items[blockIdx.x];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int qb = it.band < levels ? q : 1;         // the last band: its sum only
    S acc[P];
#pragma unroll
    for (int j = 0; j < P; ++j) acc[j] = S();
    for (int e = threadIdx.x; e < it.count; e += kLapThreads) {
        const int64_t k = it.k0 + e;
        cheb_moments<P>(tau[k], c[tperm[k]], qb, acc);
    }
#pragma unroll
    for (int j = 0; j < P; j += 8) {
        sum8(acc + j, lane);
        if ((lane & 3) == 0) red[w][j + (lane >> 2)] = lap_total(acc[j]);   // entry 4 [l & 16] + 2 [l & 8] + [l & 4] = l / 4
    }
    __syncthreads();
    if (threadIdx.x < P && threadIdx.x < q) {
        double s = 0.0;
        for (int ww = 0; ww < kLapThreads / 32; ++ww) s += red[ww][threadIdx.x];
        partial[(int64_t)blockIdx.x * q + threadIdx.x] = s;
    }
}

// The kernels of a planned transform depend on each other in turn and are short
// (4 to 20 us): each lets the next one's launch begin while it runs, and a
// kernel waits for the one before it to finish before it reads (programmatic
// dependent launch; the first kernel of a call is launched normally, whichever
// it is, so nothing of a call overlaps what precedes it on the stream).  A
// dependent is resident while partial, u, ha and g are still being written:
// they are passed as plain pointers (const __restrict__ would declare them
// unchanged for the kernel's lifetime and allow their loads to be moved before
// the wait), only the plan's tables and the caller's c and t as restricted ones.
__device__ __forceinline__ void lap_wait_previous() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... P, typename... A>
static cudaError_t lap_launch_after(bool* dependent, void (*kern)(P...), dim3 grid, dim3 block, cudaStream_t st,
                                    A... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = *dependent ? 1 : 0;
    *dependent = true;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

// u[l q + j] = sum over the items of band l of partial[item][j]: one warp per
// entry, the lanes striding over the items, a fixed shuffle tree.
__global__ void k_lap_reduce_items(int levels, int q, const int* __restrict__ first,
                                   const double* partial, double* u) {
    lap_wait_previous();
    const int i = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (i >= (levels + 1) * q) return;               // uniform across the warp
    const int l = i / q, j = i - l * q;
    double s = 0.0;
    for (int b = first[l] + lane; b < first[l + 1]; b += 32) s += partial[(int64_t)b * q + j];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) u[i] = s;
}

// a^{Y_m}_i = sum_{l = lo(m)}^{hi(m)} sum_j K''(m, l)_{ij} u^{Omega_l}_j, m = blockIdx.x
// + 1, one warp per i (blockIdx.y: groups of 8), lanes striding over (l, j), a
// fixed shuffle tree; written as LapTau<T> values (an overflow or NaN in the high
// part, with no low part).  Algorithm 1 (ell != nullptr):
// l = l_m .. M - m; the generalised algorithm: l = 1 .. M - 1.  The last block
// (the least of the others' work) also forms g_l = sum_{l' >= l} S_{l'} (S = u_0), g_{levels+1} = 0.
template <typename T> __device__ __forceinline__ LapTau<T> lap_value(double x) {
    if constexpr (sizeof(T) == 4) {
        const float hi = (float)x;
        return ff(hi, isfinite(hi) ? (float)(x - (double)hi) : 0.f);
    } else {
        return x;
    }
}

template <typename T>
__global__ void __launch_bounds__(256)
    k_lap_couple_cheb(int levels, int q, const int* __restrict__ ell, const int64_t* __restrict__ koff,
                      const double* __restrict__ Kt, const double* u, LapTau<T>* ha, LapTau<T>* g) {
    lap_wait_previous();
    const int m = blockIdx.x + 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (blockIdx.x == gridDim.x - 1 && blockIdx.y == 0 && threadIdx.x <= levels) {   // a thread per l
        const int l = threadIdx.x + 1;
        double s = 0.0;
#pragma unroll 4
        for (int k = levels; k >= l; --k) s += u[k * q];
        g[l] = lap_value<T>(s);
    }
    const int i = blockIdx.y * 8 + warp;
    if (m >= levels || i >= q) return;
    const int l0 = ell ? ell[m] : 1, l1 = ell ? levels - m : levels - 1;
    const int tot = max(l1 - l0 + 1, 0) * q;
    const double* K = Kt + (ell ? koff[m] : (int64_t)(m - 1) * tot * q) + (int64_t)i * tot;
    const double* ul = u + (int64_t)l0 * q;
    double acc = 0.0;
#pragma unroll 8
    for (int x = lane; x < tot; x += 32) acc += K[x] * ul[x];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (lane == 0) ha[m * q + i] = lap_value<T>(acc);
}

// f~_j = sum_i T_i(sigma_j) a_i + g_{L_m+1} (s_j in Y_m), g_1 (s_j in Y_M); the
// FP32 form in float pairs throughout.
template <typename T>
__global__ void __launch_bounds__(256)
    k_lap_eval_cheb(int64_t M, const LapTau<T>* __restrict__ sigma, const uint8_t* __restrict__ sband,
                    int levels, int q, const LapTau<T>* ha, const LapTau<T>* g, T* f) {
    lap_wait_previous();
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= M) return;
    const int m = sband[j];
    LapTau<T> v = g[m >= levels ? 1 : levels - m + 1];
    if constexpr (sizeof(T) == 4) {
        const float far = v.hi;
        if (m < levels) v = cheb_sum(sigma[j], ha + m * q, q) + v;
        f[j] = isinf(far) && m < levels ? cheb_sum(sigma[j], ha + m * q, q).hi + far : ff_round(v);
    } else {
        if (m < levels) v = cheb_sum(sigma[j], ha + m * q, q) + v;
        f[j] = v;
    }
}

// f~_j: barycentric weights of s_j on Y_m (double), then sum_s L_s h_s + g_{L_m + 1}.
template <typename T>
__global__ void k_lap_eval(int64_t M, const double* __restrict__ sv, int levels, int q, double y1,
                           const double* __restrict__ cheb, const double* __restrict__ h,
                           const double* __restrict__ g, T* __restrict__ f) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= M) return;
    const int m = lap_band(sv[j], y1, levels);
    if (m >= levels) {
        f[j] = (T)g[1];
        return;
    }
    const double a = ldexp(y1, -m);
    const double tau = (sv[j] - 1.5 * a) / (0.5 * a);
    double w[kMaxQ];
    int hit = -1;
    double interp;
    if (bary_batch(tau, q, cheb, w, &hit)) {
        double den = 0.0, num = 0.0;
        for (int s = 0; s < q; ++s) {
            den += w[s];
            num += w[s] * h[m * q + s];
        }
        interp = num / den;
    } else {
        interp = h[m * q + hit];
    }
    f[j] = (T)(interp + g[levels - m + 1]);
}

// Chebyshev points and barycentric weights (Section 2); same table as Algorithm 2.
__global__ void k_lap_cheb(int q, double* cheb) {
    const int s = threadIdx.x;
    if (s >= q) return;
    double sn, cs;
    sincospi((2.0 * s + 1.0) / (2.0 * q), &sn, &cs);
    cheb[s] = cs;
    cheb[q + s] = (s & 1) ? -sn : sn;
}

// ---------------------------------------------------------------------------
// Generalised Algorithm 1 (Section 3, the theorem after Algorithm 1): an
// asymptotically smooth kernel kappa(y, xi) in place of exp(-y xi).  Every
// block Y_m x Omega_l with 1 <= m, l <= M - 1 is interpolated (no block is
// replaced by 0 or 1), the near fields Y_M (every frequency) and Omega_M (every
// node) are summed directly, and M = ceil(log2(y_1 xi_1 N / eps)) + 1.
// Kernels: kind 1 exp(-y xi); kind 2 K_{1/2}(y xi) = sqrt(pi / (2 y xi)) exp(-y xi)
// (the example there, y, xi > 0).

constexpr int kGenMaxQ = 64;
static_assert(kGenMaxQ <= 64 && kMaxQ <= 64, "degrees of k_lap_moments_cheb");

__device__ __forceinline__ double gen_kappa(int kind, double y, double xi) {
    const double x = y * xi;
    return kind == 2 ? sqrt(1.5707963267948966192313216916398 / x) * exp(-x) : exp(-x);
}

// Kt[((m - 1)(M - 1) + l - 1) q^2 + s q + r] = kappa(y_s^{Y_m}, xi_r^{Omega_l}), block (m, l).
__global__ void k_gen_ktable(int kind, int levels, int q, double y1, double xi1,
                             const double* __restrict__ cheb, double* __restrict__ Kt) {
    const int m = blockIdx.x + 1, l = blockIdx.y + 1;
    const double ay = ldexp(y1, -m), ax = ldexp(xi1, -l);
    double* out = Kt + ((int64_t)(m - 1) * (levels - 1) + l - 1) * q * q;
    for (int i = threadIdx.x; i < q * q; i += blockDim.x) {
        const int r = i % q, s = i / q;
        const double ys = 1.5 * ay + 0.5 * ay * cheb[s];
        const double xr = 1.5 * ax + 0.5 * ax * cheb[r];
        out[i] = gen_kappa(kind, ys, xr);
    }
}

// f~_j: s_j in Y_m (m < M): the Chebyshev sum of the band plus the Omega_M near
// field sum_{t_k in Omega_M} c_k kappa(s_j, t_k); s_j in Y_M: the direct sum.
template <typename T, int KIND>
__global__ void k_gen_eval(int64_t M, const double* __restrict__ sv, const LapTau<T>* __restrict__ stau,
                           const uint8_t* __restrict__ sband, int levels, int q,
                           const LapTau<T>* ha, int64_t N, const double* __restrict__ t,
                           const T* __restrict__ c, const int32_t* __restrict__ nearT, int64_t nnear, T* f) {
    lap_wait_previous();
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= M) return;
    const int m = sband[j];
    const double sj = sv[j];
    double acc = 0.0;
    if (m >= levels) {
        for (int64_t k = 0; k < N; ++k) acc += (double)c[k] * gen_kappa(KIND, sj, t[k]);
    } else {
        acc = (double)cheb_sum(stau[j], ha + m * q, q);
        for (int64_t i = 0; i < nnear; ++i) {
            const int32_t k = nearT[i];
            acc += (double)c[k] * gen_kappa(KIND, sj, t[k]);
        }
    }
    f[j] = (T)acc;
}

// flag bit 1: a t_k or s_j is zero (kind 2 is singular at y xi = 0)
__global__ void k_gen_positive(int64_t N, const double* __restrict__ t, int64_t M,
                               const double* __restrict__ s, int* __restrict__ flag) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int bad = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += stride)
        if (!(t[i] > 0.0)) bad = 1;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < M; i += stride)
        if (!(s[i] > 0.0)) bad = 1;
    if (bad) atomicOr(flag, 1);
}

// ---------------------------------------------------------------------------
// Scratch layout of one Laplace evaluation (all offsets in bytes, 256-aligned).
struct LapLayout {
    size_t partial, vS, h, g, ell, total;
};

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

static LapLayout lap_layout(int levels, int q, int nblocks, size_t tsize) {
    LapLayout L;
    const size_t entries = (size_t)(levels + 1) * (q + 1);
    size_t off = 0;
    L.partial = off; off = align256(off + (size_t)nblocks * entries * tsize);
    L.vS = off;      off = align256(off + entries * sizeof(double));
    L.h = off;       off = align256(off + (size_t)(levels + 1) * q * sizeof(double));
    L.g = off;       off = align256(off + (size_t)(levels + 2) * sizeof(double));
    L.ell = off;     off = align256(off + (size_t)(levels + 1) * sizeof(int));
    L.total = off;
    return L;
}

static int lap_blocks(int64_t N) {
    const int64_t chunks = (N + 31) / 32;
    return (int)std::max<int64_t>(1, std::min<int64_t>(kLapMaxBlocks, (chunks + kLapWarps - 1) / kLapWarps));
}

// Parameters of Definition 3.2 for the whole eps (Algorithm 1).
struct LapParams {
    int q, levels;
    double y1, xi1;
    int ell[FL_MAX_LEVELS];
};

static bool lap_params(double eps, int q_in, double y1, double xi1, LapParams* P) {
    P->q = q_in > 0 ? q_in : (int)ceil(0.5 + log(1.0 / eps) / log(4.0));
    P->y1 = y1;
    P->xi1 = xi1;
    if (!(y1 > 0.0) || !(xi1 > 0.0)) {
        P->levels = 1;
    } else {
        P->levels = (int)std::max(1.0, ceil(log2(y1 * xi1 / eps)) + 1.0);
    }
    if (P->levels > 127 || P->q > kMaxQ) return false;
    for (int m = 0; m < FL_MAX_LEVELS; ++m) P->ell[m] = 0;
    for (int m = 1; m < P->levels; ++m) {
        const double lg = log2(y1 * xi1) - m - log2(log(1.0 / eps));
        P->ell[m] = std::max(1, (int)floor(lg) + 1);
    }
    return true;
}

// The allocation-free call: launches moments -> reduce -> couple -> eval on
// `scratch` (layout above), with nblocks moment blocks; the layout reserves
// partial sums for layout_blocks >= nblocks blocks.
template <typename T>
static cudaError_t noalloc_run(int64_t N, int64_t M, const double* t, const double* s, const LapParams& P,
                               const double* cheb, const T* c, T* f, unsigned char* scratch, int nblocks,
                               int layout_blocks, cudaStream_t st) {
    const LapLayout L = lap_layout(P.levels, P.q, layout_blocks, sizeof(T));
    const int entries = (P.levels + 1) * (P.q + 1);
    T* partial = (T*)(scratch + L.partial);
    double* vS = (double*)(scratch + L.vS);
    double* h = (double*)(scratch + L.h);
    double* g = (double*)(scratch + L.g);
    const int* ell = (const int*)(scratch + L.ell);
    const size_t smem = (size_t)kLapWarps * entries * sizeof(T);
    if (N > 0) {
        cudaError_t e = cudaFuncSetAttribute(k_lap_moments<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
        k_lap_moments<T><<<nblocks, kLapWarps * 32, smem, st>>>(N, t, c, P.levels, P.q, P.xi1, cheb, partial);
        k_lap_reduce<T><<<(entries * 32 + 255) / 256, 256, 0, st>>>(nblocks, entries, partial, vS);
    } else {
        cudaError_t e = cudaMemsetAsync(vS, 0, entries * sizeof(double), st);
        if (e != cudaSuccess) return e;
    }
    k_lap_couple<<<std::max(1, P.levels - 1), std::max(32, ((P.q + 31) / 32) * 32), 0, st>>>(
        P.levels, P.q, P.y1, P.xi1, ell, cheb, vS, h, g);
    if (M > 0)
        k_lap_eval<T><<<(unsigned)((M + 255) / 256), 256, 0, st>>>(M, s, P.levels, P.q, P.y1, cheb, h, g, f);
    return cudaGetLastError();
}

}  // namespace fl

using namespace fl;

static fl_status lap_fail(fl_status s, const std::string& m) { return set_error(s, m); }

namespace fl {

// Scratch of a planned transform: item partials, moments u, band functions a, g.
struct LapPlanLayout {
    size_t partial, u, ha, g, ell, first, total;
};

static LapPlanLayout lap_plan_layout(int levels, int q, int64_t items) {
    LapPlanLayout L;
    size_t off = 0;
    L.partial = off; off = align256(off + (size_t)items * q * sizeof(double));
    L.u = off;       off = align256(off + (size_t)(levels + 1) * q * sizeof(double));
    L.ha = off;      off = align256(off + (size_t)(levels + 1) * q * sizeof(double));
    L.g = off;       off = align256(off + (size_t)(levels + 2) * sizeof(double));
    L.ell = off;     off = align256(off + (size_t)(levels + 1) * sizeof(int));
    L.first = off;   off = align256(off + (size_t)(levels + 2) * sizeof(int));
    L.total = off;
    return L;
}

template <typename T, int P>
static void lap_moments_launch(Plan& p, const T* c, double* partial, cudaStream_t st) {
    k_lap_moments_cheb<T, P><<<(unsigned)p.n_lap_items, kLapThreads, 0, st>>>(
        (const LapItem*)p.d_lapitems, (const LapTau<T>*)p.d_ttau, p.d_tperm, c, p.levels, p.q, partial);
}

// moments -> reduce -> couple -> eval, both forms of the algorithm.
template <typename T>
static cudaError_t lap_plan_run(Plan& p, const T* c, T* f, cudaStream_t st) {
    const LapPlanLayout L = lap_plan_layout(p.levels, p.q, p.n_lap_items);
    unsigned char* scratch = (unsigned char*)p.d_lap;
    double* partial = (double*)(scratch + L.partial);
    double* u = (double*)(scratch + L.u);
    LapTau<T>* ha = (LapTau<T>*)(scratch + L.ha);
    LapTau<T>* g = (LapTau<T>*)(scratch + L.g);
    const int* first = (const int*)(scratch + L.first);
    const bool gen = p.lap_kernel != 0;
    int slot = -1;
    bool dependent = false;   // whether a kernel of this call precedes
    if (p.n_lap_items > 0) {
        timer_begin(p, "lap_moments", (double)p.N * (8 + 4 + sizeof(T)), st, &slot);
        switch ((p.q + 7) / 8) {
#define FL_LAP_P(X) \
    case X: lap_moments_launch<T, 8 * X>(p, c, partial, st); break;
            FL_LAP_P(1) FL_LAP_P(2) FL_LAP_P(3) FL_LAP_P(4) FL_LAP_P(5) FL_LAP_P(6) FL_LAP_P(7) FL_LAP_P(8)
#undef FL_LAP_P
        default: return cudaErrorInvalidValue;
        }
        timer_end(p, slot, st);
        ++p.launches;
        dependent = true;
    }
    // (bands without items sum to zero: no elements, no moments)
    if (!gen || (p.N > 0 && p.levels > 1)) {
        const int entries = (p.levels + 1) * p.q;
        cudaError_t e = lap_launch_after(&dependent, k_lap_reduce_items, dim3((unsigned)((entries * 32 + 255) / 256)),
                                         dim3(256), st, p.levels, p.q, first, partial, u);
        const dim3 grid((unsigned)std::max(1, p.levels - 1), (unsigned)((p.q + 7) / 8));
        if (e == cudaSuccess)
            e = lap_launch_after(&dependent, k_lap_couple_cheb<T>, grid, dim3(256), st, p.levels, p.q,
                                 gen ? (const int*)nullptr : (const int*)(scratch + L.ell), p.d_lapKoff, p.d_lapK, u,
                                 ha, g);
        if (e != cudaSuccess) return e;
        p.launches += 2;
    }
    if (p.M > 0) {
        timer_begin(p, "lap_eval", (double)p.M * (8 + 1 + sizeof(T)), st, &slot);
        const dim3 grid((unsigned)((p.M + 255) / 256)), block(256);
        const LapTau<T>* sg = (const LapTau<T>*)p.d_stau;
        const cudaError_t e =
            p.lap_kernel == 0
                ? lap_launch_after(&dependent, k_lap_eval_cheb<T>, grid, block, st, p.M, sg, p.d_sband, p.levels, p.q,
                                   ha, g, f)
                : lap_launch_after(&dependent, p.lap_kernel == 2 ? k_gen_eval<T, 2> : k_gen_eval<T, 1>, grid, block, st, p.M,
                                   p.d_s, sg, p.d_sband, p.levels, p.q, ha, p.N, p.d_t, c, p.d_nearT, p.n_nearT, f);
        if (e != cudaSuccess) return e;
        timer_end(p, slot, st);
        p.launches += 1;
    }
    return cudaGetLastError();
}

cudaError_t run_laplace(Plan& p, const void* c, void* f, cudaStream_t st) {
    return p.prec == FL_FP64 ? lap_plan_run<double>(p, (const double*)c, (double*)f, st)
                             : lap_plan_run<float>(p, (const float*)c, (float*)f, st);
}

}  // namespace fl

#define LAP_CUDA(call, where)                                                      \
    do {                                                                           \
        cudaError_t e_ = (call);                                                   \
        if (e_ != cudaSuccess)                                                     \
            return lap_fail(e_ == cudaErrorMemoryAllocation ? FL_ENOMEM : FL_ECUDA, \
                            std::string(where) + ": " + cudaGetErrorString(e_));   \
    } while (0)

__global__ void k_lap_sortprep(int64_t n, const uint8_t* __restrict__ band, uint32_t* __restrict__ keys,
                               int32_t* __restrict__ vals) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        keys[i] = band[i];
        vals[i] = (int32_t)i;
    }
}

__global__ void k_lap_sorted(int64_t n, const double* __restrict__ t, const uint32_t* __restrict__ keys,
                             const int32_t* __restrict__ vals, double* __restrict__ ts,
                             uint8_t* __restrict__ bs, int32_t* __restrict__ perm) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        ts[i] = t[vals[i]];
        bs[i] = (uint8_t)keys[i];
        perm[i] = vals[i];
    }
}

// Plan time: copies of the t_k and their bands in band order (stable: equal
// bands keep the input order), with tperm the original index of each.
static cudaError_t sort_t_by_band(Plan& p, cudaStream_t st) {
    const int64_t n = p.N;
    uint32_t *keys = nullptr, *ktmp = nullptr, *hist = nullptr;
    int32_t *vals = nullptr, *vtmp = nullptr;
    const int64_t nblocks = (n + 2047) / 2048;        // radix-sort tiles of 256 x 8
    const auto al = DevPool::rounded;
    cudaError_t e = p.scratch().reserve(4 * al(4 * n) + al(1024 * nblocks) + al(8 * n) + al(n));
    if (e == cudaSuccess) e = p.scratch().get(&keys, n);
    if (e == cudaSuccess) e = p.scratch().get(&ktmp, n);
    if (e == cudaSuccess) e = p.scratch().get(&vals, n);
    if (e == cudaSuccess) e = p.scratch().get(&vtmp, n);
    if (e == cudaSuccess) e = p.scratch().get(&hist, 256 * nblocks);
    if (e == cudaSuccess) e = p.scratch().get(&p.d_ts, n);
    if (e == cudaSuccess) e = p.scratch().get(&p.d_tbs, n);
    if (e == cudaSuccess) e = p.pool.get(&p.d_tperm, n);
    if (e != cudaSuccess) return e;
    k_lap_sortprep<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, p.d_tband, keys, vals);
    e = radix_sort_pairs(keys, vals, ktmp, vtmp, hist, n, 8, st);
    if (e != cudaSuccess) return e;
    k_lap_sorted<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, p.d_t, keys, vals, p.d_ts, p.d_tbs, p.d_tperm);
    return cudaGetLastError();
}

// Plan time, after sort_t_by_band: tau of the t_k in band order and of the s_j,
// and the moment items -- runs of up to 256 E elements of one band, E so that
// the launch has about four items per SM up to E = kLapMaxPer (N = 2^16: 256
// items of 256 elements, which the FP64 pipes of all SMs share; longer runs
// only pay once that many items are there).  last: whether the last band is
// summed too.
template <typename T>
static cudaError_t lap_tables(Plan& p, bool last, std::vector<LapItem>* items, std::vector<int>* first,
                              cudaStream_t st) {
    items->clear();
    first->assign(p.levels + 2, 0);
    cudaError_t e = cudaSuccess;
    if (p.M > 0) {
        e = p.pool.bytes(&p.d_stau, p.M * sizeof(LapTau<T>));
        if (e != cudaSuccess) return e;
        k_lap_tau<T><<<(unsigned)((p.M + 255) / 256), 256, 0, st>>>(p.M, p.d_s, p.d_sband, p.y1, p.levels,
                                                                    (LapTau<T>*)p.d_stau);
    }
    if (p.N == 0) return cudaGetLastError();
    e = p.pool.bytes(&p.d_ttau, p.N * sizeof(LapTau<T>));
    int64_t* d_first = nullptr;
    std::vector<int64_t> start(p.levels + 2);
    if (e == cudaSuccess) e = p.scratch().get(&d_first, (int64_t)start.size());
    if (e == cudaSuccess) {
        k_lap_tau<T><<<(unsigned)((p.N + 255) / 256), 256, 0, st>>>(p.N, p.d_ts, p.d_tbs, p.xi1, p.levels,
                                                                    (LapTau<T>*)p.d_ttau);
        k_lap_starts<<<1, FL_MAX_LEVELS + 32, 0, st>>>(p.N, p.d_tbs, p.levels, d_first);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(start.data(), d_first, start.size() * sizeof(int64_t), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
    if (p.N > kTmpKeep) p.tmp.release();   // (all of it has been used)
    const int64_t per = std::min<int64_t>(kLapMaxPer, std::max<int64_t>(1, p.N / (kLapThreads * 4 * 152)));
    for (int l = 1; l <= p.levels; ++l) {
        (*first)[l] = (int)items->size();
        if (l == p.levels && !last) break;
        for (int64_t k = start[l]; k < start[l + 1]; k += per * kLapThreads)
            items->push_back({k, (int)std::min<int64_t>(per * kLapThreads, start[l + 1] - k), l});
    }
    (*first)[p.levels + 1] = (int)items->size();
    return cudaSuccess;
}

// The plan's scratch with the item starts, the items, and (nk blocks Kt of the
// coupling table) the table's Chebyshev form p.d_lapK.
static cudaError_t lap_upload(Plan& p, const std::vector<LapItem>& items, const std::vector<int>& first,
                              const std::vector<int>& ell, int64_t nk, double* Kt, size_t* scratch, cudaStream_t st) {
    p.n_lap_items = (int64_t)items.size();
    const LapPlanLayout L = lap_plan_layout(p.levels, p.q, p.n_lap_items);
    *scratch = L.total + items.size() * sizeof(LapItem);
    cudaError_t e = p.pool.bytes(&p.d_lap, L.total);
    unsigned char* base = (unsigned char*)p.d_lap;
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(base + L.first, first.data(), first.size() * sizeof(int), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && !ell.empty())
        e = cudaMemcpyAsync(base + L.ell, ell.data(), ell.size() * sizeof(int), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && !items.empty()) {
        e = p.pool.bytes(&p.d_lapitems, items.size() * sizeof(LapItem));
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(p.d_lapitems, items.data(), items.size() * sizeof(LapItem),
                                cudaMemcpyHostToDevice, st);
    }
    if (e == cudaSuccess && nk > 0) {
        const size_t smem = 3 * (size_t)p.q * p.q * sizeof(double);   // <= 96 KiB (q <= 64)
        e = cudaFuncSetAttribute(k_lap_kcheb, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        e = p.pool.bytes((void**)&p.d_lapK, nk * p.q * p.q * sizeof(double));
        if (e != cudaSuccess) return e;
        const bool gen = ell.empty();
        k_lap_kcheb<<<dim3((unsigned)(p.levels - 1), (unsigned)(p.levels - 1)), 256, smem, st>>>(
            p.levels, p.q, gen ? nullptr : (const int*)(base + L.ell), p.d_lapKoff, Kt, p.d_lapK);
        e = cudaGetLastError();
    }
    return e;
}

// The arrays of a plan whose sizes follow from N and M (one block for them).
static size_t lap_known_bytes(const Plan& p) {
    const auto al = DevPool::rounded;
    const size_t N = (size_t)p.N, M = (size_t)p.M;
    size_t n = al(8 * N) + al(N) + al(4 * N) + al(8 * N) + al(8 * M) + al(M) + al(8 * M) + al(128 * sizeof(double));
    if (p.small) n += 5 * al(4 * N) + al(8 * N) + al(N) + ((size_t)1 << 17);   // the sort's too
    return n;
}

static fl_status plan_laplace_impl(Plan& p, const double* t, const double* s, int q,
                                   cudaStream_t st) {
    // interval ends and validity
    unsigned long long* dmx = nullptr;
    int* dflag = nullptr;
    p.small = p.N <= kSmallPlan && p.M <= kSmallPlan;
    cudaError_t e = p.pool.reserve(lap_known_bytes(p));
    if (e == cudaSuccess) e = p.scratch().get(&dmx, 2);
    if (e == cudaSuccess) e = p.scratch().get(&dflag, 1);
    unsigned long long mx[2] = {0, 0};
    int flag = 0;
    if (e == cudaSuccess) e = cudaMemsetAsync(dmx, 0, 2 * sizeof(unsigned long long), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(dflag, 0, sizeof(int), st);
    if (e == cudaSuccess && (p.N > 0 || p.M > 0)) {
        k_lap_minmax<<<256, 256, 0, st>>>(p.N, t, p.M, s, dmx, dflag);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(mx, dmx, sizeof(mx), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&flag, dflag, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    LAP_CUDA(e, "fl_plan_laplace: node scan");
    if (flag) return lap_fail(FL_EINVAL, "fl_plan_laplace: a t_k or s_j is negative or not finite");
    double xi1, y1;
    memcpy(&xi1, &mx[0], sizeof(double));
    memcpy(&y1, &mx[1], sizeof(double));
    LapParams P;
    if (!lap_params(p.eps, q, y1, xi1, &P))
        return lap_fail(FL_EUNSUPPORTED, "fl_plan_laplace: more than 127 levels or q above 40");
    p.q = P.q;
    p.levels = P.levels;
    p.y1 = y1;
    p.xi1 = xi1;
    p.eps_K = p.eps;
    p.bands.assign(P.levels + 1, BandHost());
    for (int m = 1; m < P.levels; ++m) {
        p.bands[m].ell = P.ell[m];
        p.bands[m].Lm = P.levels - m;
    }
    // copies of the nodes and their band ids
    const size_t N = (size_t)p.N, M = (size_t)p.M;
    if (N) {
        LAP_CUDA(p.pool.bytes((void**)&p.d_t, N * sizeof(double)), "cudaMalloc t");
        LAP_CUDA(cudaMemcpyAsync(p.d_t, t, N * sizeof(double), cudaMemcpyDeviceToDevice, st), "copy t");
        LAP_CUDA(p.pool.bytes((void**)&p.d_tband, N), "cudaMalloc t bands");
        k_lap_band<<<(unsigned)((N + 255) / 256), 256, 0, st>>>(p.N, p.d_t, xi1, P.levels, p.d_tband);
        LAP_CUDA(sort_t_by_band(p, st), "fl_plan_laplace: band order");
    }
    if (M) {
        LAP_CUDA(p.pool.bytes((void**)&p.d_s, M * sizeof(double)), "cudaMalloc s");
        LAP_CUDA(cudaMemcpyAsync(p.d_s, s, M * sizeof(double), cudaMemcpyDeviceToDevice, st), "copy s");
        LAP_CUDA(p.pool.bytes((void**)&p.d_sband, M), "cudaMalloc s bands");
        k_lap_band<<<(unsigned)((M + 255) / 256), 256, 0, st>>>(p.M, p.d_s, y1, P.levels, p.d_sband);
    }
    LAP_CUDA(p.pool.bytes((void**)&p.d_cheb, 2 * kMaxQ * sizeof(double)), "cudaMalloc cheb");
    k_lap_cheb<<<1, 64, 0, st>>>(P.q, p.d_cheb);
    // (a limit of the tables that the allocation-free call keeps in shared memory; planned
    // transforms have none, and refuse the same problems as ever)
    const size_t tsz = p.prec == FL_FP64 ? 8 : 4;
    if ((size_t)kLapWarps * (P.levels + 1) * (P.q + 1) * tsz > 200 * 1024)
        return lap_fail(FL_EUNSUPPORTED, "fl_plan_laplace: moment tables exceed shared memory "
                                         "(too many levels for this q)");
    std::vector<int> ell(P.levels + 1, 0), first;
    for (int m = 1; m < P.levels; ++m) ell[m] = P.ell[m];
    std::vector<LapItem> items;
    LAP_CUDA(p.prec == FL_FP64 ? lap_tables<double>(p, true, &items, &first, st)
                               : lap_tables<float>(p, true, &items, &first, st),
             "fl_plan_laplace: moment items");
    // coupling blocks K^{Y_m, Omega_l}, l = l_m .. L_m, as a table
    std::vector<int64_t> koff(P.levels + 1, 0);
    int64_t ktot = 0;
    for (int m = 1; m < P.levels; ++m) {
        koff[m] = ktot;
        ktot += (int64_t)std::max(0, P.levels - m - P.ell[m] + 1) * P.q * P.q;
    }
    int* d_ell = nullptr;   // l_m for the table kernel
    double* Kt = nullptr;   // the blocks at the Chebyshev points
    LAP_CUDA(p.pool.bytes((void**)&p.d_lapKoff, koff.size() * sizeof(int64_t)), "cudaMalloc coupling offsets");
    LAP_CUDA(cudaMemcpyAsync(p.d_lapKoff, koff.data(), koff.size() * sizeof(int64_t), cudaMemcpyHostToDevice, st),
             "copy coupling offsets");
    if (ktot > 0) {
        LAP_CUDA(p.scratch().get(&Kt, ktot), "cudaMalloc coupling table");
        LAP_CUDA(p.scratch().get(&d_ell, (int64_t)ell.size()), "cudaMalloc l_m");
        e = cudaMemcpyAsync(d_ell, ell.data(), ell.size() * sizeof(int), cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess) {
            k_lap_ktable<<<P.levels - 1, 256, 0, st>>>(P.levels, P.q, y1, xi1, d_ell, p.d_lapKoff, p.d_cheb, Kt);
            e = cudaGetLastError();
        }
    }
    size_t scratch = 0;
    if (e == cudaSuccess) e = lap_upload(p, items, first, ell, ktot / (P.q * P.q), Kt, &scratch, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    LAP_CUDA(e, "fl_plan_laplace: tables");
    p.tmp.release();
    const size_t ts = p.prec == FL_FP64 ? 8 : 4;
    p.scratch_bytes = (double)scratch + (N + M) * (9.0 + 8.0);
    p.model_bytes = (double)N * (8 + 1 + ts) + (double)M * (8 + 1 + ts);
    return FL_OK;
}

// Generalised Algorithm 1: rank from the block bound of the proof of
// Theorem 3.1, C mu^q q^nu 2^(1-2q) (2 + (2/pi) ln q) (dist(A,0) dist(B,0))^-s
// <= eps, with dist(A,0) dist(B,0) >= (y_1 / 2^(M-1)) (xi_1 / 2^(M-1)) and the
// asymptotic-smoothness constants of the kernel (exp: C = 1, mu = 1, nu = 0,
// s = 0; K_1/2: C = sqrt(pi/2), mu = 1, nu = 0, s = 1/2).
static int gen_rank(int kind, double eps, double dmin) {
    const double C = kind == 2 ? sqrt(M_PI / 2.0) : 1.0, sexp = kind == 2 ? 0.5 : 0.0;
    for (int q = 1; q <= kGenMaxQ; ++q) {
        const double b = C * pow(2.0, 1 - 2 * q) * (2.0 + 2.0 / M_PI * log((double)q)) * pow(dmin, -sexp);
        if (b <= eps) return q;
    }
    return kGenMaxQ + 1;
}

static fl_status plan_general_impl(Plan& p, int kind, const double* t, const double* s, int q,
                                   cudaStream_t st) {
    unsigned long long* dmx = nullptr;
    int* dflag = nullptr;
    p.small = p.N <= kSmallPlan && p.M <= kSmallPlan;
    cudaError_t e = p.pool.reserve(lap_known_bytes(p));
    if (e == cudaSuccess) e = p.scratch().get(&dmx, 2);
    if (e == cudaSuccess) e = p.scratch().get(&dflag, 2);
    unsigned long long mx[2] = {0, 0};
    int flag[2] = {0, 0};
    if (e == cudaSuccess) e = cudaMemsetAsync(dmx, 0, 2 * sizeof(unsigned long long), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(dflag, 0, 2 * sizeof(int), st);
    if (e == cudaSuccess && (p.N > 0 || p.M > 0)) {
        k_lap_minmax<<<256, 256, 0, st>>>(p.N, t, p.M, s, dmx, dflag);
        if (kind == 2) k_gen_positive<<<256, 256, 0, st>>>(p.N, t, p.M, s, dflag + 1);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(mx, dmx, sizeof(mx), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(flag, dflag, sizeof(flag), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    LAP_CUDA(e, "fl_plan_kernel: node scan");
    if (flag[0]) return lap_fail(FL_EINVAL, "fl_plan_kernel: a t_k or s_j is negative or not finite");
    if (flag[1]) return lap_fail(FL_EINVAL, "fl_plan_kernel: the K_1/2 kernel needs every t_k, s_j > 0");
    double xi1, y1;
    memcpy(&xi1, &mx[0], sizeof(double));
    memcpy(&y1, &mx[1], sizeof(double));
    int levels = 1;
    if (y1 > 0.0 && xi1 > 0.0 && p.N > 0)
        levels = (int)std::max(1.0, ceil(log2(y1 * xi1 * (double)p.N / p.eps)) + 1.0);
    if (levels > 127) return lap_fail(FL_EUNSUPPORTED, "fl_plan_kernel: more than 127 levels");
    const double dmin = ldexp(y1, 1 - levels) * ldexp(xi1, 1 - levels);
    const int qq = q > 0 ? q : gen_rank(kind, p.eps, dmin);
    if (qq > kGenMaxQ) return lap_fail(FL_EUNSUPPORTED, "fl_plan_kernel: rank above 64 for this eps");
    p.lap_kernel = kind;
    p.q = qq;
    p.levels = levels;
    p.y1 = y1;
    p.xi1 = xi1;
    p.eps_K = p.eps;
    p.bands.assign(levels + 1, BandHost());
    const size_t N = (size_t)p.N, M = (size_t)p.M;
    if (N) {
        LAP_CUDA(p.pool.bytes((void**)&p.d_t, N * sizeof(double)), "cudaMalloc t");
        LAP_CUDA(cudaMemcpyAsync(p.d_t, t, N * sizeof(double), cudaMemcpyDeviceToDevice, st), "copy t");
        LAP_CUDA(p.pool.bytes((void**)&p.d_tband, N), "cudaMalloc t bands");
        k_lap_band<<<(unsigned)((N + 255) / 256), 256, 0, st>>>(p.N, p.d_t, xi1, levels, p.d_tband);
        LAP_CUDA(sort_t_by_band(p, st), "fl_plan_kernel: band order");
    }
    if (M) {
        LAP_CUDA(p.pool.bytes((void**)&p.d_s, M * sizeof(double)), "cudaMalloc s");
        LAP_CUDA(cudaMemcpyAsync(p.d_s, s, M * sizeof(double), cudaMemcpyDeviceToDevice, st), "copy s");
        LAP_CUDA(p.pool.bytes((void**)&p.d_sband, M), "cudaMalloc s bands");
        k_lap_band<<<(unsigned)((M + 255) / 256), 256, 0, st>>>(p.M, p.d_s, y1, levels, p.d_sband);
    }
    LAP_CUDA(p.pool.bytes((void**)&p.d_cheb, 2 * kGenMaxQ * sizeof(double)), "cudaMalloc cheb");
    k_lap_cheb<<<1, kGenMaxQ, 0, st>>>(qq, p.d_cheb);
    // (of a table that earlier kernels kept in shared memory; the refusals are unchanged)
    const size_t tsz = p.prec == FL_FP64 ? 8 : 4;
    if ((size_t)(levels + 1) * (qq + 1) * tsz > 200 * 1024)
        return lap_fail(FL_EUNSUPPORTED, "fl_plan_kernel: moment tables exceed shared memory");
    std::vector<LapItem> items;
    std::vector<int> first;
    LAP_CUDA(p.prec == FL_FP64 ? lap_tables<double>(p, false, &items, &first, st)
                               : lap_tables<float>(p, false, &items, &first, st),
             "fl_plan_kernel: moment items");
    int64_t nk = 0;   // blocks of the coupling table
    double* Kt = nullptr;
    // the Omega_M near field: indices of the t_k in the last frequency band
    if (N && levels > 1) {
        std::vector<uint8_t> tb(N);
        LAP_CUDA(cudaMemcpyAsync(tb.data(), p.d_tband, N, cudaMemcpyDeviceToHost, st), "copy t bands");
        LAP_CUDA(cudaStreamSynchronize(st), "fl_plan_kernel: synchronise");
        std::vector<int32_t> near;
        for (size_t k = 0; k < N; ++k)
            if (tb[k] == levels) near.push_back((int32_t)k);
        p.n_nearT = (int64_t)near.size();
        if (!near.empty()) {
            LAP_CUDA(p.pool.bytes((void**)&p.d_nearT, near.size() * sizeof(int32_t)), "cudaMalloc near field");
            LAP_CUDA(cudaMemcpyAsync(p.d_nearT, near.data(), near.size() * sizeof(int32_t),
                                     cudaMemcpyHostToDevice, st),
                     "copy near field");
        }
        nk = (int64_t)(levels - 1) * (levels - 1);
        LAP_CUDA(p.scratch().get(&Kt, nk * qq * qq), "cudaMalloc coupling table");
        k_gen_ktable<<<dim3((unsigned)(levels - 1), (unsigned)(levels - 1)), 256, 0, st>>>(kind, levels, qq, y1, xi1,
                                                                                          p.d_cheb, Kt);
    }
    LAP_CUDA(cudaGetLastError(), "fl_plan_kernel: launch");
    size_t scratch = 0;
    e = lap_upload(p, items, first, std::vector<int>(), nk, Kt, &scratch, st);
    LAP_CUDA(e, "fl_plan_kernel: tables");
    LAP_CUDA(cudaStreamSynchronize(st), "fl_plan_kernel: synchronise");
    p.tmp.release();
    p.scratch_bytes = (double)scratch + (N + M) * (9.0 + 8.0) + (double)nk * qq * qq * 8.0;
    p.model_bytes = (double)N * (8 + 1 + tsz) + (double)M * (8 + 1 + tsz);
    return FL_OK;
}

extern "C" {

fl_status fl_plan_laplace(fl_plan_t* out, int64_t N, int64_t M, const double* t_dev,
                          const double* s_dev, int q, double eps, fl_precision prec, void* stream) {
    clear_error();
    if (!out) return lap_fail(FL_EINVAL, "fl_plan_laplace: out is NULL");
    *out = nullptr;
    if (N < 0 || M < 0) return lap_fail(FL_EINVAL, "fl_plan_laplace: need N >= 0 and M >= 0");
    if (N > ((int64_t)1 << 31) - 1 || M > ((int64_t)1 << 31) - 1)
        return lap_fail(FL_EUNSUPPORTED, "fl_plan_laplace: N or M above 2^31 - 1");
    if (!(eps > 0.0 && eps < 1.0)) return lap_fail(FL_EINVAL, "fl_plan_laplace: eps must lie in (0, 1)");
    if (q < 0 || q > kMaxQ) return lap_fail(FL_EINVAL, "fl_plan_laplace: q must lie in [0, 40]");
    if (prec != FL_FP32 && prec != FL_FP64) return lap_fail(FL_EINVAL, "fl_plan_laplace: unknown precision");
    if ((N > 0 && !t_dev) || (M > 0 && !s_dev)) return lap_fail(FL_EINVAL, "fl_plan_laplace: NULL nodes");
    fl_plan_s* h = new (std::nothrow) fl_plan_s();
    if (!h) return lap_fail(FL_ENOMEM, "fl_plan_laplace: host allocation");
    h->p.kind = 1;
    h->p.prec = prec;
    h->p.N = N;
    h->p.M = M;
    h->p.eps = eps;
    fl_status s = plan_laplace_impl(h->p, t_dev, s_dev, q, (cudaStream_t)stream);
    if (s != FL_OK) {
        delete h;
        return s;
    }
    *out = h;
    return FL_OK;
}

fl_status fl_plan_kernel(fl_plan_t* out, int kernel, int64_t N, int64_t M, const double* t_dev,
                         const double* s_dev, int q, double eps, fl_precision prec, void* stream) {
    clear_error();
    if (kernel == FL_KERNEL_LAPLACE) return fl_plan_laplace(out, N, M, t_dev, s_dev, q, eps, prec, stream);
    if (!out) return lap_fail(FL_EINVAL, "fl_plan_kernel: out is NULL");
    *out = nullptr;
    if (kernel != FL_KERNEL_EXP_GENERAL && kernel != FL_KERNEL_BESSEL_K_HALF)
        return lap_fail(FL_EINVAL, "fl_plan_kernel: unknown kernel");
    if (N < 0 || M < 0) return lap_fail(FL_EINVAL, "fl_plan_kernel: need N >= 0 and M >= 0");
    if (N > ((int64_t)1 << 31) - 1 || M > ((int64_t)1 << 31) - 1)
        return lap_fail(FL_EUNSUPPORTED, "fl_plan_kernel: N or M above 2^31 - 1");
    if (!(eps > 0.0 && eps < 1.0)) return lap_fail(FL_EINVAL, "fl_plan_kernel: eps must lie in (0, 1)");
    if (q < 0 || q > kGenMaxQ) return lap_fail(FL_EINVAL, "fl_plan_kernel: q must lie in [0, 64]");
    if (prec != FL_FP32 && prec != FL_FP64) return lap_fail(FL_EINVAL, "fl_plan_kernel: unknown precision");
    if ((N > 0 && !t_dev) || (M > 0 && !s_dev)) return lap_fail(FL_EINVAL, "fl_plan_kernel: NULL nodes");
    fl_plan_s* h = new (std::nothrow) fl_plan_s();
    if (!h) return lap_fail(FL_ENOMEM, "fl_plan_kernel: host allocation");
    h->p.kind = 1;
    h->p.prec = prec;
    h->p.N = N;
    h->p.M = M;
    h->p.eps = eps;
    fl_status s = plan_general_impl(h->p, kernel, t_dev, s_dev, q, (cudaStream_t)stream);
    if (s != FL_OK) {
        delete h;
        return s;
    }
    *out = h;
    return FL_OK;
}

fl_status fl_laplace_real(fl_plan_t h, const void* c_dev, void* f_dev, void* stream) {
    clear_error();
    if (!h || h->p.kind != 1) return lap_fail(FL_EINVAL, "fl_laplace_real: not a Laplace plan");
    if ((h->p.N > 0 && !c_dev) || (h->p.M > 0 && !f_dev))
        return lap_fail(FL_EINVAL, "fl_laplace_real: NULL buffer");
    cudaError_t e = run_laplace(h->p, c_dev, f_dev, (cudaStream_t)stream);
    if (e != cudaSuccess) return lap_fail(FL_ECUDA, std::string("fl_laplace_real: ") + cudaGetErrorString(e));
    return FL_OK;
}


}  // extern "C"

// ---------------------------------------------------------------------------
// Allocation-free variant of fl_laplace_real (fl_laplace_real_noalloc).
//
// Some callers cannot allocate device memory at the point where they need the
// transform: code running inside another framework's memory pool that forbids
// outside allocations, real-time loops where a cudaMalloc (which may
// synchronise the device) is not allowed, or a device that is already full.
// For them every buffer this entry point uses beyond the caller's inputs and
// outputs lives in g_noalloc_scratch, one static device array of
// kNoAllocScratchBytes that each GPU loading libfl.so holds until the process
// exits.  Host code cannot pass the array's name to a kernel (on the host it
// is only a stand-in for the device symbol), so the first call on each device
// looks up its device address with cudaGetSymbolAddress, with that device
// current, and keeps it.
constexpr size_t kNoAllocScratchBytes = (size_t)2 << 20;   // 2 MiB per GPU

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

namespace {

constexpr int kNoAllocMaxDevices = 64;

std::mutex g_noalloc_mutex;
unsigned char* g_noalloc_ptr[kNoAllocMaxDevices] = {};

// Device address of g_noalloc_scratch on the current device (set up once).
fl_status noalloc_scratch(unsigned char** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return set_error(FL_ECUDA, std::string("fl_laplace_real_noalloc: cudaGetDevice: ") +
                                       cudaGetErrorString(e));
    if (dev < 0 || dev >= kNoAllocMaxDevices)
        return set_error(FL_EUNSUPPORTED, "fl_laplace_real_noalloc: device index above 63");
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p)
            return set_error(FL_ECUDA, std::string("fl_laplace_real_noalloc: cudaGetSymbolAddress: ") +
                                           cudaGetErrorString(e));
        g_noalloc_ptr[dev] = (unsigned char*)p;
    }
    *out = g_noalloc_ptr[dev];
    return FL_OK;
}

struct EllArg {
    int v[FL_MAX_LEVELS];
};

__global__ void k_store_ell(EllArg a, int n, int* __restrict__ dst) {
    const int i = threadIdx.x;
    if (i < n) dst[i] = a.v[i];
}

}  // namespace

extern "C" {

fl_status fl_laplace_real_noalloc(int64_t N, int64_t M, const double* t_dev, const double* s_dev,
                                  const void* c_dev, void* f_dev, int q, double eps,
                                  fl_precision prec, void* stream) {
    clear_error();
    if (N < 0 || M < 0) return lap_fail(FL_EINVAL, "fl_laplace_real_noalloc: need N >= 0 and M >= 0");
    if (N > ((int64_t)1 << 31) - 1 || M > ((int64_t)1 << 31) - 1)
        return lap_fail(FL_EUNSUPPORTED, "fl_laplace_real_noalloc: N or M above 2^31 - 1");
    if (!(eps > 0.0 && eps < 1.0))
        return lap_fail(FL_EINVAL, "fl_laplace_real_noalloc: eps must lie in (0, 1)");
    if (q < 0 || q > kMaxQ) return lap_fail(FL_EINVAL, "fl_laplace_real_noalloc: q must lie in [0, 40]");
    if (prec != FL_FP32 && prec != FL_FP64)
        return lap_fail(FL_EINVAL, "fl_laplace_real_noalloc: unknown precision");
    if ((N > 0 && (!t_dev || !c_dev)) || (M > 0 && (!s_dev || !f_dev)))
        return lap_fail(FL_EINVAL, "fl_laplace_real_noalloc: NULL buffer");
    unsigned char* scratch = nullptr;
    fl_status st0 = noalloc_scratch(&scratch);
    if (st0 != FL_OK) return st0;
    cudaStream_t st = (cudaStream_t)stream;

    // [0, 256): interval maxima (2 x u64) and the validity flag; cleared every call
    unsigned long long* dmx = (unsigned long long*)scratch;
    int* dflag = (int*)(scratch + 2 * sizeof(unsigned long long));
    LAP_CUDA(cudaMemsetAsync(scratch, 0, 256, st), "fl_laplace_real_noalloc: clear");
    if (N > 0 || M > 0) k_lap_minmax<<<256, 256, 0, st>>>(N, t_dev, M, s_dev, dmx, dflag);
    LAP_CUDA(cudaGetLastError(), "fl_laplace_real_noalloc: launch");
    unsigned long long mx[2] = {0, 0};
    int flag = 0;
    LAP_CUDA(cudaMemcpyAsync(mx, dmx, sizeof(mx), cudaMemcpyDeviceToHost, st), "fl_laplace_real_noalloc: read");
    LAP_CUDA(cudaMemcpyAsync(&flag, dflag, sizeof(int), cudaMemcpyDeviceToHost, st),
             "fl_laplace_real_noalloc: read");
    LAP_CUDA(cudaStreamSynchronize(st), "fl_laplace_real_noalloc: synchronise");
    if (flag) return lap_fail(FL_EINVAL, "fl_laplace_real_noalloc: a t_k or s_j is negative or not finite");
    double xi1, y1;
    memcpy(&xi1, &mx[0], sizeof(double));
    memcpy(&y1, &mx[1], sizeof(double));
    LapParams P;
    if (!lap_params(eps, q, y1, xi1, &P))
        return lap_fail(FL_EUNSUPPORTED, "fl_laplace_real_noalloc: more than 127 levels or q above 40");
    const size_t tsz = prec == FL_FP64 ? 8 : 4;
    if ((size_t)kLapWarps * (P.levels + 1) * (P.q + 1) * tsz > 200 * 1024)
        return lap_fail(FL_EUNSUPPORTED, "fl_laplace_real_noalloc: moment tables exceed shared memory");

    // [256, 256 + cheb): Chebyshev table; then the Algorithm 1 layout with the
    // partial sums of kLapMaxBlocks moment blocks reserved whatever N is, so
    // whether a problem fits depends on the number of levels and q alone
    const size_t cheb_off = 256;
    const size_t lap_off = align256(cheb_off + 2 * kMaxQ * sizeof(double));
    const int nblocks = lap_blocks(N);
    const LapLayout L = lap_layout(P.levels, P.q, kLapMaxBlocks, tsz);
    if (lap_off + L.total > kNoAllocScratchBytes) {
        char msg[256];
        snprintf(msg, sizeof(msg),
                 "fl_laplace_real_noalloc: this problem needs %zu bytes of scratch (levels = %d, "
                 "q = %d); the static maximum is %zu bytes -- use fl_plan_laplace, a larger eps "
                 "or a smaller max(s) * max(t)",
                 lap_off + L.total, P.levels, P.q, kNoAllocScratchBytes);
        return lap_fail(FL_EUNSUPPORTED, msg);
    }
    double* cheb = (double*)(scratch + cheb_off);
    unsigned char* lap = scratch + lap_off;
    k_lap_cheb<<<1, 64, 0, st>>>(P.q, cheb);
    EllArg ea;
    for (int m = 0; m < FL_MAX_LEVELS; ++m) ea.v[m] = (m < P.levels) ? P.ell[m] : 0;
    k_store_ell<<<1, FL_MAX_LEVELS, 0, st>>>(ea, P.levels + 1, (int*)(lap + L.ell));
    LAP_CUDA(cudaGetLastError(), "fl_laplace_real_noalloc: launch");
    const cudaError_t e =
        prec == FL_FP64 ? noalloc_run<double>(N, M, t_dev, s_dev, P, cheb, (const double*)c_dev, (double*)f_dev, lap,
                                              nblocks, kLapMaxBlocks, st)
                        : noalloc_run<float>(N, M, t_dev, s_dev, P, cheb, (const float*)c_dev, (float*)f_dev, lap,
                                             nblocks, kLapMaxBlocks, st);
    LAP_CUDA(e, "fl_laplace_real_noalloc");
    return FL_OK;
}

}  // extern "C"
