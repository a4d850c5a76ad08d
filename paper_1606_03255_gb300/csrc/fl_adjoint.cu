// fl_adjoint.cu -- the adjoint's own steps: the spreading of the node values onto
// the band grids (the transpose of the window gather, ordered by grid cell, no
// atomics) and the combination of the transformed grids into C^* r.  The FFTs
// between them and the direct bands are those of fl_fft.cuh and fl_direct.cu.
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "fl_ffmath.cuh"
#include "fl_plan.cuh"

namespace fl {

constexpr double kPiAdj = 3.141592653589793238462643383279;
constexpr double kTwoPiAdj = 6.283185307179586476925286766559;

__device__ __forceinline__ float adj_shfl(float v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ double adj_shfl(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ ff adj_shfl(ff v, int o) { return ff(adj_shfl(v.hi, o), adj_shfl(v.lo, o)); }

// ---------------------------------------------------------------------------
// Plan time, per sorted node of an NFFT band of a single plan: its 2 m_w window
// taps, its interpolation weights L_s(y_j), and e_j = exp(-2 pi i (N_m/2) x_j) (1 for
// split bands, whose sub-bands apply their own centre phases; real exponents
// XI: taps at x_j/2 and e_j = exp(-2 pi i xc x_j) / Phi(x_j/2), the conjugate of
// the forward epilogue).  None depends on the values transformed, so an adjoint
// call only forms r_j e_j; the FP64 and float-pair gathers read the taps and
// weights too (they formed about 10^3 FP64 operations of them per node and
// call).  In double, rounded once.  FP32 with integer exponents: in float from
// the node records (X = x 2^64, tau as a pair: in double this would be 1 ms of the
// FP64 pipe at M = 2^18), each fraction the float nearest to 32 bits of X and each
// difference tau - t_s rounded once.  (Fractions cut to 24 bits, as the gather
// has them, turn every node the same way, by 2^-25 turns on average: 1.9e-7 of the
// result.)
__device__ __forceinline__ float adj_turns(uint64_t ph) { return (float)(int32_t)(ph >> 32) * 0x1p-32f; }
__device__ __forceinline__ float adj_difference(float th, float tl, float ch, float cl) {
    const float s = th - ch, z = s - th, e = (th - (s - z)) - (ch + z);   // th - ch = s + e
    return s + (e + (tl - cl));
}

template <int MW>
__global__ void __launch_bounds__(256)
    k_node_tables_f32(int64_t M, const uint4* __restrict__ ntab, const int32_t* __restrict__ bandid,
                      const BandDev* __restrict__ bands, const float* __restrict__ cheb32, int ldl,
                      float* __restrict__ sp_phi, float* __restrict__ sp_L, float2* __restrict__ sp_e) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M) return;
    const BandDev& B = bands[bandid[i]];
    if (B.route != 1) return;
    const uint4 nd = ntab[i];
    const uint64_t X = ((uint64_t)nd.y << 32) | nd.x;
    float2 e = {1.f, 0.f};
    if (B.nsub == 0) {
        e = expipi<float>(-2.f * adj_turns((uint64_t)(B.Nm >> 1) * X));
    }
    sp_e[i] = e;
    const float fr = (float)(uint32_t)((X << B.log2n) >> 32) * 0x1p-32f, kb = (float)B.kb;
#pragma unroll
    for (int t = 0; t < 2 * MW; ++t) sp_phi[i * (2 * MW) + t] = kb_window<float>(fr + (float)(MW - 1 - t), (float)MW, kb);
    if (B.nrhs == 1) return;
    const float th = __uint_as_float(nd.z), tl = __uint_as_float(nd.w);
    const int q = B.nrhs;
    const float* ch = cheb32 + 4 * B.choff;
    float* L = sp_L + i * ldl;
    float den = 0.f;
    int hit = -1;
    for (int s = 0; s < q; ++s) {
        const float d = adj_difference(th, tl, ch[s], ch[q + s]);
        if (d == 0.f) hit = s;
        L[s] = ch[2 * q + s] / d;
        den += L[s];
    }
    const float inv = 1.f / den;
    for (int s = 0; s < q; ++s) L[s] = hit >= 0 ? (s == hit ? 1.f : 0.f) : L[s] * inv;
}

template <typename T, int MW, bool XI>
__global__ void __launch_bounds__(256)
    k_node_taps(int64_t M, const double2* __restrict__ ws, const int32_t* __restrict__ bandid,
                const BandDev* __restrict__ bands, double kb_b, T* __restrict__ sp_phi, C_t<T>* __restrict__ sp_e) {
    const int64_t x0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;   // a thread per node and tap
    const int64_t i = x0 / (2 * MW);
    const int t = (int)(x0 - i * (2 * MW));
    if (i >= M) return;
    const BandDev& B = bands[bandid[i]];
    if (B.route != 1) return;
    const double wx = ws[i].x;
    const double xs = XI ? 0.5 * wx : wx;
    const double x = xs - floor(xs);
    const double t0 = (double)B.n * x;
    const double fr = t0 - floor(t0);
    const double kb = XI ? kb_b : B.kb;
    sp_phi[x0] = sizeof(T) == 8 ? T(kb_window_exact(fr, (double)(MW - 1 - t), (double)MW, kb))
                                : T(kb_window<double>(fr + (double)(MW - 1 - t), (double)MW, kb));
    if (t > 0) return;
    double2 e = {1.0, 0.0};
    if constexpr (XI) {
        const double v = kTwoPiAdj * 0.5 * wx, arg = kb_b * kb_b - v * v;
        const double i0 = cyl_bessel_i0((double)MW * sqrt(arg > 0.0 ? arg : 0.0));
        e = cscale(expipi<double>(-2.0 * frac_turns(B.xc, wx)), 1.0 / (kPiAdj * i0));
    } else if (B.nsub == 0) {
        double ph = (double)(B.Nm >> 1) * x;   // N_m a power of two: exact
        ph -= floor(ph);
        if (ph >= 0.5) ph -= 1.0;
        e = expipi<double>(-2.0 * ph);
    }
    sp_e[i] = C_t<T>{T(e.x), T(e.y)};
}

// The weights, 2^lg lanes per node (at most 32): one division each, the sum of
// the quotients by exchanges.  A thread per node took 78 us for 1024 nodes (q = 18),
// nearly all of it the latency of its divisions and windows in turn.
template <typename T>
__global__ void __launch_bounds__(256)
    k_node_weights(int64_t M, int lg, const double2* __restrict__ ws, const int32_t* __restrict__ bandid,
                   const BandDev* __restrict__ bands, const double* __restrict__ cheb, int ldl, T* __restrict__ sp_L) {
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> lg;
    const int G = 1 << lg, lane = threadIdx.x & (G - 1);
    const BandDev* B = i < M ? &bands[bandid[i]] : nullptr;
    const int q = B && B->route == 1 && B->nrhs > 1 ? B->nrhs : 0;
    const double* ch = q ? cheb + 2 * B->choff : cheb;
    const double tau = q ? (kTwoPiAdj * ws[i].y - B->yc) * B->yh_inv : 0.0;
    static_assert(kMaxQ <= 64, "two weights per lane");
    double w[2] = {0.0, 0.0}, den = 0.0;
    int hit = -1;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int s = lane + k * G;
        if (s >= q) continue;
        const double d = tau - ch[s];
        if (d == 0.0) hit = s;
        w[k] = ch[q + s] / d;
        den += w[k];
    }
    for (int off = G >> 1; off > 0; off >>= 1) {
        den += __shfl_xor_sync(0xffffffffu, den, off);
        hit = max(hit, __shfl_xor_sync(0xffffffffu, hit, off));
    }
    const double inv = 1.0 / den;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int s = lane + k * G;
        if (s < q) sp_L[i * ldl + s] = T(hit >= 0 ? (s == hit ? 1.0 : 0.0) : w[k] * inv);
    }
}

// rv_j = r_j e_j in sorted order.
template <typename A, typename O>
__global__ void __launch_bounds__(256)
    k_spread_rv(int64_t M, const int32_t* __restrict__ perm, const int32_t* __restrict__ bandid,
                const BandDev* __restrict__ bands, const O* __restrict__ r, const C_t<A>* __restrict__ sp_e,
                C_t<A>* __restrict__ sp_rv) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M) return;
    const BandDev& B = bands[bandid[i]];
    if (B.route != 1) return;
    const O v = r[perm[i]];
    const C_t<A> rv = C_t<A>{A(v.x), A(v.y)};
    sp_rv[i] = B.nsub > 0 ? rv : cmul(rv, sp_e[i]);
}

// exp(-2 pi i kc x_j) of a sub-band's centre kc (float pairs have no sub-bands).
__device__ __forceinline__ float2 adj_phase(int64_t kc, const uint4* __restrict__ ntab, const double2*, int64_t j,
                                            float) {
    const uint4 nd = ntab[j];
    const uint64_t X = ((uint64_t)nd.y << 32) | nd.x;
    return expipi<float>(-2.f * adj_turns((uint64_t)kc * X));
}
__device__ __forceinline__ double2 adj_phase(int64_t kc, const uint4*, const double2* __restrict__ ws, int64_t j,
                                             double) {
    const double x = ws[j].x - floor(ws[j].x);
    return expipi<double>(-2.0 * frac_turns((double)kc, x));
}
__device__ __forceinline__ ffc adj_phase(int64_t, const uint4*, const double2*, int64_t, ff) {
    return ffc{ff(1), ff(0)};
}

// ---------------------------------------------------------------------------
// Spreading: a_s[l] = sum_j phi_j[l - u_j + m_w - 1] rv_j L_s(y_j) over the nodes whose
// cell u_j covers grid cell l (mod n), every grid cell written once, the sums in
// node order.  k_spread_sparse (fewer than one node per cell): a block takes
// 256 / SG consecutive cells of a band, its threads one cell and 8 of the
// right-hand sides each (SG = 2^lg covers them all); the block's nodes (a
// plan-time range: consecutive in cell order) are staged in shared memory with
// their taps, weights and phased values, and a thread sums its few covering
// nodes in registers.  A thread per cell that searched its nodes and kept all
// sums in local memory took 430 us for 4.3*10^6 cells at 300007 x 250001 (97 us
// now); blocks of 256 cells that went over the right-hand sides in turn, staging
// again, 318 us for 1.6*10^6.  On the 2^18 disk nodes 40 % of the issue slots and
// 34 % of L1 are used, with the staging loads' latency beside them.
constexpr int kSpThreads = 256, kSpTile = 128, kSpQ = 8;

template <typename T> static size_t sp_smem(int mw, int q) {
    return (size_t)kSpTile * (sizeof(C_t<T>) + (2 * mw + q) * sizeof(T) + sizeof(int));
}

template <typename T, int MW>
__global__ void __launch_bounds__(kSpThreads)
    k_spread_sparse(const int4* __restrict__ blocks, int nbands, const int4* __restrict__ ranges,
                    const BandDev* __restrict__ bands, const int32_t* __restrict__ cell,
                    const T* __restrict__ sp_phi, const T* __restrict__ sp_L, const C_t<T>* __restrict__ sp_rv,
                    const uint4* __restrict__ ntab, const double2* __restrict__ ws, int ldl,
                    C_t<T>* __restrict__ grid) {
    using C = C_t<T>;
    extern __shared__ unsigned char smem_raw[];
    const int4 rg = ranges[blockIdx.x];             // main [x, y), wrapped [z, nend) before, [nb0, w) after
    int lo = 0, hi = nbands;                        // last band with first block <= blockIdx.x
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (blocks[mid].x <= (int)blockIdx.x) lo = mid;
        else hi = mid;
    }
    const int4 bl = blocks[lo];
    const BandDev& B = bands[bl.y];
    const int lg = bl.z, cells = kSpThreads >> lg;
    const int nr = B.nrhs, n = (int)B.n;
    const int c0 = ((int)blockIdx.x - bl.x) * cells;
    const int nb0 = (int)B.node_off, nend = (int)(B.node_off + B.nodes);
    const int npre = nend - rg.z, nmain = rg.y - rg.x, npost = rg.w - nb0;
    const int cnt = npre + nmain + npost;
    const int64_t kc = B.k0 + (B.Nm >> 1);
    const bool sub = B.parent >= 0;
    C* sw = reinterpret_cast<C*>(smem_raw);
    T* sphi = reinterpret_cast<T*>(sw + kSpTile);
    T* sL = sphi + kSpTile * 2 * MW;
    int* sdu = reinterpret_cast<int*>(sL + nr * kSpTile);
    const int l = threadIdx.x & (cells - 1), s0 = (threadIdx.x / cells) * kSpQ;
    const int wl = 3 + lg, wm = (1 << wl) - 1;      // SG * 8 weights per node, as a power of two
    auto node = [&](int k) {
        return k < npre ? rg.z + k : k < npre + nmain ? rg.x + (k - npre) : nb0 + (k - npre - nmain);
    };
    C acc[kSpQ];
#pragma unroll
    for (int u = 0; u < kSpQ; ++u) acc[u] = C{T(0), T(0)};
    for (int b0 = 0; b0 < cnt; b0 += kSpTile) {
        const int tn = min(kSpTile, cnt - b0);
        if (b0 > 0) __syncthreads();                // the tile before has been read
        if (threadIdx.x < tn) {
            const int e = threadIdx.x, k = b0 + e, j = node(k);
            sdu[e] = cell[j] - c0 + (k < npre ? -n : k < npre + nmain ? 0 : n);
            C w = sp_rv[j];
            if (sub) w = cmul(w, adj_phase(kc, ntab, ws, j, T(0)));
            sw[e] = w;
        }
#pragma unroll 4
        for (int x = threadIdx.x; x < tn * 2 * MW; x += kSpThreads)
            sphi[x] = sp_phi[(int64_t)node(b0 + x / (2 * MW)) * (2 * MW) + x % (2 * MW)];
        if (nr > 1) {
#pragma unroll 4
            for (int x = threadIdx.x; x < tn << wl; x += kSpThreads)
                if ((x & wm) < nr) sL[(x >> wl) * nr + (x & wm)] = sp_L[(int64_t)node(b0 + (x >> wl)) * ldl + (x & wm)];
        }
        __syncthreads();
        if (s0 < nr) {
            int a = 0, z = tn;                      // the staged nodes with du in [l - m_w, l + m_w - 1]
            while (a < z) {
                const int mid = (a + z) >> 1;
                if (sdu[mid] < l - MW) a = mid + 1;
                else z = mid;
            }
            for (int e = a; e < tn; ++e) {
                const int t = l - sdu[e] + MW - 1;
                if (t < 0) break;
                if (t >= 2 * MW) continue;
                const C w = cscale(sw[e], sphi[e * 2 * MW + t]);
                if (nr == 1) {
                    acc[0] = cadd(acc[0], w);
                    continue;
                }
                const T* L = sL + e * nr + s0;
#pragma unroll
                for (int u = 0; u < kSpQ; ++u) {
                    const T Lu = s0 + u < nr ? L[u] : T(0);
                    acc[u].x += Lu * w.x;
                    acc[u].y += Lu * w.y;
                }
            }
        }
    }
    if (c0 + l >= n) return;
    C* out = grid + B.grid_off + c0 + l + (int64_t)s0 * n;
#pragma unroll
    for (int u = 0; u < kSpQ; ++u)
        if (s0 + u < nr) out[(int64_t)u * n] = acc[u];
}

// v[0 .. 2 H) summed over the lanes by halving: in step OFF a lane keeps one half
// of its values and takes its partner's sums of that half.
template <int H, int OFF, typename T> __device__ __forceinline__ void adj_halve(T* v, int lane) {
    if constexpr (OFF > 0) {
        static_assert(H > 0, "at least 32 values");
        const bool up = lane & OFF;
#pragma unroll
        for (int i = 0; i < H; ++i) {
            const T give = up ? v[i] : v[i + H];
            const T keep = up ? v[i + H] : v[i];
            v[i] = keep + adj_shfl(give, OFF);
        }
        adj_halve<H / 2, OFF / 2>(v, lane);
    }
}

// Dense bands (at least one node per cell): CG neighbouring cells x 8 right-hand
// sides per warp (WPG = 1), or per CTA where the covering nodes are several
// hundred (WPG = 8); the lanes stride over the nodes (plan-time cell starts), the
// sums in registers -- a node's weights are read once for CG cells -- then a
// halving exchange, and the warps in order.  Bound by load latency at 20 % of
// the warps (115 registers): 17 and 20 us on the 2^18 disk nodes in FP32, where a CTA
// per cell with the sums in local memory took 82 us (222 us in pairs).
template <typename T> struct SpreadDense {
    static constexpr int CG = sizeof(T) == 4 ? 4 : 2;
};

template <typename T, int MW, int WPG>
__global__ void __launch_bounds__(256)
    k_spread_dense(const int4* __restrict__ groups, int nbands, const int32_t* __restrict__ start,
                   const BandDev* __restrict__ bands, const int32_t* __restrict__ cell,
                   const T* __restrict__ sp_phi, const T* __restrict__ sp_L, const C_t<T>* __restrict__ sp_rv,
                   const uint4* __restrict__ ntab, const double2* __restrict__ ws, int ldl,
                   C_t<T>* __restrict__ grid) {
    using C = C_t<T>;
    constexpr int CG = SpreadDense<T>::CG, P = 2 * CG * kSpQ, NT = 32 * WPG;
    __shared__ T red[8][P];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int gid = WPG == 8 ? (int)blockIdx.x : (int)blockIdx.x * 8 + w;   // (8 groups of one band per block)
    int lo = 0, hi = nbands;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (groups[mid].x <= gid) lo = mid;
        else hi = mid;
    }
    const int4 gr = groups[lo];
    const BandDev& B = bands[gr.y];
    const int nr = B.nrhs, n = (int)B.n, s0 = blockIdx.y * kSpQ;
    if (s0 >= nr) return;                           // uniform over the block
    const int l0 = (gid - gr.x) * CG;
    const int32_t* st = start + gr.z;               // st[l]: first node of the band with cell >= l, l = 0 .. n
    const int64_t kc = B.k0 + (B.Nm >> 1);
    const bool sub = B.parent >= 0;
    T v[P];
#pragma unroll
    for (int i = 0; i < P; ++i) v[i] = T(0);
    const int a = l0 - MW, z = l0 + CG - 1 + MW;   // cells [a, z) mod n (n >= 32 > their number)
    for (int part = 0; part < 2; ++part) {
        int j0, j1;
        if (part == 0) {
            j0 = st[max(a, 0)];
            j1 = st[min(z, n)];
        } else if (a < 0) {
            j0 = st[n + a];
            j1 = st[n];
        } else if (z > n) {
            j0 = st[0];
            j1 = st[z - n];
        } else {
            break;
        }
        for (int j = j0 + (WPG == 8 ? (int)threadIdx.x : lane); j < j1; j += NT) {
            int t0 = l0 - cell[j] + MW - 1;        // tap of cell l0
            if (part == 1) t0 += a < 0 ? n : -n;
            C wv = sp_rv[j];
            if (sub) wv = cmul(wv, adj_phase(kc, ntab, ws, j, T(0)));
            C wc[CG];
#pragma unroll
            for (int g = 0; g < CG; ++g) {
                const int t = t0 + g;
                const T ph = t >= 0 && t < 2 * MW ? sp_phi[(int64_t)j * (2 * MW) + t] : T(0);
                wc[g] = cscale(wv, ph);
            }
#pragma unroll
            for (int u = 0; u < kSpQ; ++u) {
                if (s0 + u >= nr) break;
                const T L = nr > 1 ? sp_L[(int64_t)j * ldl + s0 + u] : T(1);
#pragma unroll
                for (int g = 0; g < CG; ++g) {
                    v[2 * (g * kSpQ + u)] += L * wc[g].x;
                    v[2 * (g * kSpQ + u) + 1] += L * wc[g].y;
                }
            }
        }
    }
    adj_halve<P / 2, 16>(v, lane);
    int e0 = 0;
#pragma unroll
    for (int h = P / 2, off = 16; off > 0; h >>= 1, off >>= 1)
        if (lane & off) e0 += h;
#pragma unroll
    for (int i = 0; i < P / 32; ++i) red[w][e0 + i] = v[i];
    if constexpr (WPG == 8) __syncthreads();
    else __syncwarp();
    const int e = WPG == 8 ? (int)threadIdx.x : lane;   // (cell g, right-hand side u) of this thread
    for (int x = e; x < CG * kSpQ; x += NT) {
        if (s0 + x % kSpQ >= nr) continue;
        const T* r0 = red[WPG == 8 ? 0 : w];
        C sum = {r0[2 * x], r0[2 * x + 1]};
        if constexpr (WPG == 8)
            for (int ww = 1; ww < 8; ++ww) sum = cadd(sum, C{red[ww][2 * x], red[ww][2 * x + 1]});
        grid[B.grid_off + l0 + x / kSpQ + (int64_t)(s0 + x % kSpQ) * n] = sum;
    }
}

// Plan time.  First node of [lo, hi) with cell >= v (cells ascend within a band).
__device__ __forceinline__ int adj_lower(const int32_t* __restrict__ cell, int lo, int hi, int v) {
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (cell[mid] < v) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

__global__ void k_spread_ranges(int nblocks, const int4* __restrict__ blocks, int nbands,
                                const BandDev* __restrict__ bands, const int32_t* __restrict__ cell, int mw,
                                int4* __restrict__ ranges) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nblocks) return;
    int lo = 0, hi = nbands;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (blocks[mid].x <= b) lo = mid;
        else hi = mid;
    }
    const BandDev& B = bands[blocks[lo].y];
    const int cells = kSpThreads >> blocks[lo].z;
    const int n = (int)B.n, c0 = (b - blocks[lo].x) * cells, c1 = min(c0 + cells, n);
    const int j0 = (int)B.node_off, j1 = (int)(B.node_off + B.nodes);
    int4 r;
    r.x = adj_lower(cell, j0, j1, c0 - mw);
    r.y = adj_lower(cell, j0, j1, c1 - 1 + mw);        // cells <= c1 - 1 + m_w - 1
    r.z = c0 == 0 ? adj_lower(cell, j0, j1, n - mw) : j1;
    r.w = c1 == n ? adj_lower(cell, j0, j1, mw - 1) : j0;   // cells <= m_w - 2, shifted by n
    ranges[b] = r;
}

// start[z + l], l = 0 .. n, of every dense band {first group, band, z, n}
__global__ void k_spread_starts(int total, const int4* __restrict__ groups, int nbands,
                                const BandDev* __restrict__ bands, const int32_t* __restrict__ cell,
                                int32_t* __restrict__ start) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    int lo = 0, hi = nbands;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (groups[mid].z <= i) lo = mid;
        else hi = mid;
    }
    const BandDev& B = bands[groups[lo].y];
    start[i] = adj_lower(cell, (int)B.node_off, (int)(B.node_off + B.nodes), i - groups[lo].z);
}

template <typename E> static cudaError_t adj_upload(Plan& p, const std::vector<E>& v, E** dev, cudaStream_t st) {
    if (v.empty()) return cudaSuccess;
    cudaError_t e = p.pool.get(dev, (int64_t)v.size());
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(*dev, v.data(), v.size() * sizeof(E), cudaMemcpyHostToDevice, st);
    return e;
}

cudaError_t build_spread(Plan& p, cudaStream_t st) {
    const int cg = p.prec == FL_FP32 ? SpreadDense<float>::CG : SpreadDense<double>::CG;
    static_assert(SpreadDense<double>::CG == SpreadDense<ff>::CG, "one group size per element size");
    std::vector<int4> blocks, warps, wide;   // sparse bands, dense ones by warp and by CTA
    int64_t nblocks = 0, nwarps = 0, nwide = 0, nstart = 0;
    std::vector<CombineItem> comb;
    for (int b = 0; b < (int)p.bands.size(); ++b) {
        const BandHost& bh = p.bands[b];
        const BandDev& d = bh.dev;
        if (d.route != 1 || d.nsub > 0) continue;
        comb.push_back({d.k0, d.K, d.D_off, d.grid_off, d.Nm / 2, d.n, d.nrhs, 0});
        if (bh.nodes < d.n) {
            int lg = 0;
            while (kSpQ << lg < d.nrhs) ++lg;
            const int cells = kSpThreads >> lg;
            blocks.push_back(make_int4((int)nblocks, b, lg, 0));
            nblocks += (d.n + cells - 1) / cells;
        } else if (bh.nodes * (cg - 1 + 2 * p.mw) < 512 * d.n) {
            warps.push_back(make_int4((int)nwarps, b, 0, 0));
            nwarps += d.n / cg;                    // a multiple of 8 (n >= 32)
        } else {
            wide.push_back(make_int4((int)nwide, b, 0, 0));
            nwide += d.n / cg;
        }
    }
    p.n_sp_bands = (int)blocks.size();
    p.n_sp_blocks = nblocks;
    p.n_dn_bands[0] = (int)warps.size();
    p.n_dn_groups[0] = nwarps;
    p.n_dn_bands[1] = (int)wide.size();
    p.n_dn_groups[1] = nwide;
    p.n_comb = (int)comb.size();
    std::vector<int4> groups = warps;
    groups.insert(groups.end(), wide.begin(), wide.end());
    for (int4& g : groups) {
        g.z = (int)nstart;
        nstart += p.bands[g.y].dev.n + 1;
    }
    cudaError_t e = adj_upload(p, blocks, &p.d_sp_blocks, st);
    if (e == cudaSuccess) e = adj_upload(p, groups, &p.d_dn_groups, st);
    if (e == cudaSuccess) e = adj_upload(p, comb, &p.d_comb, st);
    if (e == cudaSuccess && nblocks > 0) {
        e = p.pool.bytes((void**)&p.d_sp_ranges, nblocks * sizeof(int4));
        if (e == cudaSuccess)
            k_spread_ranges<<<(unsigned)((nblocks + 255) / 256), 256, 0, st>>>(
                (int)nblocks, p.d_sp_blocks, p.n_sp_bands, p.d_bands, p.d_cell, p.mw, p.d_sp_ranges);
    }
    if (e == cudaSuccess && nstart > 0) {
        e = p.pool.bytes((void**)&p.d_dn_start, nstart * sizeof(int32_t));
        if (e == cudaSuccess)
            k_spread_starts<<<(unsigned)((nstart + 255) / 256), 256, 0, st>>>(
                (int)nstart, p.d_dn_groups, (int)groups.size(), p.d_bands, p.d_cell, p.d_dn_start);
    }
    return e == cudaSuccess ? cudaGetLastError() : e;
}

template <typename T, int MW> static cudaError_t node_tables_t(Plan& p, cudaStream_t st) {
    if constexpr (sizeof(T) == 4) {
        if (!p.xi_mode) {
            k_node_tables_f32<MW><<<(unsigned)((p.M + 255) / 256), 256, 0, st>>>(
                p.M, p.d_ntab, p.d_bandid, p.d_bands, p.d_cheb32, p.qmax, (T*)p.d_sp_phi, (T*)p.d_sp_L,
                (C_t<T>*)p.d_sp_e);
            return cudaGetLastError();
        }
    }
    auto kern = p.xi_mode ? k_node_taps<T, MW, true> : k_node_taps<T, MW, false>;
    kern<<<(unsigned)((p.M * 2 * MW + 255) / 256), 256, 0, st>>>(p.M, p.d_ws, p.d_bandid, p.d_bands, p.kb_b,
                                                                  (T*)p.d_sp_phi, (C_t<T>*)p.d_sp_e);
    int lg = 0;
    while (lg < 5 && (1 << lg) < p.qmax) ++lg;
    k_node_weights<T><<<(unsigned)(((p.M << lg) + 255) / 256), 256, 0, st>>>(p.M, lg, p.d_ws, p.d_bandid, p.d_bands,
                                                                             p.d_cheb, p.qmax, (T*)p.d_sp_L);
    return cudaGetLastError();
}

template <typename T, int MW>
static cudaError_t spread_t(Plan& p, const void* r, cudaStream_t st) {
    using C = C_t<T>;
    using O = std::conditional_t<sizeof(T) == 4, float2, double2>;
    if (p.n_sp_blocks + p.n_dn_groups[0] + p.n_dn_groups[1] == 0) return cudaSuccess;
    int slot;
    timer_begin(p, "spread", 0.0, st, &slot);
    k_spread_rv<T, O><<<(unsigned)((p.M + 255) / 256), 256, 0, st>>>(
        p.M, p.d_perm, p.d_bandid, p.d_bands, (const O*)r, (const C*)p.d_sp_e, (C*)p.d_sp_rv);
    if (p.n_sp_blocks > 0) {
        const size_t smem = sp_smem<T>(MW, p.qmax);    // FP64 and pairs: up to 67 KiB
        cudaError_t e = cudaFuncSetAttribute(k_spread_sparse<T, MW>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
        k_spread_sparse<T, MW><<<(unsigned)p.n_sp_blocks, kSpThreads, smem, st>>>(
            p.d_sp_blocks, p.n_sp_bands, p.d_sp_ranges, p.d_bands, p.d_cell, (const T*)p.d_sp_phi,
            (const T*)p.d_sp_L, (const C*)p.d_sp_rv, p.d_ntab, p.d_ws, p.qmax, (C*)p.d_grid);
    }
    const unsigned chunks = (unsigned)((p.qmax + kSpQ - 1) / kSpQ);
    for (int k = 0; k < 2; ++k) {
        if (p.n_dn_groups[k] == 0) continue;
        auto kern = k == 0 ? k_spread_dense<T, MW, 1> : k_spread_dense<T, MW, 8>;
        const dim3 g((unsigned)(k == 0 ? p.n_dn_groups[0] / 8 : p.n_dn_groups[1]), chunks);
        kern<<<g, 256, 0, st>>>(p.d_dn_groups + (k == 0 ? 0 : p.n_dn_bands[0]), p.n_dn_bands[k], p.d_dn_start,
                                p.d_bands, p.d_cell, (const T*)p.d_sp_phi, (const T*)p.d_sp_L,
                                (const C*)p.d_sp_rv, p.d_ntab, p.d_ws, p.qmax, (C*)p.d_grid);
        ++p.launches;
    }
    timer_end(p, slot, st);
    p.launches += 1 + (p.n_sp_blocks > 0);
    return cudaGetLastError();
}

template <typename T> static cudaError_t spread_dispatch(Plan& p, const void* r, bool tables, cudaStream_t st) {
    switch (p.mw) {
#define FL_MW_CASE(W) \
    case W: return tables ? node_tables_t<T, W>(p, st) : spread_t<T, W>(p, r, st);
        FL_MW_CASE(2) FL_MW_CASE(3) FL_MW_CASE(4) FL_MW_CASE(5) FL_MW_CASE(6) FL_MW_CASE(7)
        FL_MW_CASE(8) FL_MW_CASE(9) FL_MW_CASE(10) FL_MW_CASE(11) FL_MW_CASE(12)
#undef FL_MW_CASE
        default: return cudaErrorInvalidValue;
    }
}

static cudaError_t spread_any(Plan& p, const void* r, bool tables, cudaStream_t st) {
    if (p.prec == FL_FP64_FF) return spread_dispatch<ff>(p, r, tables, st);
    return p.prec == FL_FP64 ? spread_dispatch<double>(p, r, tables, st)
                             : spread_dispatch<float>(p, r, tables, st);
}

cudaError_t build_node_weights(Plan& p, cudaStream_t st) { return spread_any(p, nullptr, true, st); }
cudaError_t launch_spread(Plan& p, const void* r, cudaStream_t st) { return spread_any(p, r, false, st); }

// ---------------------------------------------------------------------------
// Sum of r over the Z^0 nodes (the first z0 sorted nodes): out gets it.
template <typename T>
__global__ void k_z0_sum(int64_t z0, const int32_t* __restrict__ perm,
                         const C_t<T>* __restrict__ r, C_t<T>* __restrict__ out) {
    __shared__ T sx[256], sy[256];
    T ax = 0, ay = 0;
    for (int64_t i = threadIdx.x; i < z0; i += 256) {
        const C_t<T> v = r[perm[i]];
        ax += v.x;
        ay += v.y;
    }
    sx[threadIdx.x] = ax;
    sy[threadIdx.x] = ay;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (threadIdx.x < h) {
            sx[threadIdx.x] += sx[threadIdx.x + h];
            sy[threadIdx.x] += sy[threadIdx.x + h];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = C_t<T>{sx[0], sy[0]};
}

// c_out[k] = [k == 0] z0sum + cdir[k] + sum over the grids of sum_s D[s][k - k0]
// b_s[(k - k0 - N_m/2) mod n], one thread per k over a plan-time list of the grids
// (three fields decide whether a grid holds k; the walk over the band table
// read 200 bytes per band and thread).  Bound by the latency of its loads of D and
// the grids (N = M = 2^18 FP32: 23 warps waiting on them per issue, DRAM at 12 % of its
// peak); the sums in the plan's arithmetic.  Float pairs: in pairs, where double took
// 185 us of FP64 conversions and products at N = 2^18; a term adds a rounding of
// 2^-46 of the sum of the terms' magnitudes, so the up to 130 terms of a frequency
// add 130^(1/2) 2^-46 = 1.6e-13 of it, below the 2^-46 of each of the 40 layers of
// FFTs times the gain of 8.6 before it (measured: 4.6e-14 at N = M = 2^18, eps = 1e-12).
template <typename A, typename O>
__global__ void __launch_bounds__(128)
    k_combine(int64_t N, int n_items, const CombineItem* __restrict__ items, const A* __restrict__ D,
              const C_t<A>* __restrict__ grid, const O* __restrict__ z0sum, const O* __restrict__ cdir,
              O* __restrict__ cout) {
    using C = C_t<A>;
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= N) return;
    C acc = {A(0), A(0)};
    for (int it = 0; it < n_items; ++it) {
        const int64_t kl = k - items[it].k0;
        if ((uint64_t)kl >= (uint64_t)items[it].K) continue;
        const CombineItem I = items[it];
        const A* Dk = D + I.D_off + kl;
        const C* g = grid + I.grid_off + ((kl - I.half) & (I.n - 1));
#pragma unroll 4
        for (int s = 0; s < I.nrhs; ++s) {
            const A d = Dk[(int64_t)s * I.K];
            const C v = g[(int64_t)s * I.n];
            acc.x += d * v.x;
            acc.y += d * v.y;
        }
    }
    O out;
    if constexpr (std::is_same<A, ff>::value) out = O{(double)acc.x, (double)acc.y};
    else out = acc;
    if (cdir) out = cadd(out, cdir[k]);
    if (k == 0 && z0sum) out = cadd(out, *z0sum);
    cout[k] = out;
}

template <typename A, typename O>
static cudaError_t combine_t(Plan& p, const void* r, void* cout, cudaStream_t st) {
    using R = decltype(O().x);
    const O* z0sum = nullptr;
    if (p.z0_nodes > 0) {
        k_z0_sum<R><<<1, 256, 0, st>>>(p.z0_nodes, p.d_perm, (const O*)r, (O*)p.d_z0);
        z0sum = (const O*)p.d_z0;
        ++p.launches;
    }
    int slot;
    timer_begin(p, "combine", 0.0, st, &slot);
    k_combine<A, O><<<(unsigned)((p.N + 127) / 128), 128, 0, st>>>(
        p.N, p.n_comb, p.d_comb, (const A*)p.d_D, (const C_t<A>*)p.d_grid, z0sum,
        p.dadj_work.empty() ? nullptr : (const O*)p.d_cdir, (O*)cout);
    timer_end(p, slot, st);
    ++p.launches;
    return cudaGetLastError();
}

cudaError_t launch_combine(Plan& p, const void* r, void* cout, cudaStream_t st) {
    if (p.prec == FL_FP64_FF) return combine_t<ff, double2>(p, r, cout, st);
    return p.prec == FL_FP64 ? combine_t<double, double2>(p, r, cout, st)
                             : combine_t<float, float2>(p, r, cout, st);
}

}  // namespace fl
