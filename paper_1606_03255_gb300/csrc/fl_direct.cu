// fl_direct.cu -- direct evaluation of the bands whose node count is too small
// to pay for an NFFT with q right-hand sides, and of their adjoint.
//
// A band routed here computes the plain sum f_j = sum_{k<K} c_k z_j^k over the
// frequencies the band keeps (K = k <= xi_1 / 2^(l_m - 1), the region-(ii)
// truncation of Lemma A.2, or K = N for the Y_M band), i.e. eq. (4.1) itself
// -- the "naive matrix vector multiplication" the paper times in Section 5 --
// restricted to those frequencies.  The sum is blocked: each block of 32 terms
// is evaluated as four Horner polynomials of eight terms in z_j, combined by
// Horner in z_j^8 -- as many steps as one chain of 32, in four independent
// ones, and the rounding of z_j enters with its 7th power instead of its 31st
// (z_j and z_j^8 are rounded once at plan time).  z_j^{k_b} at the block start
// is formed from an exactly reduced phase (k_b x_j mod 1) and exp(-y_j k_b), so
// the error does not grow with k.
//
// Neighbouring direct bands with the same K are one segment (their nodes are
// consecutive in sorted order), so a handful of nodes per band still shares a
// work item.  The arithmetic is float, double or float pairs (A below).
#include <algorithm>
#include <type_traits>

#include "fl_f32x2.cuh"
#include "fl_ffmath.cuh"
#include "fl_plan.cuh"

namespace fl {

constexpr double kTwoPiDir = 6.283185307179586476925286766559;

// Shared-memory stride of a staged Horner block: one element of padding, so
// lanes on different blocks read different bank offsets (blocks of 32 complex
// values are 256 or 512 bytes apart, a whole number of bank rows).
constexpr int kDirBlockLd = kDirBlock + 1;

static size_t dir_tile(int64_t kmax, size_t csize) {
    const int64_t k = std::min<int64_t>(kmax, kDirChunk);
    return (size_t)((k + kDirBlock - 1) / kDirBlock * kDirBlockLd) * csize;
}

// FP32 form without FP64 arithmetic per block: x in [0, 1) held as the 64-bit
// fixed-point X = x 2^64 (exact for the 53-bit x), so frac(k x) is the
// wrapped product k X, read as a signed value in [-1/2, 1/2); y as a float pair
// (hi + lo), so y k = p + e with p = fl(hi k) and e its error plus lo k, and
// exp(-y k) = exp(-p) (1 - e) (|e| < 2^-20 p).
struct DirF32Node {
    uint64_t X;
    float yh, yl;
};

// z^k = exp(-y k) e^(2 pi i frac(k x)) for 0 <= k < 2^24 (SIGN = -1: the conjugate
// phase); false when y k > lim (the power underflows: so do all later ones).
// The phase is the float nearest to the top 32 bits of the product; pin: to its
// top 24 bits, half up, the rounding of pinned transforms (kPinnedN).
template <int SIGN>
__device__ __forceinline__ bool dir_f32_power(const DirF32Node& d, int64_t k, float lim, bool pin, float2* zk) {
    const float kf = (float)k;                 // exact: k < 2^24
    const float p = d.yh * kf;
    if (p > lim) return false;
    const float e = fmaf(d.yh, kf, -p) + d.yl * kf;
    const float mag = expf(-p) * (1.f - e);
    const uint64_t ph = (uint64_t)k * d.X;
    const float phase = pin ? (float)((int64_t)(ph + (1ull << 39)) >> 40) * 0x1p-24f
                            : (float)(int32_t)(ph >> 32) * 0x1p-32f;
    *zk = cscale(expipi<float>((float)(2 * SIGN) * phase), mag);
    return true;
}

// A node as the powers need it: from the plan-time record (X = x 2^64, y =
// 2 pi Im w as a float pair, k_node_tab) in the FP32 form, from the sorted
// nodes otherwise.
template <typename A> struct DirNode {
    double x, y;
};
template <> struct DirNode<float> {
    DirF32Node d;
};
template <typename A>
__device__ __forceinline__ DirNode<A> dir_node(const double2* __restrict__ ws, const uint4* __restrict__ ntab,
                                               int64_t i) {
    DirNode<A> n;
    if constexpr (sizeof(A) == 4) {
        const uint4 rec = ntab[i];
        n.d.X = ((uint64_t)rec.y << 32) | (uint64_t)rec.x;
        n.d.yh = __uint_as_float(rec.z);
        n.d.yl = __uint_as_float(rec.w);
    } else {
        const double2 wv = ws[i];
        n.x = wv.x - floor(wv.x);
        n.y = kTwoPiDir * wv.y;
    }
    return n;
}

// z^k (SIGN = -1: its conjugate); false once the power underflows.  Double and
// float pairs reduce k x mod 1 exactly (FMA) in double.
template <int SIGN>
__device__ __forceinline__ bool dir_power(const DirNode<float>& n, int64_t k, float2* zk, bool pin = false) {
    return dir_f32_power<SIGN>(n.d, k, 104.f, pin, zk);
}
template <int SIGN> __device__ __forceinline__ bool dir_power(const DirNode<double>& n, int64_t k, double2* zk) {
    const double yk = n.y * (double)k;
    if (yk > 745.0) return false;
    *zk = cscale(expipi<double>((double)(2 * SIGN) * frac_turns((double)k, n.x)), exp(-yk));
    return true;
}
template <int SIGN> __device__ __forceinline__ bool dir_power(const DirNode<ff>& n, int64_t k, ffc* zk) {
    const double yk = n.y * (double)k;
    if (yk > 104.0) return false;   // below 2^-150 |c|
    ff_sincospi(ff((double)(2 * SIGN) * frac_turns((double)k, n.x)), &zk->y, &zk->x);
    const ff mk = ff_exp(ff(-yk));
    *zk = ffc{zk->x * mk, zk->y * mk};
    return true;
}

// z = exp(-y) e^(2 pi i x) of a pinned transform, in float from the record: x - [x >= 1/2]
// is the signed X 2^-64, rounded once.
__device__ __forceinline__ float2 dir_f32_base(const DirF32Node& d) {
    const float xr = (float)(int64_t)d.X * 0x1p-64f;
    return cscale(expipi<float>(2.f * xr), expf(-d.yh));
}

// Plan time: z_j and z_j^8 (entries 2 t and 2 t + 1 of the t-th node with a base),
// formed in double and rounded once.
template <typename A> __device__ __forceinline__ C_t<A> dir_round(double2 v) { return {A(v.x), A(v.y)}; }
template <typename A>
__global__ void k_dir_base(int64_t total, const DirectSeg* __restrict__ segs, int nsegs,
                           const double2* __restrict__ ws, C_t<A>* __restrict__ z) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= total) return;
    int lo = 0, hi = nsegs;                      // last segment whose first base is <= t
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (segs[mid].node_off + segs[mid].z_off <= t) lo = mid;
        else hi = mid;
    }
    const DirNode<double> n = dir_node<double>(ws, nullptr, t - segs[lo].z_off);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const double k = e ? 8.0 : 1.0;
        z[2 * t + e] = dir_round<A>(cscale(expipi<double>(2.0 * frac_turns(k, n.x)), exp(-n.y * k)));
    }
}

// One Horner step P z + c: four fused operations (double), or the pairs' own.
__device__ __forceinline__ double2 dir_step(double2 P, double2 z, double2 c) {
    return {fma(P.x, z.x, fma(-P.y, z.y, c.x)), fma(P.x, z.y, fma(P.y, z.x, c.y))};
}
__device__ __forceinline__ ffc dir_step(ffc P, ffc z, ffc c) { return cadd(cmul(P, z), c); }
struct f2c {   // two nodes' complex values in packed pairs
    f2 x, y;
};
__device__ __forceinline__ f2c dir_step(f2c P, f2c z, f2 nzy, f2c c) {
    return {f2_fma(P.x, z.x, f2_fma(P.y, nzy, c.x)), f2_fma(P.x, z.y, f2_fma(P.y, z.x, c.y))};
}
// The steps of pinned transforms (kPinnedN): products and sums rounded as these
// always had them.  Re (P z) is a rounded product and a fused one, the
// addend a separate sum; which product of the imaginary part is the fused one
// differs between segments summed in order (SEQ) and the others.
template <bool XY> __device__ __forceinline__ f2c dir_mul_pin(f2c a, f2c b, f2 nby) {
    return {f2_fma(a.x, b.x, f2_mul(a.y, nby)),
            XY ? f2_fma(a.x, b.y, f2_mul(a.y, b.x)) : f2_fma(a.y, b.x, f2_mul(a.x, b.y))};
}
template <bool SEQ>
__device__ __forceinline__ f2c dir_block_pin(const float2* cb, f2c z, f2 nzy, f2c zk, f2 nzky, bool la, bool lb) {
    f2c P = {f2_dup(cb[kDirBlock - 1].x), f2_dup(cb[kDirBlock - 1].y)};
#pragma unroll
    for (int t = kDirBlock - 2; t >= 0; --t) {
        const float2 ct = cb[t];
        const f2c m = dir_mul_pin<!SEQ>(P, z, nzy);
        P = f2c{f2_add(m.x, f2_dup(ct.x)), f2_add(m.y, f2_dup(ct.y))};
    }
    if (!la) P = f2c{f2_make(0.f, f2_hi(P.x)), f2_make(0.f, f2_hi(P.y))};
    if (!lb) P = f2c{f2_make(f2_lo(P.x), 0.f), f2_make(f2_lo(P.y), 0.f)};
    return dir_mul_pin<!SEQ>(P, zk, nzky);   // zk P
}
__device__ __forceinline__ f2c dir_pair(float2 a, float2 b) { return {f2_make(a.x, b.x), f2_make(a.y, b.y)}; }

__device__ __forceinline__ float dir_shfl(float v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ double dir_shfl(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ ff dir_shfl(ff v, int o) { return ff(dir_shfl(v.hi, o), dir_shfl(v.lo, o)); }

template <typename C> __device__ __forceinline__ C dir_zero() {
    using T = decltype(C().x);
    return C{T(0), T(0)};
}

// The result of node i: written to f (with rmul: rmul_j conj(result), the
// node-gradient epilogue) when the segment has one chunk, else to its partial.
__device__ __forceinline__ float2 dir_out(float2 v) { return v; }
__device__ __forceinline__ double2 dir_out(double2 v) { return v; }
__device__ __forceinline__ double2 dir_out(ffc v) { return double2{(double)v.x, (double)v.y}; }

template <typename A, typename O>
__device__ __forceinline__ void dir_write(const DirectSeg& S, int64_t i, int chunk, C_t<A> v,
                                          const int32_t* __restrict__ perm, const O* __restrict__ rmul,
                                          O* __restrict__ f, C_t<A>* __restrict__ part) {
    if (S.nchunk > 1) {
        part[S.dslot + (i - S.node_off) * S.nchunk + chunk] = v;
        return;
    }
    const int32_t j = perm[i];
    const O o = dir_out(v);
    f[j] = rmul ? cmulc(rmul[j], o) : o;
}

// One CTA (64 or 256 threads) per work item: consecutive sorted nodes of one segment against one
// chunk of up to kDirChunk coefficients staged in shared memory.  G = 2^lg
// consecutive lanes share a node (two nodes in the FP32 form) and take its
// Horner blocks l, l + G, ... of the chunk, so that a segment of few frequencies
// keeps all lanes busy: a whole warp per node left 30 of 32 lanes idle at K =
// 64.  Bound by the FMA pipe of its arithmetic (4 operations a term; FP64: 16
// cycles of the SM per warp instruction, active lanes or not, 93 % of the pipe at N
// = M = 2^18), the FP32 form there by the staging loads too (FMA pipe 40 %).  The
// FP32 form
// steps two nodes at once in packed pairs (fl_f32x2.cuh), 5 issues per term and
// node pair against 2 x 7.
//
// Segments of a pinned transform (DirectSeg::pin) keep its steps, their rounding
// and the order of its sums: one Horner chain per block, z from the node record
// in float, the blocks of a node in ascending order (pin = 2, G = 1) or one per
// lane, summed by the shuffle tree (pin = 1).
template <typename A, typename O, bool DERIV>
__global__ void __launch_bounds__(256)
    k_direct(const DirectItem* __restrict__ items, const DirectSeg* __restrict__ segs,
             const double2* __restrict__ ws, const uint4* __restrict__ ntab, const C_t<A>* __restrict__ zb,
             const C_t<A>* __restrict__ c, const int32_t* __restrict__ perm, const O* __restrict__ rmul,
             O* __restrict__ f, C_t<A>* __restrict__ part) {
    using C = C_t<A>;
    constexpr int NP = sizeof(A) == 4 ? 2 : 1;   // nodes per lane group
    extern __shared__ unsigned char smem_raw[];
    C* tile = reinterpret_cast<C*>(smem_raw);
    const DirectItem it = items[blockIdx.x];
    const DirectSeg S = segs[it.seg];
    const int64_t k0 = (int64_t)it.chunk * kDirChunk;
    const int kn = (int)min(S.K - k0, (int64_t)kDirChunk);
    const int nblk = (kn + kDirBlock - 1) / kDirBlock;   // zeros past kn
    for (int i = threadIdx.x; i < nblk * kDirBlock; i += blockDim.x) {
        C v = dir_zero<C>();
        if (i < kn) {
            const int64_t k = k0 + i;
            v = c[S.c_off + k];
            if constexpr (DERIV) {
                A wgt;
                if constexpr (sizeof(A) == 4) wgt = (float)k * 6.28318530717958647692f;   // k < 2^24: one rounding
                else wgt = kTwoPiDir * (double)k;
                v = C{-v.y * wgt, v.x * wgt};
            }
        }
        tile[i + i / kDirBlock] = v;
    }
    __syncthreads();
    const int lg = it.lg, G = 1 << lg;
    const int sub = threadIdx.x & (G - 1);
    // every lane of a warp runs the same trips (the shuffles below)
    for (int n0 = 0; n0 < it.nnodes; n0 += NP * ((int)blockDim.x >> lg)) {
        const int n = n0 + NP * (threadIdx.x >> lg);
        const bool on = n < it.nnodes;
        const int64_t i = it.node0 + (on ? n : 0);
        if constexpr (NP == 2) {
            const bool two = n + 1 < it.nnodes;
            const int64_t i1 = two ? i + 1 : i;
            const DirNode<A> na = dir_node<A>(ws, ntab, i), nb = dir_node<A>(ws, ntab, i1);
            f2c z, z8 = {};
            if (S.pin) {
                z = dir_pair(dir_f32_base(na.d), dir_f32_base(nb.d));
            } else {
                const C *za = zb + 2 * (i + S.z_off), *zc = zb + 2 * (i1 + S.z_off);
                z = dir_pair(za[0], zc[0]);
                z8 = dir_pair(za[1], zc[1]);
            }
            const f2 nz = f2_make(-f2_lo(z.y), -f2_hi(z.y)), nz8 = f2_make(-f2_lo(z8.y), -f2_hi(z8.y));
            f2c acc = {f2_dup(0.f), f2_dup(0.f)};
            for (int b = sub; on && b < nblk; b += G) {
                float2 ka = {0.f, 0.f}, kb = {0.f, 0.f};
                const bool la = dir_power<1>(na, k0 + b * kDirBlock, &ka, S.pin);
                const bool lb = dir_power<1>(nb, k0 + b * kDirBlock, &kb, S.pin);
                if (!la && !lb) break;          // both powers underflow: so do later blocks
                const float2* cb = reinterpret_cast<const float2*>(tile) + b * kDirBlockLd;
                const f2c zk = dir_pair(ka, kb);
                const f2 nzk = f2_make(-ka.y, -kb.y);
                if (S.pin) {
                    const f2c m = S.pin == 2 ? dir_block_pin<true>(cb, z, nz, zk, nzk, la, lb)
                                             : dir_block_pin<false>(cb, z, nz, zk, nzk, la, lb);
                    acc = f2c{f2_add(acc.x, m.x), f2_add(acc.y, m.y)};
                } else {
                    f2c P;
#pragma unroll
                    for (int h = kDirBlock / 8 - 1; h >= 0; --h) {
                        f2c Q = {f2_dup(cb[8 * h + 7].x), f2_dup(cb[8 * h + 7].y)};
#pragma unroll
                        for (int t = 6; t >= 0; --t) {
                            const float2 ct = cb[8 * h + t];
                            Q = dir_step(Q, z, nz, f2c{f2_dup(ct.x), f2_dup(ct.y)});
                        }
                        P = h == kDirBlock / 8 - 1 ? Q : dir_step(P, z8, nz8, Q);
                    }
                    if (!la)                        // (a power of zero takes nothing from its block)
                        P = f2c{f2_make(0.f, f2_hi(P.x)), f2_make(0.f, f2_hi(P.y))};
                    if (!lb) P = f2c{f2_make(f2_lo(P.x), 0.f), f2_make(f2_lo(P.y), 0.f)};
                    acc = dir_step(P, zk, nzk, acc);
                }
            }
            const f2 ar = acc.x, ai = acc.y;
            float ax = f2_lo(ar), ay = f2_lo(ai), bx = f2_hi(ar), by = f2_hi(ai);
            for (int off = G >> 1; off > 0; off >>= 1) {
                ax += dir_shfl(ax, off);
                ay += dir_shfl(ay, off);
                bx += dir_shfl(bx, off);
                by += dir_shfl(by, off);
            }
            if (sub == 0 && on) {
                dir_write<A>(S, i, it.chunk, float2{ax, ay}, perm, rmul, f, part);
                if (two) dir_write<A>(S, i1, it.chunk, float2{bx, by}, perm, rmul, f, part);
            }
        } else {
            const DirNode<A> nd = dir_node<A>(ws, ntab, i);
            C acc = dir_zero<C>();
            const C z = zb[2 * (i + S.z_off)], z8 = zb[2 * (i + S.z_off) + 1];
            for (int b = sub; on && b < nblk; b += G) {
                C zk;
                if (!dir_power<1>(nd, k0 + b * kDirBlock, &zk)) break;
                const C* cb = tile + b * kDirBlockLd;
                C P;
#pragma unroll
                for (int h = kDirBlock / 8 - 1; h >= 0; --h) {
                    C Q = cb[8 * h + 7];
#pragma unroll
                    for (int t = 6; t >= 0; --t) Q = dir_step(Q, z, cb[8 * h + t]);
                    P = h == kDirBlock / 8 - 1 ? Q : dir_step(P, z8, Q);
                }
                acc = cadd(acc, cmul(zk, P));
            }
            for (int off = G >> 1; off > 0; off >>= 1)
                acc = cadd(acc, C{dir_shfl(acc.x, off), dir_shfl(acc.y, off)});
            if (sub == 0 && on) dir_write<A>(S, i, it.chunk, acc, perm, rmul, f, part);
        }
    }
}

// The segment holding flattened node t: the last range whose prefix is
// <= t (prefixes ascend; binary search).
__device__ __forceinline__ int find_direct_range(const DirectRange* __restrict__ ranges, int nranges,
                                                 int64_t t) {
    int lo = 0, hi = nranges;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (ranges[mid].prefix <= t) lo = mid;
        else hi = mid;
    }
    return lo;
}

// Segments of several chunks: f[perm[i]] = sum over the node's chunks (in chunk
// order); with rmul, rmul[perm[i]] * conj(sum).
template <typename A, typename O>
__global__ void k_direct_reduce(int nranges, const DirectRange* __restrict__ ranges, int64_t total,
                                const DirectSeg* __restrict__ segs, const int32_t* __restrict__ perm,
                                const C_t<A>* __restrict__ part, const O* __restrict__ rmul,
                                O* __restrict__ f) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= total) return;
    const DirectRange R = ranges[find_direct_range(ranges, nranges, t)];
    const DirectSeg S = segs[R.seg];
    const int64_t local = t - R.prefix;
    const C_t<A>* p = part + S.dslot + local * S.nchunk;
    C_t<A> acc = dir_zero<C_t<A>>();
    for (int ch = 0; ch < S.nchunk; ++ch) acc = cadd(acc, p[ch]);
    const int32_t j = perm[S.node_off + local];
    const O o = dir_out(acc);
    f[j] = rmul ? cmulc(rmul[j], o) : o;
}

// Adjoint of the direct segments, cdir[k] += sum_j r_j conj(z_j)^k for k < K: the
// transpose of the blocked Horner sum.  One warp per work item (segment, chunk
// of 32 KL frequencies, node group).  The lanes split into KB = 2^lkb blocks of
// KL frequencies (the fewest that cover the chunk's share of K) and 32 / KB node
// subgroups; a lane forms conj(z_j)^k0 from an exactly reduced phase, then
// steps through its KL frequencies multiplying by conj(z_j); a shuffle tree adds
// the subgroups and the first adds the result to cdir (atomics across node
// groups).  The FP32 form steps two nodes at once in packed pairs.  The node
// groups are cut so that the launch has several warps per SM: at 256 nodes each
// the K = 512 band of N = M = 2^18 disk nodes had 160 warps (float pairs:
// 570 us, and the bands with K <= 256 in double 990 us).  Still bound by its few
// warps there (14 % active, 18 % of the issue slots).
constexpr int kAdjKL = kDirAdjKL;
static_assert(kAdjKL == 16, "two chains of eight steps");

template <typename A, typename O>
__global__ void __launch_bounds__(32)
    k_direct_adj(const DirectItem* __restrict__ items, const DirectSeg* __restrict__ segs,
                 const double2* __restrict__ ws, const uint4* __restrict__ ntab, const C_t<A>* __restrict__ zb,
                 const int32_t* __restrict__ perm, const O* __restrict__ r, O* __restrict__ cdir) {
    using C = C_t<A>;
    const DirectItem it = items[blockIdx.x];
    const DirectSeg S = segs[it.seg];
    const int lane = threadIdx.x, lkb = it.lg, g = lane >> lkb, G = 32 >> lkb;
    zb += 2 * S.z_off;
    const int64_t k0 = (int64_t)it.chunk * (32 * kAdjKL) + (int64_t)(lane & ((1 << lkb) - 1)) * kAdjKL;
    const bool active = k0 < S.K;
    C acc[kAdjKL];
    if constexpr (sizeof(A) == 4) {
        f2 ar[kAdjKL], ai[kAdjKL];
#pragma unroll
        for (int t = 0; t < kAdjKL; ++t) ar[t] = ai[t] = f2_dup(0.f);
        for (int jn = 2 * g; active && jn < it.nnodes; jn += 2 * G) {
            const int64_t i = it.node0 + jn;
            const bool two = jn + 1 < it.nnodes;
            const int64_t i1 = two ? i + 1 : i;
            const DirNode<A> na = dir_node<A>(ws, ntab, i), nb = dir_node<A>(ws, ntab, i1);
            float2 wa = {0.f, 0.f}, wb = {0.f, 0.f};
            const bool la = dir_power<-1>(na, k0, &wa);
            const bool lb = dir_power<-1>(nb, k0, &wb) && two;
            if (!la && !lb) continue;
            wa = la ? cmul(r[perm[i]], wa) : float2{0.f, 0.f};
            wb = lb ? cmul(r[perm[i1]], wb) : float2{0.f, 0.f};
            // conj(z): w conj(z) = (wx zx + wy zy, wy zx - wx zy)
            const float2 a1 = zb[2 * i], b1 = zb[2 * i1], a8 = zb[2 * i + 1], b8 = zb[2 * i1 + 1];
            const f2c zq = {f2_make(a1.x, b1.x), f2_make(-a1.y, -b1.y)};
            const f2 nzq = f2_make(a1.y, b1.y);
            f2c w = dir_pair(wa, wb), v = dir_pair(cmulc(wa, a8), cmulc(wb, b8));   // k0 and k0 + 8
#pragma unroll
            for (int t = 0; t < kAdjKL / 2; ++t) {
                ar[t] = f2_add(ar[t], w.x);
                ai[t] = f2_add(ai[t], w.y);
                ar[t + 8] = f2_add(ar[t + 8], v.x);
                ai[t + 8] = f2_add(ai[t + 8], v.y);
                w = f2c{f2_fma(w.y, nzq, f2_mul(w.x, zq.x)), f2_fma(w.x, zq.y, f2_mul(w.y, zq.x))};
                v = f2c{f2_fma(v.y, nzq, f2_mul(v.x, zq.x)), f2_fma(v.x, zq.y, f2_mul(v.y, zq.x))};
            }
        }
#pragma unroll
        for (int t = 0; t < kAdjKL; ++t) acc[t] = float2{f2_lo(ar[t]) + f2_hi(ar[t]), f2_lo(ai[t]) + f2_hi(ai[t])};
    } else {
#pragma unroll
        for (int t = 0; t < kAdjKL; ++t) acc[t] = dir_zero<C>();
        for (int jn = g; active && jn < it.nnodes; jn += G) {
            const int64_t i = it.node0 + jn;
            C w0;
            if (!dir_power<-1>(dir_node<A>(ws, ntab, i), k0, &w0)) continue;
            const O rj = r[perm[i]];
            const C z = zb[2 * i];
            const C zq = C{z.x, -z.y};
            C rw;
            if constexpr (std::is_same<A, ff>::value) rw = cmul(ffc{ff(rj.x), ff(rj.y)}, w0);
            else rw = cmul(rj, w0);
            C rv = cmulc(rw, zb[2 * i + 1]);         // from k0 + 8
#pragma unroll
            for (int t = 0; t < kAdjKL / 2; ++t) {
                acc[t] = cadd(acc[t], rw);
                acc[t + 8] = cadd(acc[t + 8], rv);
                rw = cmul(rw, zq);
                rv = cmul(rv, zq);
            }
        }
    }
    for (int off = 1 << lkb; off < 32; off <<= 1) {
#pragma unroll
        for (int t = 0; t < kAdjKL; ++t)
            acc[t] = cadd(acc[t], C{dir_shfl(acc[t].x, off), dir_shfl(acc[t].y, off)});
    }
    if (g != 0 || !active) return;
#pragma unroll
    for (int t = 0; t < kAdjKL; ++t) {
        const int64_t k = k0 + t;
        if (k < S.K) {
            const O o = dir_out(acc[t]);
            atomicAdd(&cdir[k].x, o.x);
            atomicAdd(&cdir[k].y, o.y);
        }
    }
}

template <typename A>
static cudaError_t dir_base_t(Plan& p, cudaStream_t st) {
    k_dir_base<A><<<(unsigned)((p.base_nodes + 255) / 256), 256, 0, st>>>(
        p.base_nodes, p.d_dsegs, (int)p.direct_segs.size(), p.d_ws, (C_t<A>*)p.d_dz);
    return cudaGetLastError();
}

cudaError_t build_direct_base(Plan& p, cudaStream_t st) {
    if (p.prec == FL_FP64_FF) return dir_base_t<ff>(p, st);
    return p.prec == FL_FP64 ? dir_base_t<double>(p, st) : dir_base_t<float>(p, st);
}

// (float pairs read the coefficients as pairs, k-weighted by the caller for the
// derivative)
template <typename A, typename O, bool DERIV>
static cudaError_t direct_forward_t(Plan& p, const void* c, void* f, const void* rmul, cudaStream_t st) {
    using C = C_t<A>;
    if (p.direct_work.empty()) return cudaSuccess;
    const size_t smem = dir_tile(p.direct_kmax, sizeof(C));
    auto kern = k_direct<A, O, DERIV>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int slot;
    timer_begin(p, "direct", (double)p.direct_terms * sizeof(C) / 32.0, st, &slot);
    kern<<<(unsigned)p.direct_work.size(), p.direct_threads, smem, st>>>(
        p.d_direct, p.d_dsegs, p.d_ws, p.d_ntab, (const C*)p.d_dz, (const C*)c, p.d_perm, (const O*)rmul, (O*)f,
        (C*)p.d_dpart);
    if (p.direct_nodes > 0) {
        k_direct_reduce<A, O><<<(unsigned)((p.direct_nodes + 255) / 256), 256, 0, st>>>(
            (int)p.direct_ranges.size(), p.d_dranges, p.direct_nodes, p.d_dsegs, p.d_perm, (const C*)p.d_dpart,
            (const O*)rmul, (O*)f);
        ++p.launches;
    }
    timer_end(p, slot, st);
    ++p.launches;
    return cudaGetLastError();
}

cudaError_t run_direct_forward(Plan& p, const void* c, void* f, bool deriv, const void* rmul,
                               cudaStream_t st) {
    if (p.prec == FL_FP64_FF) return direct_forward_t<ff, double2, false>(p, p.d_cff, f, rmul, st);
    if (p.prec == FL_FP64)
        return deriv ? direct_forward_t<double, double2, true>(p, c, f, rmul, st)
                     : direct_forward_t<double, double2, false>(p, c, f, rmul, st);
    return deriv ? direct_forward_t<float, float2, true>(p, c, f, rmul, st)
                 : direct_forward_t<float, float2, false>(p, c, f, rmul, st);
}

template <typename A, typename O>
static cudaError_t direct_adjoint_t(Plan& p, const void* r, cudaStream_t st) {
    if (p.dadj_work.empty()) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(p.d_cdir, 0, p.N * sizeof(O), st);
    if (e != cudaSuccess) return e;
    int slot;
    timer_begin(p, "direct_adj", 0.0, st, &slot);
    k_direct_adj<A, O><<<(unsigned)p.dadj_work.size(), 32, 0, st>>>(
        p.d_dadj, p.d_dsegs, p.d_ws, p.d_ntab, (const C_t<A>*)p.d_dz, p.d_perm, (const O*)r, (O*)p.d_cdir);
    ++p.launches;
    timer_end(p, slot, st);
    return cudaGetLastError();
}

cudaError_t run_direct_adjoint(Plan& p, const void* r, cudaStream_t st) {
    if (p.prec == FL_FP64_FF) return direct_adjoint_t<ff, double2>(p, r, st);
    return p.prec == FL_FP64 ? direct_adjoint_t<double, double2>(p, r, st)
                             : direct_adjoint_t<float, float2>(p, r, st);
}

}  // namespace fl
