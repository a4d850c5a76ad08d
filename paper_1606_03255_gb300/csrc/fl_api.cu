// fl_api.cu -- the C ABI of libfl.so (include/fl.h): parameter selection
// (Definition 3.2 and Algorithm 2 of Kunis & Melzer), band sizing, plan
// construction, execution, timing and error reporting.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <mutex>
#include <string>

#include "fl_plan.cuh"

namespace fl {

static thread_local std::string g_err;

fl_status set_error(fl_status s, const std::string& msg) {
    g_err = msg;
    return s;
}

void clear_error() { g_err.clear(); }

static fl_status fail(fl_status s, const std::string& msg) { return set_error(s, msg); }

static fl_status cuda_fail(cudaError_t e, const char* where) {
    g_err = std::string(where) + ": " + cudaGetErrorString(e);
    return e == cudaErrorMemoryAllocation ? FL_ENOMEM : FL_ECUDA;
}

#define FL_CUDA(call, where)                          \
    do {                                              \
        cudaError_t e_ = (call);                      \
        if (e_ != cudaSuccess) return cuda_fail(e_, where); \
    } while (0)

Plan::~Plan() {
    if (gexec) cudaGraphExecDestroy(gexec);
    void* ptrs[] = {d_stage_c, d_stage_f, d_stage_r, d_boff, d_bptr};   // made by calls
    for (void* q : ptrs)
        if (q) cudaFree(q);
    for (Timer& t : timers) {
        cudaEventDestroy(t.start);
        cudaEventDestroy(t.stop);
    }
}

void timer_begin(Plan& p, const char* name, double bytes, cudaStream_t st, int* slot) {
    *slot = -1;
    if (!p.timing) return;
    Timer t;
    t.name = name;
    t.bytes = bytes;
    if (cudaEventCreate(&t.start) != cudaSuccess) return;
    if (cudaEventCreate(&t.stop) != cudaSuccess) {
        cudaEventDestroy(t.start);
        return;
    }
    cudaEventRecord(t.start, st);
    p.timers.push_back(t);
    *slot = (int)p.timers.size() - 1;
}

void timer_end(Plan& p, int slot, cudaStream_t st) {
    if (slot >= 0) cudaEventRecord(p.timers[slot].stop, st);
}

static int ilog2_ceil(int64_t v) {
    int l = 0;
    while (((int64_t)1 << l) < v) ++l;
    return l;
}

// Smallest Kaiser-Bessel half-width m whose aliasing-plus-truncation estimate
// 4 pi (sqrt(m) + m) (1 - 1/sigma)^(1/4) exp(-2 pi m sqrt(1 - 1/sigma))
// (the error bound of the Kaiser-Bessel NFFT) is at most eps.
static int window_width(double eps, double sigma) {
    const double a = sqrt(1.0 - 1.0 / sigma);
    for (int m = 2; m <= 12; ++m) {
        const double bound = 4.0 * M_PI * (sqrt((double)m) + m) * sqrt(a) * exp(-2.0 * M_PI * m * a);
        if (bound <= eps) return m;
    }
    return 12;
}

// Parameters of Algorithm 2 (Section 4) with the error split of Lemma 4.1 that
// do not depend on N: q, y_1 = ln(1/eps), the window.
// One-sided interpolation rank: the smallest q whose per-entry bound
// max_k |exp(-y k) - sum_s L_s(y) exp(-y_s k)| <= 2 q^q e^-q / (4^q q!) on a
// band (a, 2a] is at most eps_K.  The bound is the interpolation error formula
// of Section 2 with diam = a and max |d^q/dy^q exp(-y k)| = k^q exp(-a k),
// maximised over k a = q.
static int onesided_rank(double eps_K) {
    for (int q = 1; q <= kMaxQ; ++q) {
        const double lb = log(2.0) + q * log((double)q) - q - q * log(4.0) - lgamma(q + 1.0);
        if (lb <= log(eps_K)) return q;
    }
    return kMaxQ + 1;
}

static fl_status select_common(Plan& p, int q_in) {
    p.eps_K = p.eps / 3.0;
    p.eps_A = p.eps / 3.0;
    p.q_given = q_in > 0;
    if (q_in > 0)
        p.q = q_in;
    else if (p.variant == 1)
        p.q = onesided_rank(p.eps_K);
    else
        p.q = (int)ceil(0.5 + log(1.0 / p.eps_K) / log(4.0));
    if (p.q > kMaxQ) return fail(FL_EUNSUPPORTED, "interpolation rank q above 40");
    p.y1 = log(1.0 / p.eps);            // Z^0 removed: y in [0, ln(1/eps)]
    // real exponents: two windows (frequency spreading and the outer NFFT),
    // the latter's error amplified by up to Phi(0)/Phi(1/4) < 8 in the division
    // by Phi(x/2): each gets eps_A / 8
    p.mw = window_width(p.xi_mode ? p.eps_A / 8.0 : p.eps_A, 2.0);
    p.kb_b = M_PI * (2.0 - 1.0 / 2.0);
    return FL_OK;
}

// Real exponents: Definition 3.2 with xi_1 = max xi_k; band m keeps the sorted
// exponents xi_k <= xi_1 / 2^(l_m - 1) (a prefix of length K).  Its NNFFT
// spreads them, centred on xc (2 xc = floor(xi_min + cut), an integer), onto the
// frequency grid of spacing 1/2 (grid frequency g <-> xi = xc + g/2; taps
// g in (2(xi - xc) - m_w, 2(xi - xc) + m_w]); the occupied |g| <= gh, and the
// outer NFFT has bandwidth Nm = 2^lg >= 2 gh + 2 on n = 2 Nm points.  The
// dyadic cuts lie just below powers of two, so the window margin m_w + 1 alone
// would double Nm; the half-size Nm is kept when it misses at most m_w + 3
// occupied frequencies, e = gh - (Nm/2 - 1), and these raise the
// Kaiser-Bessel aliasing term by at most 1 %: the nearest alias of frequency
// Nm/2 - 1 + e sits at |nu| = 3/4 - e/n, where Phi = pi I_0(m_w pi sqrt(6 e / n))
// (b = 3 pi / 2), so the condition is m_w pi sqrt(6 e / n) <= 0.2 (I_0(0.2) = 1.01).
static fl_status select_bands_xi(Plan& p, Instance& in, int inst_index) {
    const std::vector<double>& xs = p.h_xis;
    in.xi1 = xs.empty() ? 0.0 : xs.back();
    const double lv = ceil(log2(p.y1 * in.xi1 / p.eps_K)) + 1.0;
    in.levels = (int)std::max(1.0, lv);
    if (in.levels > 127) return fail(FL_EUNSUPPORTED, "more than 127 dyadic levels");
    in.band_base = (int)p.bands.size();
    for (int b = 0; b <= in.levels; ++b) {
        BandHost bh;
        bh.inst = inst_index;
        bh.local = b;
        bh.dev.c_off = in.noff;
        bh.dev.parent = -1;
        bh.dev.kb = p.kb_b;
        if (b == 0) {
            p.bands.push_back(bh);
            continue;
        }
        double cut = in.xi1;
        if (b < in.levels) {
            const double lg = log2(p.y1 * in.xi1) - b - log2(log(1.0 / p.eps_K));
            bh.ell = std::max(1, (int)floor(lg) + 1);
            bh.Lm = in.levels - b;
            cut = std::min(in.xi1, ldexp(in.xi1, 1 - bh.ell));
            bh.dev.nrhs = p.q;
            const double a = ldexp(p.y1, -b);
            bh.dev.yc = 1.5 * a;
            bh.dev.yh = 0.5 * a;
            bh.dev.yh_inv = 1.0 / bh.dev.yh;
        } else {
            bh.dev.nrhs = 1;
        }
        const int64_t K = (int64_t)(std::upper_bound(xs.begin(), xs.end(), cut) - xs.begin());
        const double lo = K > 0 ? xs[0] : cut;
        const double two_xc = floor(lo + cut);
        bh.dev.xc = 0.5 * two_xc;
        bh.dev.gh = (int64_t)std::max(ceil(two_xc - 2.0 * lo), ceil(2.0 * cut - two_xc)) + p.mw + 1;
        int lg = std::max(4, ilog2_ceil(2 * bh.dev.gh + 2));
        if (lg > 4) {
            const int64_t e = bh.dev.gh - (((int64_t)1 << (lg - 1)) / 2 - 1);
            if (e <= p.mw + 3 && p.mw * M_PI * sqrt(6.0 * (double)e / ldexp(1.0, lg)) <= 0.2) --lg;
        }
        bh.dev.K = K;
        bh.dev.Nm = (int64_t)1 << lg;
        bh.dev.log2n = lg + 1;
        bh.dev.n = (int64_t)1 << (lg + 1);
        if (bh.dev.log2n > kMaxLog2n) return fail(FL_EUNSUPPORTED, "NNFFT grid above 2^24 points");
        p.bands.push_back(bh);
    }
    return FL_OK;
}

// Right-hand sides per chunk of the real-exponent spreading, QC in {4, 8, 12,
// 16}: each chunk passes over a grid frequency's exponents once, at about
// 10 + QC/4 + 2 QC instructions per exponent (index, window and coefficient;
// the 16-byte weight loads; the complex multiply-adds), the last chunk padded
// with zero weights.  The QC of least total cost for q.
static int xi_chunk(int q) {
    int best = 4, best_cost = 1 << 30;
    for (int qc : {16, 12, 8, 4}) {
        const int cost = (q + qc - 1) / qc * (10 + qc / 4 + 2 * qc);
        if (cost < best_cost) {
            best = qc;
            best_cost = cost;
        }
    }
    return best;
}

// The dyadic partition of one transform (Definition 3.2 with xi_1 = N - 1):
// appends its bands 0..levels to p.bands.
static fl_status select_bands(Plan& p, Instance& in, int inst_index) {
    if (p.xi_mode) return select_bands_xi(p, in, inst_index);
    in.xi1 = (double)(in.N - 1);        // frequencies 0..N-1
    if (in.N == 1) {
        in.levels = 1;
    } else {
        const double lv = ceil(log2(p.y1 * in.xi1 / p.eps_K)) + 1.0;
        in.levels = (int)std::max(1.0, lv);
    }
    if (in.levels > 127) return fail(FL_EUNSUPPORTED, "more than 127 dyadic levels");
    in.band_base = (int)p.bands.size();
    for (int b = 0; b <= in.levels; ++b) {
        BandHost bh;
        bh.inst = inst_index;
        bh.local = b;
        bh.dev.c_off = in.noff;
        bh.dev.parent = -1;
        bh.dev.kb = p.kb_b;
        if (b == 0) {
            p.bands.push_back(bh);
            continue;
        }
        int64_t K;
        if (b < in.levels) {
            const double lg = log2(p.y1 * in.xi1) - b - log2(log(1.0 / p.eps_K));
            bh.ell = std::max(1, (int)floor(lg) + 1);
            bh.Lm = in.levels - b;
            // frequencies k <= xi1 / 2^(l_m - 1) carry weight (Lemma A.2(ii))
            K = std::min<int64_t>(in.N, (int64_t)floor(ldexp(in.xi1, 1 - bh.ell)) + 1);
            bh.dev.nrhs = p.q;
            const double a = ldexp(p.y1, -b);
            bh.dev.yc = 1.5 * a;
            bh.dev.yh = 0.5 * a;
            bh.dev.yh_inv = 1.0 / bh.dev.yh;
        } else {
            K = in.N;           // Z_M band: kernel ~ 1, one plain NFFT
            bh.dev.nrhs = 1;
        }
        const int lg = std::max(4, ilog2_ceil(K));
        bh.dev.K = K;
        bh.dev.Nm = (int64_t)1 << lg;
        bh.dev.log2n = lg + 1;
        bh.dev.n = (int64_t)1 << (lg + 1);
        if (bh.dev.log2n > kMaxLog2n) return fail(FL_EUNSUPPORTED, "grid above 2^24 points");
        p.bands.push_back(bh);
    }
    return FL_OK;
}

// Route of a non-empty band: NFFT with nrhs right-hand sides, or the direct sum
// over its K frequencies.  Costs in issued instructions: an FFT grid point
// ~ (log2 n + 8) over both passes and the prep (twice that in double); per
// gathered node, 2 per tap and right-hand side plus the window (2 m_w
// sinh/sqrt) and the barycentric divisions, both several times dearer in
// double on this part; a fixed launch and latency share per NFFT band; a direct
// term ~ 6 (one complex Horner step and its share of the block's phase).  The
// constants were fitted when double twiddles, windows and weights were formed in
// the call.  Twiddles now come from tables, and so do the taps and weights of
// single FP64 and float-pair plans, so there the model charges an NFFT more than
// it costs and leaves bands to the direct sum; batches form the windows and
// weights in the call as before.
static int route_of(const Plan& p, const BandHost& bh) {
    if (p.route_mode == 1) return 1;
    if (p.route_mode == 2) return 2;
    const BandDev& d = bh.dev;
    const bool dbl = p.prec != FL_FP32;   // float pairs: gather and direct bands in double
    const double fft_pt = dbl ? 2.0 : 1.0, win = dbl ? 150.0 : 20.0, div = dbl ? 40.0 : 4.0;
    const double per_node = (double)d.nrhs * 2 * p.mw * 2 + 2.0 * p.mw * win + (d.nrhs > 1 ? d.nrhs * div : 0.0);
    const double fft = (double)d.nrhs * d.n * (d.log2n + 8) * fft_pt + (double)bh.nodes * per_node + 2.0e5;
    const double direct = (double)bh.nodes * d.K * 6.0 * p.direct_bias;
    return direct < fft ? 2 : 1;
}

static bool pinned(const Plan& p, const Instance& in) {
    return p.prec == FL_FP32 && !p.xi_mode && in.N <= kPinnedN;
}

// The nodes of a direct band: appended to the last segment when they follow it
// and sum over the same coefficients, else a segment of their own.
static void add_direct_band(Plan& p, const BandHost& bh) {
    const BandDev& d = bh.dev;
    const int pin = !pinned(p, p.inst[bh.inst]) ? 0 : d.K <= kDirSeqK && bh.nodes >= kDirSeqNodes ? 2 : 1;
    if (!p.direct_segs.empty()) {
        DirectSeg& s = p.direct_segs.back();
        if (s.K == d.K && s.pin == pin && s.c_off == d.c_off && s.node_off + s.nodes == bh.node_off) {
            s.nodes += bh.nodes;
            return;
        }
    }
    p.direct_segs.push_back({bh.node_off, bh.nodes, d.K, d.c_off, 0, 0, (int)((d.K + kDirChunk - 1) / kDirChunk), pin});
}

// Work items of the direct segments.  Forward: the lanes per node G cover the
// chunk's Horner blocks with `r` blocks per lane, r the largest power of two (up
// to kDirMaxBlocks) that still leaves every SM about 1024 busy lanes (pinned
// transforms: r = 1, or G = 1 for DirectSeg::pin = 2); an item
// holds the nodes of one pass of its threads, or of two when there are
// plenty of items (the staged chunk then serves twice as many).  Adjoint: node
// groups of `steps` nodes (pairs in FP32) per lane, doubled from 8 while the
// launch keeps 24 warps per SM, since every group adds its sums to cdir with
// atomics.
static void build_direct_items(Plan& p) {
    constexpr int64_t kSMs = 152;
    const int np = p.prec == FL_FP32 ? 2 : 1;   // nodes per lane group
    p.direct_work.clear();
    p.dadj_work.clear();
    p.direct_ranges.clear();
    p.direct_nodes = p.dpart_elems = p.direct_kmax = p.base_nodes = 0;
    int64_t lane_blocks = 0;
    for (DirectSeg& s : p.direct_segs) {
        lane_blocks += (s.nodes + np - 1) / np * ((s.K + kDirBlock - 1) / kDirBlock);
        p.direct_kmax = std::max(p.direct_kmax, s.K);
        s.z_off = p.base_nodes - s.node_off;
        if (s.pin == 0 || !p.batched) p.base_nodes += s.nodes;   // (single plans: the adjoint reads them)
        if (s.nchunk == 1) continue;
        s.dslot = p.dpart_elems;
        p.dpart_elems += s.nodes * s.nchunk;
        p.direct_ranges.push_back({(int)(&s - p.direct_segs.data()), 0, s.nodes, p.direct_nodes});
        p.direct_nodes += s.nodes;
    }
    int r = 1;
    while (r < kDirMaxBlocks && lane_blocks >= 2 * r * kSMs * 1024) r *= 2;
    auto lanes = [&](const DirectSeg& s) {   // log2 G
        if (s.pin == 2) return 0;
        const int64_t nblk = (std::min<int64_t>(s.K, kDirChunk) + kDirBlock - 1) / kDirBlock;
        return std::min(5, ilog2_ceil(s.pin ? nblk : (nblk + r - 1) / r));
    };
    // few items (a small transform) in FP64: CTAs of 64 threads, so that all SMs
    // take part (46 CTAs of 256 threads at N = M = 1024).  FP32 and float pairs keep 256:
    // staging the coefficients is their larger part (FP32 3001 x 2500: 24.0 us, 28.7
    // with 64; pairs 17576 x 266: 30.9, 39.1 with 64)
    p.direct_threads = 256;
    auto items = [&](int passes, bool make) {
        int64_t count = 0;
        for (size_t g = 0; g < p.direct_segs.size(); ++g) {
            const DirectSeg& s = p.direct_segs[g];
            const int lg = lanes(s);
            const int64_t per = (int64_t)passes * np * (p.direct_threads >> lg);
            for (int64_t n0 = 0; n0 < s.nodes; n0 += per) {
                count += s.nchunk;
                for (int ch = 0; make && ch < s.nchunk; ++ch)
                    p.direct_work.push_back({(int)g, ch, s.node_off + n0, (int)std::min(per, s.nodes - n0), lg});
            }
        }
        return count;
    };
    const int64_t full = items(1, false);
    if (p.prec == FL_FP64 && full < 2 * kSMs) p.direct_threads = 64;
    items(full >= 16 * kSMs ? 2 : 1, true);
    if (p.batched) return;   // forward only
    auto adj_items = [&](int64_t steps, bool make) {
        int64_t count = 0;
        for (size_t g = 0; g < p.direct_segs.size(); ++g) {
            const DirectSeg& s = p.direct_segs[g];
            const int64_t span = 32 * kDirAdjKL;
            for (int64_t k = 0; k < s.K; k += span) {
                const int lkb = ilog2_ceil((std::min(span, s.K - k) + kDirAdjKL - 1) / kDirAdjKL);
                const int64_t per = steps * np * (32 >> lkb);
                count += (s.nodes + per - 1) / per;
                for (int64_t n0 = 0; make && n0 < s.nodes; n0 += per)
                    p.dadj_work.push_back({(int)g, (int)(k / span), s.node_off + n0,
                                           (int)std::min(per, s.nodes - n0), lkb});
            }
        }
        return count;
    };
    int64_t steps = 8;
    while (steps < kDirAdjSteps && adj_items(steps, false) > 24 * kSMs) steps *= 2;
    adj_items(steps, true);
}

// (pageable host memory: copied to staging memory before the call returns)
template <typename E>
static cudaError_t upload(DevPool& pool, const std::vector<E>& v, E** dev, cudaStream_t st) {
    if (v.empty()) return cudaSuccess;
    cudaError_t e = pool.get(dev, (int64_t)v.size());
    if (e == cudaSuccess) e = cudaMemcpyAsync(*dev, v.data(), v.size() * sizeof(E), cudaMemcpyHostToDevice, st);
    return e;
}

// Four-step work items of the large bands, grouped by grid size into launches
// of at most rhs_per_launch items (0: a whole size class) and at most
// kMaxYElems intermediate elements, a band's items never split between two
// launches (a launch holding one band may exceed the cap); sets Y_elems.
constexpr int64_t kMaxYElems = (int64_t)1 << 28;

static void build_pass_groups(Plan& p) {
    p.pass_items.clear();
    p.pass_groups.clear();
    p.Y_elems = 0;
    for (int lg = kSmallMaxLog2 + 1; lg <= kMaxLog2n; ++lg) {
        const int64_t n = (int64_t)1 << lg;
        int cap = (int)std::min<int64_t>(65535, std::max<int64_t>(1, kMaxYElems / n));
        if (p.rhs_per_launch > 0) cap = std::min(cap, p.rhs_per_launch);
        int cnt = 0;
        auto close = [&]() {
            if (cnt == 0) return;
            p.pass_groups.push_back(PassGroup{(int)p.pass_items.size() - cnt, cnt, lg});
            p.Y_elems = std::max<int64_t>(p.Y_elems, (int64_t)cnt * n);
            cnt = 0;
        };
        for (int b : p.large_bands) {
            const BandDev& d = p.bands[b].dev;
            if (d.log2n != lg) continue;
            if (cnt > 0 && cnt + d.nrhs > cap) close();
            for (int s = 0; s < d.nrhs; ++s) {
                p.pass_items.push_back({b, s, (int64_t)cnt * n});
                ++cnt;
            }
        }
        close();
    }
}

// Estimated cost of a gather from the grids, all right-hand sides.
static double unfused_cost(int64_t nodes, int nrhs, int mw) {
    return (double)nodes * ((double)nrhs * 2 * mw * 2 + 2.0 * mw * 20.0);
}

// FP32 transforms that may merge bands (not pinned): the same with the traffic
// of the grids and partial sums (constants from N = M = 2^20), in the same units (0.26 ps: an FFT point costs
// log2 n + 8 of them, 7 ps measured at N = M = 2^20; a byte of HBM about 0.56).
// A gather from the grid pays for writing it and reads it once, or 128 bytes
// per node, whichever is less (it measured 0.16 ms for 1.5*10^5 nodes and 35
// grids of 2^21 points); a fused one writes and reads a partial sum per node
// and tile.  *fuse: the cheaper of the two.
static double free_gather_cost(int64_t nodes, int nrhs, int64_t n, int log2n, int mw, bool fusable, bool* fuse) {
    const double bytes = std::min<double>(8.0 * n, 128.0 * nodes);
    const double grid = unfused_cost(nodes, nrhs, mw) + nrhs * (0.56 * 8.0 * n + 0.8 * bytes);
    *fuse = false;
    if (!fusable || log2n <= kSmallMaxLog2) return grid;
    const int TR = pass_tiles(8, (log2n + 1) / 2, FL_P2_THREADS_F32);
    const int parts = (2 * mw - 1 + TR - 1) / TR + 1;
    const double fused = nrhs * ((double)nodes * (TR + 2 * mw - 1) / TR * 24.0 + (double)nodes * parts * 15.0);
    *fuse = fused < grid;
    return std::min(fused, grid);
}

// Window gather fused into pass 2 (FP32 forward, four-step grids).  A band
// qualifies when its nodes are few for its grid: per right-hand side the
// unfused path writes the grid (8 n bytes) and gathers about three 32-byte
// sectors per node, the fused one reads its entries (8 + 16 NQ bytes: slot,
// column, window values) and writes and later reads one partial sum per entry.  Each node's
// window of 2 m_w taps at grid indices lo .. lo + 2 m_w - 1 (lo = floor(n x) -
// m_w + 1, mod n) is cut into entries, one per pass-2 row block its taps fall
// in (tile rows TR of the length-n1 pass, rows l2 = g mod n2, column l1 = g /
// n2); the window values are those of the gather kernel, phi_t = kb(frac(n x)
// + m_w - 1 - t), in FP64 rounded once.
static fl_status build_fused(Plan& p, cudaStream_t st) {
    p.fused_bands = p.fused_entries = 0;
    if (p.prec != FL_FP32 || p.xi_mode || p.fuse_mode == 1 || p.M == 0) return FL_OK;
    struct Cand {
        int b, l1, l2, TR, P;
    };
    std::vector<Cand> cands;
    const int taps = 2 * p.mw;
    for (int b = 0; b < (int)p.bands.size(); ++b) {
        BandHost& bh = p.bands[b];
        BandDev& d = bh.dev;
        d.fused = 0;
        if (d.route != 1 || d.nsub > 0 || d.log2n <= kSmallMaxLog2 || bh.nodes == 0) continue;
        const int l2 = d.log2n / 2, l1 = (d.log2n + 1) / 2;
        const int TR = pass_tiles(8, l1, FL_P2_THREADS_F32);
        const int P = (taps - 1 + TR - 1) / TR + 1;
        const int NQ = (TR + 3) / 4;
        const double parts = (double)(TR + taps - 1) / TR;
        const double unfused = 8.0 * d.n + std::min<double>(8.0 * d.n, 96.0 * bh.nodes);
        const double fused = bh.nodes * parts * (8.0 + 16.0 * NQ + 8.0) + 8.0 * P * bh.nodes;
        bool fuse = d.parent >= 0 || fused <= 0.5 * unfused;   // pinned transforms: sub-bands always
        if (!pinned(p, p.inst[bh.inst])) free_gather_cost(bh.nodes, d.nrhs, d.n, d.log2n, p.mw, true, &fuse);
        if (p.fuse_mode == 2 || fuse) cands.push_back({b, l1, l2, TR, P});
    }
    if (cands.empty()) return FL_OK;
    std::vector<FusedBand> list(cands.size());
    int64_t chunks = 0, hist_len = 0;
    int nrb_max = 0;
    for (size_t c = 0; c < cands.size(); ++c) {
        const Cand& cd = cands[c];
        const BandDev& d = p.bands[cd.b].dev;
        FusedBand& f = list[c];
        f.node_off = p.bands[cd.b].node_off;
        f.nodes = p.bands[cd.b].nodes;
        f.n = d.n;
        f.kb = d.kb;
        f.l2 = cd.l2;
        f.tr = cd.TR;
        f.parts = cd.P;
        f.nq = (cd.TR + 3) / 4;
        f.nrb = (1 << cd.l2) / cd.TR;
        f.chunk0 = (int)chunks;
        f.hist0 = hist_len;
        const int64_t nc = (f.nodes + kFusedChunk - 1) / kFusedChunk;
        chunks += nc;
        hist_len += nc * f.nrb;
        nrb_max = std::max(nrb_max, f.nrb);
    }
    FusedBand* d_list = nullptr;
    int32_t* d_hist = nullptr;
    cudaError_t e = upload(p.scratch(), list, &d_list, st);
    if (e == cudaSuccess) e = p.scratch().get(&d_hist, hist_len);
    std::vector<int32_t> hist(hist_len);
    if (e == cudaSuccess) e = launch_fused_entries(p, d_list, (int)list.size(), chunks, nrb_max, false, d_hist, st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(hist.data(), d_hist, hist_len * sizeof(int32_t), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    // first entry of every (row block, chunk of nodes), row blocks first
    std::vector<int32_t> rbs;
    int64_t ents = 0, phis = 0, pp = 0;
    for (size_t c = 0; c < cands.size() && e == cudaSuccess; ++c) {
        const Cand& cd = cands[c];
        BandHost& bh = p.bands[cd.b];
        BandDev& d = bh.dev;
        FusedBand& f = list[c];
        d.fused = 1;
        d.pparts = cd.P;
        d.ent_off = f.ent_off = ents;
        d.rbs_off = (int64_t)rbs.size();
        d.ph_off = f.ph_off = phis;
        d.pp_off = pp;
        const int64_t nc = (f.nodes + kFusedChunk - 1) / kFusedChunk;
        int32_t run = 0;
        for (int rb = 0; rb < f.nrb; ++rb) {
            rbs.push_back(run);
            for (int64_t k = 0; k < nc; ++k) {
                int32_t& h = hist[f.hist0 + k * f.nrb + rb];
                const int32_t cnt = h;
                h = run;
                run += cnt;
            }
        }
        rbs.push_back(run);
        bh.fentries = run;
        ents += run;
        phis += (int64_t)run * f.nq;
        pp += (int64_t)d.nrhs * f.nodes * cd.P;   // per right-hand side: one slot per (node, row block)
        ++p.fused_bands;
    }
    p.fused_entries = ents;
    if (e == cudaSuccess) e = p.pool.bytes((void**)&p.d_frbs, rbs.size() * sizeof(int32_t));
    if (e == cudaSuccess) e = p.pool.bytes((void**)&p.d_fent, ents * sizeof(int2));
    if (e == cudaSuccess) e = p.pool.bytes((void**)&p.d_fphi, phis * sizeof(float4));
    if (e == cudaSuccess) e = p.pool.bytes((void**)&p.d_fpp, pp * sizeof(float2));
    if (e == cudaSuccess) e = cudaMemsetAsync(p.d_fphi, 0, phis * sizeof(float4), st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(p.d_frbs, rbs.data(), rbs.size() * sizeof(int32_t), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(d_hist, hist.data(), hist_len * sizeof(int32_t), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(d_list, list.data(), list.size() * sizeof(FusedBand), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = launch_fused_entries(p, d_list, (int)list.size(), chunks, nrb_max, true, d_hist, st);
    FL_CUDA(e, "fl_plan: fused gather entries");
    // slots beyond a node's parts are never written and must read as zero
    FL_CUDA(cudaMemsetAsync(p.d_fpp, 0, pp * sizeof(float2), st), "clear fused partials");
    return FL_OK;
}

// Oversampling picked from the tolerance (FP32 forward plans).  The NFFT of a
// band with K frequencies may be computed as P NFFTs over contiguous
// sub-ranges of about K/P frequencies, each centred on its own range and
// evaluated on a power-of-two grid n >= sigma_min K_p: e.g. K = 2^20 as 3
// grids of 2^19 points (sigma = 1.5) or 5 of 2^18 (sigma = 1.25) instead of
// one of 2^21 (sigma = 2) -- linearity of A~ in its frequency columns.  The
// window half-width m_w is the smallest meeting the Kaiser-Bessel estimate at
// eps/3 for the smallest sigma used (one m_w for the plan, every band at least
// as accurate); each grid gets the window shape b = pi (2 - 1/sigma) of its
// own sigma.  Split bands always gather inside pass 2 (see build_fused), so
// only bands that qualify for that are candidates.  For each floor sigma_min
// in {2, 1.75, 1.5, 1.25} every band takes its cheapest split with sigma >=
// sigma_min by an estimate of issued instructions (FFT points x (log2 n + 8),
// fused entries and partial sums, the unfused gather's taps and window
// values, at the m_w of sigma_min); the cheapest floor wins, and m_w is then
// set for the smallest sigma it actually chose.
static double fft_cost(int nrhs, int64_t n, int log2n) { return (double)nrhs * n * (log2n + 8); }

// FP32 rounding of a band grid is amplified by the deconvolution: the weights
// 1/Phi(nu) of the highest frequency (nu = 1/(2 sigma)) exceed those of the
// lowest by Phi(0)/Phi(1/(2 sigma)) ~ exp(m_w (b - sqrt(b^2 - (pi/sigma)^2))),
// b = pi (2 - 1/sigma): about 4 at sigma = 2 (m_w = 5), 29 at sigma = 1.5
// (m_w = 6), 300 at sigma = 1.31 (m_w = 7).  Sub-bands are used only where
// it stays <= 32, the factor the FP32 error bound allows for rounding.
constexpr double kMaxDeconvGain = 32.0;

static double deconv_gain(double sigma, int mw) {
    const double b = M_PI * (2.0 - 1.0 / sigma), v = M_PI / sigma;
    return exp((double)mw * (b - sqrt(b * b - v * v)));
}

// FP64 plans: the gain times the grids' rounding, 2^6 units of 2^-53, stays
// below the NFFT's share of the tolerance (e.g. <= 47 at eps = 1e-12, so
// sigma >= 1.75 there; no practical limit at 1e-6).
static double deconv_gain_limit64(double eps_A) { return eps_A * ldexp(1.0, 47); }

static double fused_cost(int64_t nodes, int log2n, int mw) {   // per right-hand side
    const int TR = pass_tiles(8, (log2n + 1) / 2, FL_P2_THREADS_F32);
    const double entries = (double)nodes * (TR + 2 * mw - 1) / TR;
    const int parts = (2 * mw - 1 + TR - 1) / TR + 1;
    return entries * 24.0 + (double)nodes * parts * 6.0;
}

struct SplitChoice {
    int P = 1, log2n = 0;
    int64_t Kp = 0, Nc = 0;
};

// The splits of a band of K frequencies that sigma >= smin and the gain limit
// admit at window half-width mw: the same for every band of these, so they are
// listed once per plan (merge_bands asks for hundreds of estimates).
static const std::vector<SplitOption>& split_options(const Plan& p, int64_t K, double smin, int mw) {
    const auto key = std::make_tuple(K, smin, mw);
    const auto hit = p.split_memo.find(key);
    if (hit != p.split_memo.end()) return hit->second;
    std::vector<SplitOption>& v = p.split_memo[key];
    const double gain_max = p.prec == FL_FP32 ? kMaxDeconvGain : deconv_gain_limit64(p.eps_A);
    // (the window shape and gain are those of the candidate's own sigma)
    for (int P = 2; P <= 9; ++P) {
        const int64_t Kp = (K + P - 1) / P;
        const int64_t Nc = Kp + (Kp & 1);
        const int lg = ilog2_ceil((int64_t)ceil(smin * (double)Nc));
        if (lg <= kSmallMaxLog2 || lg > kMaxLog2n) continue;
        const int64_t n = (int64_t)1 << lg;
        if ((double)n >= 2.0 * (double)Nc) continue;   // no gain over sigma = 2
        // the half-width this sigma needs, and the FP32 limit at it
        const int mc = std::max(mw, window_width(p.eps_A, (double)n / (double)Nc));
        if (deconv_gain((double)n / (double)Nc, mc) > gain_max) continue;
        v.push_back({P, lg, mc, Kp, Nc});
    }
    return v;
}

// Best split of band bh at sigma_min >= smin with window half-width mw
// (P = 1: unsplit); force: fewest grid points regardless of the gather.
static SplitChoice best_split(const Plan& p, const BandHost& bh, double smin, int mw, bool force,
                             double* cost) {
    const BandDev& d = bh.dev;
    SplitChoice best;
    const bool four_step = d.log2n > kSmallMaxLog2;
    // FP32: sub-bands gather inside pass 2 (fused; from their grids where that is
    // cheaper, not in pinned transforms); FP64: from their grids
    const bool fusable = p.prec == FL_FP32 && p.fuse_mode != 1;
    const bool free32 = p.prec == FL_FP32 && !p.xi_mode && !pinned(p, p.inst[bh.inst]);
    bool fz = false;
    double c1 = fft_cost(d.nrhs, d.n, d.log2n) +
                (free32 ? free_gather_cost(bh.nodes, d.nrhs, d.n, d.log2n, mw, fusable, &fz)
                 : four_step && fusable
                     ? std::min(d.nrhs * fused_cost(bh.nodes, d.log2n, mw), unfused_cost(bh.nodes, d.nrhs, mw))
                     : unfused_cost(bh.nodes, d.nrhs, mw));
    double bc = force ? (double)d.n : c1;
    const bool eligible = smin < 2.0 && four_step && !p.xi_mode && bh.nodes > 0 &&
                          (fusable || p.prec == FL_FP64);
    if (eligible) {
        for (const SplitOption& o : split_options(p, d.K, smin, mw)) {
            const int64_t n = (int64_t)1 << o.log2n;
            const double gather = free32    ? free_gather_cost(bh.nodes, d.nrhs, n, o.log2n, o.mc, fusable, &fz)
                                  : fusable ? d.nrhs * fused_cost(bh.nodes, o.log2n, o.mc)
                                            : unfused_cost(bh.nodes, d.nrhs, o.mc);
            const double c = force ? (double)o.P * n : o.P * (fft_cost(d.nrhs, n, o.log2n) + gather);
            if (c < bc) {
                bc = c;
                best.P = o.P;
                best.log2n = o.log2n;
                best.Kp = o.Kp;
                best.Nc = o.Nc;
            }
        }
    }
    *cost = best.P == 1 ? c1 : (force ? 0.0 : bc);
    return best;
}

static fl_status plan_splits(Plan& p, const std::vector<int>& nfft, cudaStream_t st) {
    p.sigma_min = 2.0;
    if (p.sigma_mode == 1 || p.xi_mode || p.prec == FL_FP64_FF || (p.prec == FL_FP32 && p.fuse_mode == 1))
        return FL_OK;
    // (sigma_mode 2: every eligible band takes its split of fewest grid points)
    const double cands[4] = {2.0, 1.75, 1.5, 1.25};   // floors (1.25: only where the gain allows)
    double best_total = 0.0;
    std::vector<SplitChoice> best_ch;
    for (double smin : cands) {
        if (p.sigma_mode == 2 && smin != 1.25) continue;   // the lowest floor, fewest grid points
        const int mw = p.mw;   // sigma = 2; a split's own sigma may need more (best_split)
        std::vector<SplitChoice> ch;
        double total = 0.0;
        for (int b : nfft) {
            double c = 0.0;
            ch.push_back(best_split(p, p.bands[b], smin, mw, p.sigma_mode >= 2, &c));
            total += c;
        }
        if (best_ch.empty() || total < best_total) {
            best_total = total;
            best_ch = ch;
        }
    }
    bool any = false;
    double smin_used = 2.0;   // the smallest sigma actually chosen fixes m_w
    for (const SplitChoice& c : best_ch)
        if (c.P > 1) {
            any = true;
            smin_used = std::min(smin_used, ldexp(1.0, c.log2n) / (double)c.Nc);
        }
    if (!any) return FL_OK;
    p.mw = std::max(p.mw, window_width(p.eps_A, smin_used));
    p.sigma_min = smin_used;
    for (size_t i = 0; i < nfft.size(); ++i) {
        const SplitChoice c = best_ch[i];
        if (c.P == 1) continue;
        const int b = nfft[i];
        const int shift = p.bands[b].dev.log2n - c.log2n;   // node cells at the sub-band grid
        const int64_t n = (int64_t)1 << c.log2n;
        const double kb = M_PI * (2.0 - (double)c.Nc / (double)n);
        const int sub0 = (int)p.bands.size();
        for (int s = 0; s < c.P; ++s) {
            BandHost ch = p.bands[b];
            const int64_t k0 = s * c.Kp;
            ch.dev.parent = b;
            ch.dev.nsub = 0;
            ch.dev.k0 = k0;
            ch.dev.K = std::min<int64_t>(c.Kp, p.bands[b].dev.K - k0);
            ch.dev.Nm = c.Nc;
            ch.dev.n = n;
            ch.dev.log2n = c.log2n;
            ch.dev.kb = kb;
            ch.dev.c_off = p.bands[b].dev.c_off + k0;
            p.bands.push_back(ch);
        }
        BandDev& d = p.bands[b].dev;
        d.nsub = c.P;
        d.sub0 = sub0;
        d.n = n;
        d.log2n = c.log2n;
        d.kb = kb;
        cudaError_t e = launch_cell_shift(p.d_cell, p.bands[b].node_off, p.bands[b].nodes, shift, st);
        if (e != cudaSuccess) return cuda_fail(e, "fl_plan: sub-band cells");
    }
    return FL_OK;
}

// ---------------------------------------------------------------------------
// Merged bands.  The dyadic bands with l_m = 1 all keep the same K frequencies,
// each with q right-hand sides, although on the ones near the circle y xi is
// small and exp(-y xi) all but linear there.  Neighbouring ones are therefore
// interpolated together, in y alone (the weights exp(-y_s k) are exact at the
// Chebyshev points y_s of the union), at the rank that leaves no larger an
// error than rank q leaves on a single dyadic band: at N = M = 2^20, eps = 1e-6 the
// six bands of the clustered nodes take 35 right-hand sides instead of 72, at
// 2^18 and 1e-12 nine bands 82 instead of 198.  In FP64 a directly summed band
// only where another band goes through an NFFT anyway, and then with wider windows
// (widen_windows): where all were direct, merging raised the error at 300 x 5000 and
// eps = 1e-10 from 6.6e-15 to 3.8e-14 (adjoint 6.7e-16 to 8.9e-15), and the call took
// 148 us instead of 45.

// Bounds of the interpolation error of exp(-y x) on y in [a, b], relative to the
// kernel's bound 1, at 0 .. kMaxQ points: the Chebyshev coefficients of
// exp(-(c + h t) x) are 2 (-1)^j I_j(h x) e^{-c x}, and interpolation at q Chebyshev
// points errs by at most twice the sum of the coefficients from q on; the
// largest over x in (0, xmax], sampled four to the octave over the top three
// octaves (the bounds are unimodal in x, and the bands reach at most about that
// far beyond the peak).
static void interp_error(double a, double b, double xmax, double tol, double* err) {
    constexpr int kTerms = 96, kSamples = 13, kPad = 16;   // (padded: the loops over the samples are vectors)
    constexpr double kQuarter[4] = {1.0, 0.84089641525371454, 0.70710678118654752, 0.59460355750136053};
    const double h = 0.5 * (b - a);
    // e^-z I_j(z) <= (z/2)^j / j!: the terms from J on are below tol 10^-8 together
    int J = 1;
    for (double t = 0.5 * h * xmax; J < kTerms && t > 1e-9 * tol; t *= 0.5 * h * xmax / ++J)
        ;
    double iz[kPad], scale[kPad], sum[kPad], p[kTerms + 2][kPad];
    for (int i = 0; i < kPad; ++i) {
        const int k = std::min(i, kSamples - 1);
        const double x = ldexp(xmax * kQuarter[k & 3], -(k >> 2));
        iz[i] = 2.0 / (h * x);
        scale[i] = 4.0 * exp(-a * x);
        sum[i] = p[0][i] = 1.0;
        p[J + 1][i] = 0.0;
    }
    for (int j = J + 1; j <= kMaxQ; ++j) err[j] = 0.0;
    // I_j(z) / I_{j-1}(z) backwards, then I_j / I_0 = their products, normalised by I_0 + 2 sum I_j = e^z
    for (int j = J; j > 0; --j)
        for (int i = 0; i < kPad; ++i) p[j][i] = 1.0 / (j * iz[i] + p[j + 1][i]);
    for (int j = 1; j <= J; ++j)
        for (int i = 0; i < kPad; ++i) {
            p[j][i] *= p[j - 1][i];
            sum[i] += 2.0 * p[j][i];
        }
    for (int i = 0; i < kPad; ++i) {
        scale[i] /= sum[i];
        sum[i] = 0.0;                            // from here the tails
    }
    for (int j = J; j >= 0; --j) {
        double most = 0.0;
        for (int i = 0; i < kPad; ++i) {
            sum[i] += p[j][i] * scale[i];
            most = std::max(most, sum[i]);
        }
        if (j <= kMaxQ) err[j] = most;
    }
}

// The smallest rank whose bound on [a, 2^octaves a], x <= xmax, is at most tol
// (kMaxQ + 1: none).  It depends on a xmax alone, rounded up to a sixteenth of an
// octave and kept per plan (a batch asks for the same few again and again).
static int merged_rank(Plan& p, double a, int octaves, double xmax, double tol) {
    const int key = (int)ceil(16.0 * log2(a * xmax));
    const auto hit = p.rank_memo.find({octaves, key});
    if (hit != p.rank_memo.end()) return hit->second;
    // beyond z = h x = 60 the coefficients fall below 1e-6 after kMaxQ only
    const double b = ldexp(1.0, std::min(octaves, 60)), xm = pow(2.0, key / 16.0);
    int r = kMaxQ + 1;
    if (0.5 * (b - 1.0) * xm <= 60.0) {
        double err[kMaxQ + 1];
        interp_error(1.0, b, xm, tol, err);
        r = 2;
        while (r <= kMaxQ && err[r] > tol) ++r;
    }
    p.rank_memo[{octaves, key}] = r;
    return r;
}

// FP64 plans that merge a directly summed band take windows one point wider on
// each side: nodes without a window error come under one, 1.2 times the error
// against 64 bits of the bands before (5.5e-14 against 4.5e-14 at N = M = 3000, eps =
// 1e-10).  A point more divides the window's error by e^(2 pi sqrt(1 - 1/sigma)) (85
// at sigma = 2: 8.7e-16 there) and costs two taps per node and right-hand side.  Not
// below kWindowEps, where the NFFT errs by rounding (at 1e-12 1.0e-15 either way), and
// not where the gain would pass its limit.
constexpr double kWindowEps = 0x1p-36;
static void widen_windows(Plan& p) {
    if (p.prec != FL_FP64 || !p.merged_direct || p.eps < kWindowEps || p.mw >= 12) return;
    if (deconv_gain(p.sigma_min, p.mw + 1) <= deconv_gain_limit64(p.eps_A)) ++p.mw;
}

// Estimated cost of an NFFT band (the units of route_of), at its best split.
static double nfft_cost(const Plan& p, const BandHost& bh) {
    double best = 0.0;
    const bool split = p.sigma_mode != 1 && !p.xi_mode && p.prec != FL_FP64_FF && bh.dev.log2n > kSmallMaxLog2;
    for (double smin : {2.0, 1.75, 1.5, 1.25}) {
        double c = 0.0;
        best_split(p, bh, smin, p.mw, false, &c);
        if (smin == 2.0 || c < best) best = c;
        if (!split) break;
    }
    return best + 2.0e5;
}

// Merges neighbouring non-empty bands of a transform with l_m = 1 (where bands
// are routed by cost and the rank comes from eps: a caller's q is that of every
// band; and not in pinned transforms): the partition of least
// estimated cost by dynamic programming; a band left alone keeps its route and
// Algorithm 2's weights.  The nodes of a merged band are put in cell order (they
// are consecutive and share a grid size) under its first band.
static fl_status merge_bands(Plan& p, const Instance& in, cudaStream_t st) {
    if ((p.route_mode != 0 && !p.xi_mode) || p.q_given || pinned(p, in)) return FL_OK;
    std::vector<int> list;   // candidates, ascending band
    for (int lb = 1; lb < in.levels; ++lb)
        if (p.bands[in.band_base + lb].nodes > 0 && p.bands[in.band_base + lb].ell == 1) list.push_back(lb);
    const int n = (int)list.size();
    if (n == 0) return FL_OK;
    // FP64: where every band is summed directly the transform has no error but
    // rounding, and keeps it
    bool merge_direct = p.prec != FL_FP64;
    for (int lb = 1; lb <= in.levels; ++lb) merge_direct |= p.bands[in.band_base + lb].dev.route == 1;
    double tol;
    {
        double err[kMaxQ + 1];   // the dyadic band at rank q, over every x
        interp_error(1.0, 2.0, 64.0, 0.0, err);
        tol = err[p.q];
        // in double an error below half a unit of rounding is none (rank 22 at
        // eps = 1e-12 leaves 6e-18)
        if (p.prec != FL_FP32) tol = std::max(tol, ldexp(1.0, -54));
    }
    // A direct term is dearer in the model than in fact, next to an NFFT of many
    // right-hand sides.  FP64 and float pairs at eps = 1e-10, N = 1024 to 65536, M =
    // 1000 to 10000 near the circle: with estimates 1.4 to 3.9 times the merged
    // band's the direct sums were faster (16384 x 3000, 3.9: 259 us against 439
    // merged; 65536 x 1000, 1.4: 273 against 768; pairs 1024 x 10000, 3.8: 58 against
    // 84), from 5.8 on the merged band (4096 x 10000, 5.8: 222 against 159; 65536 x
    // 10000, 6.9: 2057 against 1487).  FP32 at 1e-6: 270001 x 3000 78 us against 312,
    // 600000 x 6000 171 against 293 (merged at a share of 4.5).
    const double direct_share = p.prec == FL_FP32 ? 7.0 : 4.5;
    struct Part {
        double cost;
        int from, rank;
    };
    std::vector<Part> best(n + 1, Part{0.0, 0, 0});
    std::vector<int64_t> before(n + 1, 0);          // nodes of the candidates before
    for (int t = 0; t < n; ++t) before[t + 1] = before[t] + p.bands[in.band_base + list[t]].nodes;
    auto merged = [&](int i, int j, int rank) {   // candidates list[i .. j] as one band
        BandHost g = p.bands[in.band_base + list[i]];
        g.nodes = before[j + 1] - before[i];
        const double a = ldexp(p.y1, -list[j]), b = ldexp(p.y1, 1 - list[i]);
        g.dev.nodes = g.nodes;
        g.dev.yc = 0.5 * (a + b);
        g.dev.yh = 0.5 * (b - a);
        g.dev.yh_inv = 1.0 / g.dev.yh;
        g.dev.nrhs = rank;
        return g;
    };
    std::vector<int> floor_rank(n, 2);               // known of the interval from candidate i on
    for (int j = 0; j < n; ++j) {
        const BandHost& alone = p.bands[in.band_base + list[j]];
        const double single = alone.dev.route == 2
                                  ? (double)alone.nodes * alone.dev.K * 6.0 * p.direct_bias / direct_share
                                  : nfft_cost(p, alone);
        best[j + 1] = Part{best[j].cost + single, j, 0};
        int least = 2;   // the rank grows with the interval: no less than those of parts of it
        for (int i = j; i >= 0; --i) {
            if (!merge_direct && p.bands[in.band_base + list[i]].dev.route == 2) break;
            least = floor_rank[i] = std::max(floor_rank[i], least);
            if (best[i].cost + nfft_cost(p, merged(i, j, least)) >= best[j + 1].cost) continue;   // not even at that rank
            const int r = merged_rank(p, ldexp(p.y1, -list[j]), list[j] - list[i] + 1, in.xi1, tol);
            if (r > kMaxQ) break;
            least = floor_rank[i] = r;
            if (i == j && r >= p.q) continue;
            const double c = best[i].cost + nfft_cost(p, merged(i, j, r));
            if (c < best[j + 1].cost) best[j + 1] = Part{c, i, r};
        }
    }
    for (int j = n; j > 0; j = best[j].from) {
        const int i = best[j].from, r = best[j].rank;
        if (r == 0) continue;
        for (int t = i; t < j; ++t)
            p.merged_direct |= p.bands[in.band_base + list[t]].dev.route == 2;
        const int lead = in.band_base + list[i];
        const BandHost g = merged(i, j - 1, r);
        for (int t = i; t < j; ++t) {
            BandHost& bh = p.bands[in.band_base + list[t]];
            bh.leader = lead;
            bh.nodes = bh.dev.nodes = 0;
            bh.dev.route = 0;
        }
        const int64_t own = p.bands[lead].own;
        p.bands[lead] = g;
        p.bands[lead].own = own;
        p.bands[lead].leader = lead;
        p.bands[lead].dev.route = 1;
        int off = 0, k = 0;
        while (k < (int)p.ranks.size() && p.ranks[k] != r) off += p.ranks[k++];
        if (k == (int)p.ranks.size()) p.ranks.push_back(r);
        p.bands[lead].dev.choff = off;
        p.qmax = std::max(p.qmax, r);
        if (i == j - 1) continue;   // one band at a lower rank: its nodes are in order
        const cudaError_t e = launch_cell_sort(p, g.node_off, g.nodes, lead, g.dev.log2n, st);
        if (e != cudaSuccess) return cuda_fail(e, "fl_plan: merged bands");
    }
    return FL_OK;
}

// Plans the transforms Ns[i] x Ms[i], i < B, whose nodes are consecutive in
// `nodes` (a single plan is B = 1).  Every band of every transform gets an
// entry of one global band table, and each kernel launch of fl_execute covers
// all transforms at once.
static fl_status plan_multi(Plan& p, int B, const int64_t* Ns, const int64_t* Ms,
                            const double* nodes, int q, bool shared, cudaStream_t st) {
    fl_status s = select_common(p, q);
    if (s != FL_OK) return s;
    p.bands.clear();
    p.inst.assign(B, Instance());
    int64_t noff = 0, moff = 0, maxM = 0;
    for (int i = 0; i < B; ++i) {
        Instance& in = p.inst[i];
        in.N = Ns[i];
        in.M = Ms[i];
        in.noff = noff;
        in.moff = moff;
        in.src_off = shared ? 0 : moff;
        // a shared node set: the first transform of the same N is sorted, the
        // others copy its order (same bands, cells and routes)
        for (int j = 0; shared && j < i && in.twin < 0; ++j)
            if (Ns[j] == in.N) in.twin = j;
        noff += in.N;
        moff += in.M;
        maxM = std::max(maxM, in.M);
        if ((s = select_bands(p, in, i)) != FL_OK) return s;
    }
    p.N = noff;
    p.M = moff;
    p.levels = p.inst[0].levels;
    p.xi1 = p.inst[0].xi1;
    int nb = (int)p.bands.size();
    const auto al = DevPool::rounded;
    const int64_t nodes_all = moff;
    const int64_t sort_hist = 256 * ((maxM + 2047) / 2048);   // radix-sort tiles of 2048
    const size_t sort_bytes = 5 * al(maxM * 4) + al(maxM * sizeof(double2)) + al(sort_hist * 4) +
                              al(nb * sizeof(int64_t)) + al(sizeof(int));
    p.small = nodes_all <= kSmallPlan;
    FL_CUDA(p.pool.reserve(al(nb * sizeof(BandDev)) + al(16) + al(nodes_all * sizeof(double2)) + 3 * al(nodes_all * 4) +
                           (p.small ? sort_bytes + ((size_t)1 << 17) : 0)),
            "cudaMalloc nodes");
    FL_CUDA(p.pool.bytes((void**)&p.d_bands, nb * sizeof(BandDev)), "cudaMalloc bands");
    std::vector<BandDev> hb(nb);
    for (int b = 0; b < nb; ++b) hb[b] = p.bands[b].dev;
    FL_CUDA(cudaMemcpyAsync(p.d_bands, hb.data(), nb * sizeof(BandDev), cudaMemcpyHostToDevice, st),
            "copy bands");
    FL_CUDA(p.pool.bytes(&p.d_z0, 2 * sizeof(double)), "cudaMalloc z0");

    // classify and sort the nodes of every transform into its slice
    const int64_t M = p.M;
    std::vector<int64_t> counts(nb, 0);
    if (M > 0) {
        FL_CUDA(p.pool.bytes((void**)&p.d_ws, M * sizeof(double2)), "cudaMalloc nodes");
        FL_CUDA(p.pool.bytes((void**)&p.d_perm, M * sizeof(int32_t)), "cudaMalloc perm");
        FL_CUDA(p.pool.bytes((void**)&p.d_bandid, M * sizeof(int32_t)), "cudaMalloc band ids");
        FL_CUDA(p.pool.bytes((void**)&p.d_cell, M * sizeof(int32_t)), "cudaMalloc cells");
        SortScratch& ss = p.sort;
        int64_t* dcount = nullptr;
        int* dflag = nullptr;
        cudaError_t e = p.scratch().reserve(sort_bytes);
        if (e == cudaSuccess && (e = p.scratch().get(&ss.keys, maxM)) == cudaSuccess &&
            (e = p.scratch().get(&ss.keys2, maxM)) == cudaSuccess && (e = p.scratch().get(&ss.vals, maxM)) == cudaSuccess &&
            (e = p.scratch().get(&ss.vals2, maxM)) == cudaSuccess && (e = p.scratch().get(&ss.perm, maxM)) == cudaSuccess &&
            (e = p.scratch().get(&ss.ws, maxM)) == cudaSuccess && (e = p.scratch().get(&ss.hist, sort_hist)) == cudaSuccess &&
            (e = p.scratch().get(&dcount, nb)) == cudaSuccess && (e = p.scratch().get(&dflag, 1)) == cudaSuccess &&
            (e = cudaMemsetAsync(dcount, 0, nb * sizeof(int64_t), st)) == cudaSuccess &&
            (e = cudaMemsetAsync(dflag, 0, sizeof(int), st)) == cudaSuccess) {
            for (int i = 0; i < B && e == cudaSuccess; ++i) {
                const Instance& in = p.inst[i];
                if (in.twin >= 0) {
                    e = launch_copy_sorted(p, in, p.inst[in.twin], st);
                    continue;
                }
                if ((e = launch_classify(p, in, nodes, ss.keys, ss.vals, dcount, dflag, st)) == cudaSuccess &&
                    (e = radix_sort_pairs(ss.keys, ss.vals, ss.keys2, ss.vals2, ss.hist, in.M, 32, st)) == cudaSuccess)
                    e = launch_permute(p, in, nodes, ss.keys, ss.vals, st);
            }
            int flag = 0;
            if (e == cudaSuccess)
                e = cudaMemcpyAsync(counts.data(), dcount, nb * sizeof(int64_t), cudaMemcpyDeviceToHost, st);
            if (e == cudaSuccess) e = cudaMemcpyAsync(&flag, dflag, sizeof(int), cudaMemcpyDeviceToHost, st);
            if (e == cudaSuccess) e = cudaStreamSynchronize(st);
            if (e == cudaSuccess && flag)
                return fail(FL_EINVAL, p.xi_mode ? "fl_plan_xi: a node has Im w < 0, a non-finite part or |Re w| > 1/2"
                                                 : "fl_plan: a node has Im w < 0 or a non-finite part");
        }
        if (e != cudaSuccess) return cuda_fail(e, "fl_plan: node classification");
        for (const Instance& in : p.inst)
            if (in.twin >= 0)
                for (int lb = 0; lb <= in.levels; ++lb)
                    counts[in.band_base + lb] = counts[p.inst[in.twin].band_base + lb];
    }

    // routes, offsets and work lists
    p.grid_elems = p.D_elems = p.Y_elems = 0;
    p.xqc = p.xi_mode ? xi_chunk(p.q) : 0;
    p.small_work.clear();
    p.large_bands.clear();
    p.direct_segs.clear();
    p.direct_terms = 0;
    p.z0_nodes = 0;
    p.ranks.assign(1, p.q);
    p.qmax = p.q;
    p.own_gather = p.merged_direct = false;
    for (const Instance& in : p.inst) p.own_gather = p.own_gather || !pinned(p, in);
    std::vector<int> nfft_bands;   // bands evaluated by an NFFT, in order
    for (int i = 0; i < B; ++i) {
        Instance& in = p.inst[i];
        in.z0_nodes = counts[in.band_base];
        p.z0_nodes += in.z0_nodes;
        int64_t off = in.moff + in.z0_nodes;
        p.bands[in.band_base].node_off = in.moff;
        p.bands[in.band_base].dev.node_off = in.moff;
        p.bands[in.band_base].nodes = in.z0_nodes;
        for (int lb = 1; lb <= in.levels; ++lb) {
            const int b = in.band_base + lb;
            BandHost& bh = p.bands[b];
            bh.nodes = bh.own = counts[b];
            bh.node_off = off;
            off += counts[b];
            BandDev& d = bh.dev;
            d.node_off = bh.node_off;
            d.nodes = bh.nodes;
            d.route = bh.nodes > 0 ? route_of(p, bh) : 0;
        }
        if ((s = merge_bands(p, in, st)) != FL_OK) return s;
        for (int lb = 1; lb <= in.levels; ++lb) {
            const int b = in.band_base + lb;
            BandHost& bh = p.bands[b];
            BandDev& d = bh.dev;
            if (d.route == 2) {
                p.direct_terms += bh.nodes * d.K;
                add_direct_band(p, bh);
                continue;
            }
            if (d.route == 1) nfft_bands.push_back(b);
        }
    }
    if (M > kTmpKeep) {   // large: planning's scratch given back before the grids are allocated
        FL_CUDA(cudaStreamSynchronize(st), "fl_plan: synchronise");
        p.tmp.release();
    }
    // oversampling from the tolerance: split sparse bands into sub-bands
    if ((s = plan_splits(p, nfft_bands, st)) != FL_OK) return s;
    widen_windows(p);
    // a transform that copies its twin's nodes shares its twin's weight tables
    // (same N, bands and splits); shares_D[i] records that every band did
    std::vector<char> shares_D(B, 0);
    for (int i = 0; i < B; ++i) shares_D[i] = p.inst[i].twin >= 0 && !p.xi_mode;
    for (int b : nfft_bands) {
        const int nsub = p.bands[b].dev.nsub;
        const Instance& in = p.inst[p.bands[b].inst];
        const int tb = in.twin >= 0 ? b - in.band_base + p.inst[in.twin].band_base : -1;
        const bool twin_ok = tb >= 0 && p.bands[tb].dev.route == 1 && p.bands[tb].dev.nsub == nsub &&
                             p.bands[tb].dev.K == p.bands[b].dev.K;
        if (tb >= 0 && !twin_ok) shares_D[p.bands[b].inst] = 0;
        for (int c = 0; c < std::max(1, nsub); ++c) {
            const int g = nsub > 0 ? p.bands[b].dev.sub0 + c : b;
            BandDev& d = p.bands[g].dev;
            d.grid_off = p.grid_elems;
            p.grid_elems += (int64_t)d.nrhs * d.n;
            if (twin_ok && !p.xi_mode) {
                d.D_off = p.bands[nsub > 0 ? p.bands[tb].dev.sub0 + c : tb].dev.D_off;
            } else if (p.xi_mode) {
                // exponent-major rows of whole spreading chunks, 16-byte aligned
                d.dld = d.nrhs == 1 ? 1 : (d.nrhs + p.xqc - 1) / p.xqc * p.xqc;
                p.D_elems = (p.D_elems + 3) & ~(int64_t)3;
                d.D_off = p.D_elems;
                p.D_elems += (int64_t)d.dld * d.K;
            } else {
                d.D_off = p.D_elems;
                p.D_elems += (int64_t)d.nrhs * d.K;
            }
            if (d.log2n <= kSmallMaxLog2) {
                // 4096 points per CTA (256 threads x 16); n = 32 at 8 points per thread
                const int per = std::max(1, (int)((d.log2n >= 6 ? 4096 : 2048) / d.n));
                for (int s0 = 0; s0 < d.nrhs; s0 += per)
                    p.small_work.push_back({g, s0, std::min(per, d.nrhs - s0), d.log2n});
            } else {
                p.large_bands.push_back(g);
            }
        }
    }
    build_direct_items(p);
    build_pass_groups(p);
    if ((s = build_fused(p, st)) != FL_OK) return s;
    if ((int)p.bands.size() != nb) {   // sub-bands were appended: a larger table
        nb = (int)p.bands.size();
        hb.resize(nb);
        FL_CUDA(p.pool.bytes((void**)&p.d_bands, nb * sizeof(BandDev)), "cudaMalloc bands");
    }
    for (int b = 0; b < nb; ++b) hb[b] = p.bands[b].dev;
    FL_CUDA(cudaMemcpyAsync(p.d_bands, hb.data(), nb * sizeof(BandDev), cudaMemcpyHostToDevice, st),
            "copy bands");
    const size_t cs = p.prec != FL_FP32 ? 16 : 8, rs = cs / 2;   // complex128 I/O for FP64 and float pairs
    {   // one block for what follows (128 KiB of it for lists that are not known yet)
        size_t n = (size_t)1 << 17;
        auto add = [&](bool on, int64_t count, size_t size) { n += on ? al((size_t)count * size) : 0; };
        const bool node_tables = !p.batched && !(p.small_work.empty() && p.large_bands.empty());
        add(true, (int64_t)p.small_work.size(), sizeof(SmallWork));
        add(true, (int64_t)p.pass_items.size(), sizeof(PassItem));
        add(true, (int64_t)(p.direct_work.size() + p.dadj_work.size()), sizeof(DirectItem));
        add(p.prec == FL_FP32 && !p.xi_mode, M, sizeof(uint4));
        add(true, p.dpart_elems, cs);
        add(!p.dadj_work.empty(), p.N, cs);
        add(true, 2 * p.base_nodes, cs);
        add(node_tables, M * 2 * p.mw, rs);
        add(node_tables, M * p.qmax, rs);
        add(node_tables, M, cs);
        add(node_tables, M, cs);
        add(true, p.grid_elems, cs);
        add(true, p.D_elems, rs);
        add(true, p.Y_elems, cs);
        add(!p.small_work.empty() || p.Y_elems > 0, kTwEntries + 8192, cs);
        add(p.prec == FL_FP64_FF, p.N, sizeof(ffc));
        if (n > ((size_t)1 << 18) && n < kOneBlock) FL_CUDA(p.pool.reserve(n), "cudaMalloc tables and grids");
    }
    if (p.prec == FL_FP32 && !p.xi_mode && p.M > 0) {
        FL_CUDA(p.pool.bytes((void**)&p.d_ntab, p.M * sizeof(uint4)), "cudaMalloc node records");
        FL_CUDA(build_node_table(p, st), "fl_plan: node records");
    }
    if (!p.small_work.empty()) {
        FL_CUDA(p.pool.bytes((void**)&p.d_small, p.small_work.size() * sizeof(SmallWork)), "cudaMalloc work");
        FL_CUDA(cudaMemcpyAsync(p.d_small, p.small_work.data(), p.small_work.size() * sizeof(SmallWork),
                                cudaMemcpyHostToDevice, st),
                "copy work");
    }
    if (!p.pass_items.empty()) {
        FL_CUDA(p.pool.bytes((void**)&p.d_pass, p.pass_items.size() * sizeof(PassItem)), "cudaMalloc pass items");
        FL_CUDA(cudaMemcpyAsync(p.d_pass, p.pass_items.data(), p.pass_items.size() * sizeof(PassItem),
                                cudaMemcpyHostToDevice, st),
                "copy pass items");
    }
    if (!p.direct_work.empty()) {
        FL_CUDA(upload(p.pool, p.direct_segs, &p.d_dsegs, st), "fl_plan: direct segments");
        FL_CUDA(upload(p.pool, p.direct_work, &p.d_direct, st), "fl_plan: direct work");
        FL_CUDA(upload(p.pool, p.direct_ranges, &p.d_dranges, st), "fl_plan: direct ranges");
        FL_CUDA(upload(p.pool, p.dadj_work, &p.d_dadj, st), "fl_plan: adjoint work");
        if (p.dpart_elems > 0) FL_CUDA(p.pool.bytes(&p.d_dpart, p.dpart_elems * cs), "cudaMalloc direct partials");
        if (!p.dadj_work.empty()) FL_CUDA(p.pool.bytes(&p.d_cdir, p.N * cs), "cudaMalloc direct adjoint");
        if (p.base_nodes > 0) {
            FL_CUDA(p.pool.bytes(&p.d_dz, 2 * p.base_nodes * cs), "cudaMalloc direct bases");
            FL_CUDA(build_direct_base(p, st), "fl_plan: direct bases");
        }
    }
    // adjoint of the NFFT bands (single plans): per-node taps and weights, cell lists
    if (!p.batched && M > 0) {
        FL_CUDA(build_spread(p, st), "fl_plan: adjoint lists");
        if (p.n_sp_blocks + p.n_dn_groups[0] + p.n_dn_groups[1] > 0) {
            FL_CUDA(p.pool.bytes(&p.d_sp_phi, (size_t)M * 2 * p.mw * rs), "cudaMalloc adjoint taps");
            FL_CUDA(p.pool.bytes(&p.d_sp_L, (size_t)M * p.qmax * rs), "cudaMalloc adjoint weights");
            FL_CUDA(p.pool.bytes(&p.d_sp_e, (size_t)M * cs), "cudaMalloc adjoint shifts");
            FL_CUDA(p.pool.bytes(&p.d_sp_rv, (size_t)M * cs), "cudaMalloc adjoint residuals");
        }
    }
    if (p.grid_elems) FL_CUDA(p.pool.bytes(&p.d_grid, p.grid_elems * cs), "cudaMalloc grids");
    if (p.D_elems) FL_CUDA(p.pool.bytes(&p.d_D, p.D_elems * rs), "cudaMalloc weights");
    if (p.D_elems && p.xi_mode)   // the padding of the exponent-major rows
        FL_CUDA(cudaMemsetAsync(p.d_D, 0, p.D_elems * rs, st), "clear weights");
    if (p.Y_elems) FL_CUDA(p.pool.bytes(&p.d_Y, p.Y_elems * cs), "cudaMalloc intermediate");
    if (p.Y_elems || !p.small_work.empty()) {   // stage twiddles of the passes and the small FFTs
        FL_CUDA(p.pool.bytes(&p.d_tw, (size_t)(kTwEntries + (p.prec != FL_FP32 ? 8192 : 0)) * cs),
                "cudaMalloc twiddles");
        FL_CUDA(build_twiddles(p, st), "fl_plan: twiddles");
    }
    if (p.prec == FL_FP64_FF)
        FL_CUDA(p.pool.bytes(&p.d_cff, (size_t)p.N * sizeof(ffc)), "cudaMalloc float-pair coefficients");
    int cheb_len = 0;
    for (int r : p.ranks) cheb_len += r;
    FL_CUDA(p.pool.bytes((void**)&p.d_cheb, 2 * cheb_len * sizeof(double)), "cudaMalloc cheb");
    FL_CUDA(p.pool.bytes((void**)&p.d_cheb32, 4 * cheb_len * sizeof(float)), "cudaMalloc cheb32");
    FL_CUDA(build_cheb(p, st), "fl_plan: tables");
    if (p.d_sp_phi) FL_CUDA(build_node_weights(p, st), "fl_plan: node weights");
    for (int i = 0; i < B; ++i)
        if (!shares_D[i]) FL_CUDA(build_tables(p, p.inst[i], st), "fl_plan: tables");
    FL_CUDA(cudaStreamSynchronize(st), "fl_plan: synchronise");
    p.tmp.release();
    p.scratch_bytes = (double)p.grid_elems * cs + (double)p.D_elems * rs + (double)p.Y_elems * cs +
                      (double)M * (sizeof(double2) + 8) + (double)p.dpart_elems * cs +
                      (p.direct_work.empty() ? 0.0 : 2.0 * p.base_nodes * cs + (double)(p.dadj_work.empty() ? 0 : p.N) * cs);
    // algorithmic bytes of one execute: c once, D once, each grid written and read
    // once per FFT pass, the nodes, and f
    double mb = (double)p.N * cs + (double)p.D_elems * rs + (double)M * (sizeof(double2) + 8 + cs);
    for (int b = 0; b < nb; ++b) {
        const BandDev& d = p.bands[b].dev;
        if (d.route != 1 || d.nsub > 0) continue;   // split bands: their sub-bands
        const double g = (double)d.nrhs * d.n * cs;
        if (d.fused) {   // Y write + read; entries read, partials written and gathered
            const int NQ = (pass_tiles(8, (d.log2n + 1) / 2, FL_P2_THREADS_F32) + 3) / 4;
            mb += 2.0 * g + (double)d.nrhs * p.bands[b].fentries * (8.0 + 16.0 * NQ + 8.0) +
                  (double)d.nrhs * p.bands[b].nodes * d.pparts * cs;
            continue;
        }
        mb += (d.log2n <= kSmallMaxLog2) ? g : 3.0 * g;   // small: write; large: Y write+read, grid write
        mb += std::min<double>(g, (double)p.bands[b].nodes * d.nrhs * 2 * p.mw * cs);   // gather
    }
    if (!p.direct_work.empty())   // c tiles
        mb += (double)p.direct_work.size() * std::min<int64_t>(p.direct_kmax, kDirChunk) * cs;
    p.model_bytes = mb;
    return FL_OK;
}


// Everything that defines a Fourier-Laplace plan besides the route bias.
struct PlanSpec {
    int B;
    const int64_t* Ns;
    const int64_t* Ms;
    const double* nodes;
    int q;
    double eps;
    fl_precision prec;
    bool batched;
    int route_mode;
    int rhs_per_launch;
    bool use_graph;
    int variant;
    int fuse_mode;
    int sigma_mode;
    bool shared_nodes;
};

static fl_status build_plan(const PlanSpec& sp, double bias, fl_plan_s** out, cudaStream_t st) {
    fl_plan_s* h = new (std::nothrow) fl_plan_s();
    if (!h) return fail(FL_ENOMEM, "fl_plan: host allocation");
    h->p.kind = 0;
    h->p.batched = sp.batched;
    h->p.prec = sp.prec;
    h->p.eps = sp.eps;
    h->p.route_mode = sp.route_mode;
    h->p.direct_bias = bias;
    h->p.rhs_per_launch = sp.rhs_per_launch;
    h->p.use_graph = sp.use_graph;
    h->p.variant = sp.variant;
    h->p.fuse_mode = sp.fuse_mode;
    h->p.sigma_mode = sp.sigma_mode;
    fl_status s = plan_multi(h->p, sp.B, sp.Ns, sp.Ms, sp.nodes, sp.q, sp.shared_nodes, st);
    if (s != FL_OK) {
        delete h;
        return s;
    }
    *out = h;
    return FL_OK;
}

// Autotuner: plans the workload for candidate settings, times three executes
// of each (CUDA events on the caller's stream, after one warm-up, on zero
// coefficients: the work does not depend on the values), and keeps the
// fastest.  Coordinate search, each setting from the best so far: the route
// bias (route 0), then -- where the caller left them at their defaults -- the
// oversampling (sigma from the tolerance or 2), the fused gather (by cost or
// never) and the grids per four-step launch.  The choice is cached for the
// process by a signature of the workload (sizes, eps, precision, the caller's
// settings and the node count of every band), so planning the same workload
// again costs one plan.
struct Tuned {
    double bias;
    int sigma_mode, fuse_mode, rhs;
};
static std::vector<std::pair<uint64_t, Tuned>> g_tuned;
static std::mutex g_tuned_mutex;

static uint64_t plan_signature(const Plan& p, const PlanSpec& sp) {
    uint64_t h = 1469598103934665603ull;
    auto mix = [&](uint64_t v) { h = (h ^ v) * 1099511628211ull; };
    mix((uint64_t)p.N);
    mix((uint64_t)p.M);
    mix((uint64_t)p.inst.size());
    mix((uint64_t)p.prec);
    uint64_t e;
    memcpy(&e, &p.eps, sizeof(e));
    mix(e);
    mix((uint64_t)p.q);
    mix((uint64_t)p.variant);
    mix((uint64_t)sp.route_mode);
    mix((uint64_t)sp.sigma_mode);
    mix((uint64_t)sp.fuse_mode);
    mix((uint64_t)sp.rhs_per_launch);
    for (const Instance& in : p.inst) mix((uint64_t)(in.twin + 1));
    for (const BandHost& bh : p.bands) mix((uint64_t)bh.own * 131 + (uint64_t)bh.local);   // before merging
    return h;
}

static fl_status time_plan(Plan& p, cudaStream_t st, double* ms) {
    const size_t cs = p.prec != FL_FP32 ? 16 : 8;
    void *c = nullptr, *f = nullptr;
    cudaEvent_t a = nullptr, b = nullptr;
    cudaError_t e = cudaMalloc(&c, std::max<int64_t>(1, p.N) * cs);
    if (e == cudaSuccess) e = cudaMalloc(&f, std::max<int64_t>(1, p.M) * cs);
    if (e == cudaSuccess) e = cudaMemsetAsync(c, 0, std::max<int64_t>(1, p.N) * cs, st);
    if (e == cudaSuccess) e = cudaEventCreate(&a);
    if (e == cudaSuccess) e = cudaEventCreate(&b);
    const int64_t launches = p.launches;
    if (e == cudaSuccess) e = run_forward(p, c, f, false, st);
    if (e == cudaSuccess) e = cudaEventRecord(a, st);
    for (int r = 0; r < 3 && e == cudaSuccess; ++r) e = run_forward(p, c, f, false, st);
    if (e == cudaSuccess) e = cudaEventRecord(b, st);
    if (e == cudaSuccess) e = cudaEventSynchronize(b);
    float t = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&t, a, b);
    p.launches = launches;
    if (a) cudaEventDestroy(a);
    if (b) cudaEventDestroy(b);
    cudaFree(c);
    cudaFree(f);
    if (e != cudaSuccess) return cuda_fail(e, "fl_plan: autotune");
    *ms = t / 3.0;
    return FL_OK;
}

static PlanSpec with_tuned(const PlanSpec& sp, const Tuned& t) {
    PlanSpec r = sp;
    r.sigma_mode = t.sigma_mode;
    r.fuse_mode = t.fuse_mode;
    r.rhs_per_launch = t.rhs;
    return r;
}

static void set_tuned(Plan& p, const Tuned& t) {
    p.tuned_bias = t.bias;
    p.tuned_sigma_mode = t.sigma_mode;
    p.tuned_fuse_mode = t.fuse_mode;
    p.tuned_rhs = t.rhs;
}

static fl_status build_plan_tuned(const PlanSpec& sp, double bias, bool autotune, fl_plan_s** out,
                                  cudaStream_t st) {
    fl_plan_s* h = nullptr;
    fl_status s = build_plan(sp, bias, &h, st);
    if (s != FL_OK || !autotune) {
        *out = h;
        return s;
    }
    const uint64_t sig = plan_signature(h->p, sp);
    const Tuned start{bias, sp.sigma_mode, sp.fuse_mode, sp.rhs_per_launch};
    bool hit = false;
    Tuned cached = start;
    {
        std::lock_guard<std::mutex> lock(g_tuned_mutex);
        for (const auto& kv : g_tuned)
            if (kv.first == sig) {
                cached = kv.second;
                hit = true;
            }
    }
    if (hit) {
        if (cached.bias != start.bias || cached.sigma_mode != start.sigma_mode ||
            cached.fuse_mode != start.fuse_mode || cached.rhs != start.rhs) {
            delete h;
            h = nullptr;
            if ((s = build_plan(with_tuned(sp, cached), cached.bias, &h, st)) != FL_OK) return s;
        }
        set_tuned(h->p, cached);
        *out = h;
        return FL_OK;
    }
    double best_ms = 0;
    if ((s = time_plan(h->p, st, &best_ms)) != FL_OK) {
        delete h;
        return s;
    }
    Tuned best = start;
    auto try_cand = [&](const Tuned& t) -> fl_status {
        fl_plan_s* c = nullptr;
        fl_status r = build_plan(with_tuned(sp, t), t.bias, &c, st);
        if (r != FL_OK) return r;
        double ms = 0;
        if ((r = time_plan(c->p, st, &ms)) != FL_OK) {
            delete c;
            return r;
        }
        if (ms < best_ms) {
            delete h;
            h = c;
            best_ms = ms;
            best = t;
        } else {
            delete c;
        }
        return FL_OK;
    };
    std::vector<Tuned> cands;
    const bool fp32 = sp.prec == FL_FP32;
    if (sp.route_mode == 0)
        for (double cand : {0.125, 0.25, 0.5, 2.0, 4.0, 8.0}) {
            Tuned t = best;
            t.bias = cand;
            if ((s = try_cand(t)) != FL_OK) break;
        }
    if (s == FL_OK && fp32 && sp.sigma_mode == 0) {
        Tuned t = best;
        t.sigma_mode = 1;
        s = try_cand(t);
    }
    if (s == FL_OK && fp32 && sp.fuse_mode == 0) {
        Tuned t = best;
        t.fuse_mode = 1;
        s = try_cand(t);
    }
    if (s == FL_OK && sp.rhs_per_launch == 0)
        for (int r : {12, 36}) {
            Tuned t = best;
            t.rhs = r;
            if ((s = try_cand(t)) != FL_OK) break;
        }
    if (s != FL_OK) {
        delete h;
        return s;
    }
    {
        std::lock_guard<std::mutex> lock(g_tuned_mutex);
        g_tuned.push_back({sig, best});
    }
    set_tuned(h->p, best);
    *out = h;
    return FL_OK;
}

// The forward transform where f may overlap c.  The direct bands write their
// results while other blocks still read c, and the Z^0 nodes read c_0 in the last
// kernel; the FFT passes are through with c before anything is written, and the
// float-pair form reads a converted copy.  Where it matters, c is copied first
// (stream-ordered scratch: the call stays asynchronous and can be captured).
static bool reads_c_late(const Plan& p, const void* c, const void* f) {
    if (p.z0_nodes == 0 && (p.direct_work.empty() || p.prec == FL_FP64_FF)) return false;
    const size_t cs = p.prec != FL_FP32 ? 16 : 8;
    const uintptr_t a = (uintptr_t)c, b = (uintptr_t)f;
    return a < b + (size_t)p.M * cs && b < a + (size_t)p.N * cs;
}

static cudaError_t forward_call(Plan& p, const void* c, void* f, bool deriv, const void* rmul, cudaStream_t st) {
    if (!reads_c_late(p, c, f)) return run_forward(p, c, f, deriv, st, rmul);
    const size_t bytes = (size_t)p.N * (p.prec != FL_FP32 ? 16 : 8);
    void* copy = nullptr;
    cudaError_t e = cudaMallocAsync(&copy, bytes, st);
    if (e != cudaSuccess) return e;
    e = cudaMemcpyAsync(copy, c, bytes, cudaMemcpyDeviceToDevice, st);
    if (e == cudaSuccess) e = run_forward(p, copy, f, deriv, st, rmul);
    const cudaError_t e2 = cudaFreeAsync(copy, st);
    return e != cudaSuccess ? e : e2;
}

// fl_execute through a CUDA graph of its launches, captured on the first call
// (and again when the buffers or the stream change), then replayed.
static cudaError_t forward_graphed(Plan& p, const void* c, void* f, cudaStream_t st) {
    if (!p.use_graph || p.timing || st == nullptr || reads_c_late(p, c, f))
        return forward_call(p, c, f, false, nullptr, st);
    if (!p.gexec || p.g_c != c || p.g_f != f || p.g_st != st) {
        if (p.gexec) {
            cudaGraphExecDestroy(p.gexec);
            p.gexec = nullptr;
        }
        cudaError_t e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
        if (e != cudaSuccess) return e;
        const int64_t launches = p.launches;
        cudaError_t er = run_forward(p, c, f, false, st);
        cudaGraph_t g = nullptr;
        e = cudaStreamEndCapture(st, &g);
        if (er != cudaSuccess) {
            if (g) cudaGraphDestroy(g);
            return er;
        }
        if (e != cudaSuccess) return e;
        e = cudaGraphInstantiate(&p.gexec, g, 0);
        cudaGraphDestroy(g);
        if (e != cudaSuccess) {
            p.gexec = nullptr;
            return e;
        }
        p.graph_launches = p.launches - launches;
        p.launches = launches;
        p.g_c = c;
        p.g_f = f;
        p.g_st = st;
    }
    p.launches += p.graph_launches;
    return cudaGraphLaunch(p.gexec, st);
}

// Batched plans with per-transform buffers: element e of the concatenation
// belongs to transform b with off[b] <= e < off[b + 1] (binary search);
// pack copies the callers' arrays into the concatenation, unpack back out.
template <typename E>
__global__ void k_batch_pack(int B, const int64_t* __restrict__ off, const E* const* __restrict__ src,
                             int64_t total, E* __restrict__ dst) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= total) return;
    int lo = 0, hi = B;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= e) lo = mid;
        else hi = mid;
    }
    dst[e] = src[lo][e - off[lo]];
}

template <typename E>
__global__ void k_batch_unpack(int B, const int64_t* __restrict__ off, const E* __restrict__ src,
                               int64_t total, E* const* __restrict__ dst) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= total) return;
    int lo = 0, hi = B;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= e) lo = mid;
        else hi = mid;
    }
    dst[lo][e - off[lo]] = src[e];
}

// pack: c pointers -> d_stage_c; else d_stage_f -> f pointers (offsets and
// pointers from d_boff / d_bptr).
static cudaError_t launch_batch_pack(Plan& p, size_t cs, bool pack, cudaStream_t st) {
    const int B = (int)p.inst.size();
    const int64_t total = pack ? p.N : p.M;
    if (total == 0) return cudaSuccess;
    const unsigned grid = (unsigned)((total + 255) / 256);
    const int64_t* off = pack ? p.d_boff : p.d_boff + B + 1;
    if (cs == 16) {
        if (pack)
            k_batch_pack<double2><<<grid, 256, 0, st>>>(B, off, (const double2* const*)p.d_bptr, total,
                                                        (double2*)p.d_stage_c);
        else
            k_batch_unpack<double2><<<grid, 256, 0, st>>>(B, off, (const double2*)p.d_stage_f, total,
                                                          (double2* const*)(p.d_bptr + B));
    } else {
        if (pack)
            k_batch_pack<float2><<<grid, 256, 0, st>>>(B, off, (const float2* const*)p.d_bptr, total,
                                                       (float2*)p.d_stage_c);
        else
            k_batch_unpack<float2><<<grid, 256, 0, st>>>(B, off, (const float2*)p.d_stage_f, total,
                                                         (float2* const*)(p.d_bptr + B));
    }
    ++p.launches;
    return cudaGetLastError();
}

}  // namespace fl

using namespace fl;

extern "C" {

const char* fl_last_error(void) { return g_err.c_str(); }

const char* fl_version(void) { return "fastfl 0.1 (sm_103a)"; }

static bool options_valid(const fl_options* opt) {
    return !opt || (opt->route >= 0 && opt->route <= 2 && opt->direct_bias >= 0.0 &&
                    opt->rhs_per_launch >= 0 && opt->variant >= 0 && opt->variant <= 1 &&
                    opt->fuse_gather >= 0 && opt->fuse_gather <= 2 && opt->oversampling >= 0 &&
                    opt->oversampling <= 2 && opt->shared_nodes >= 0 && opt->shared_nodes <= 1);
}

fl_status fl_plan(fl_plan_t* out, int64_t N, int64_t M, const double* nodes_dev, int q, double eps,
                  fl_precision prec, void* stream) {
    return fl_plan_ex(out, N, M, nodes_dev, q, eps, prec, nullptr, stream);
}

fl_status fl_plan_ex(fl_plan_t* out, int64_t N, int64_t M, const double* nodes_dev, int q,
                     double eps, fl_precision prec, const fl_options* opt, void* stream) {
    g_err.clear();
    if (!options_valid(opt))
        return fail(FL_EINVAL, "fl_plan: invalid options");
    if (!out) return fail(FL_EINVAL, "fl_plan: out is NULL");
    *out = nullptr;
    if (N < 1 || M < 0) return fail(FL_EINVAL, "fl_plan: need N >= 1 and M >= 0");
    if (N > ((int64_t)1 << 23)) return fail(FL_EUNSUPPORTED, "fl_plan: N above 2^23");
    if (M > ((int64_t)1 << 31) - 1) return fail(FL_EUNSUPPORTED, "fl_plan: M above 2^31 - 1");
    if (!(eps > 0.0 && eps < 1.0)) return fail(FL_EINVAL, "fl_plan: eps must lie in (0, 1)");
    if (q < 0 || q > kMaxQ) return fail(FL_EINVAL, "fl_plan: q must lie in [0, 40]");
    if (prec != FL_FP32 && prec != FL_FP64 && prec != FL_FP64_FF)
        return fail(FL_EINVAL, "fl_plan: unknown precision");
    if (M > 0 && !nodes_dev) return fail(FL_EINVAL, "fl_plan: nodes is NULL");
    PlanSpec sp{1, &N, &M, nodes_dev, q, eps, prec, false,
                 opt ? opt->route : 0, opt ? opt->rhs_per_launch : 0, opt ? opt->use_graph != 0 : false,
                 opt ? opt->variant : 0, opt ? opt->fuse_gather : 0, opt ? opt->oversampling : 0,
                 false};
    const double bias = (opt && opt->direct_bias > 0.0) ? opt->direct_bias : 1.0;
    fl_plan_s* h = nullptr;
    fl_status s = build_plan_tuned(sp, bias, opt && opt->autotune, &h, (cudaStream_t)stream);
    if (s != FL_OK) return s;
    *out = h;
    return FL_OK;
}

fl_status fl_execute(fl_plan_t h, const void* c_dev, void* f_dev, void* stream) {
    if (!h || h->p.kind != 0) return fail(FL_EINVAL, "fl_execute: not a Fourier-Laplace plan");
    if (h->p.M > 0 && (!c_dev || !f_dev)) return fail(FL_EINVAL, "fl_execute: NULL buffer");
    if (h->p.batched) return fail(FL_EINVAL, "fl_execute: batched plan (use fl_execute_batched)");
    cudaError_t e = h->p.xi_mode ? run_forward_xi(h->p, c_dev, f_dev, (cudaStream_t)stream)
                                 : forward_graphed(h->p, c_dev, f_dev, (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(e, "fl_execute");
    return FL_OK;
}

fl_status fl_execute_deriv(fl_plan_t h, const void* c_dev, void* f_dev, void* stream) {
    if (!h || h->p.kind != 0) return fail(FL_EINVAL, "fl_execute_deriv: not a Fourier-Laplace plan");
    if (h->p.M > 0 && (!c_dev || !f_dev)) return fail(FL_EINVAL, "fl_execute_deriv: NULL buffer");
    if (h->p.batched) return fail(FL_EUNSUPPORTED, "fl_execute_deriv: batched plans are forward only");
    if (h->p.xi_mode) return fail(FL_EUNSUPPORTED, "fl_execute_deriv: real-exponent plans are forward only");
    cudaError_t e = forward_call(h->p, c_dev, f_dev, true, nullptr, (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(e, "fl_execute_deriv");
    return FL_OK;
}

fl_status fl_grad_w(fl_plan_t h, const void* c_dev, const void* r_dev, void* gw_dev, void* stream) {
    if (!h || h->p.kind != 0) return fail(FL_EINVAL, "fl_grad_w: not a Fourier-Laplace plan");
    if (h->p.M > 0 && (!c_dev || !r_dev || !gw_dev)) return fail(FL_EINVAL, "fl_grad_w: NULL buffer");
    if (h->p.batched) return fail(FL_EUNSUPPORTED, "fl_grad_w: batched plans are forward only");
    if (h->p.xi_mode) return fail(FL_EUNSUPPORTED, "fl_grad_w: real-exponent plans are forward only");
    cudaError_t e = forward_call(h->p, c_dev, gw_dev, true, r_dev, (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(e, "fl_grad_w");
    return FL_OK;
}

fl_status fl_execute_host(fl_plan_t h, const void* c_host, void* f_host, void* stream) {
    if (!h || h->p.kind != 0) return fail(FL_EINVAL, "fl_execute_host: not a Fourier-Laplace plan");
    Plan& p = h->p;
    if (!c_host || (p.M > 0 && !f_host)) return fail(FL_EINVAL, "fl_execute_host: NULL buffer");
    const size_t cs = p.prec != FL_FP32 ? 16 : 8;
    cudaStream_t st = (cudaStream_t)stream;
    if (!p.d_stage_c) FL_CUDA(cudaMalloc(&p.d_stage_c, p.N * cs), "cudaMalloc staging");
    if (!p.d_stage_f && p.M > 0) FL_CUDA(cudaMalloc(&p.d_stage_f, p.M * cs), "cudaMalloc staging");
    FL_CUDA(cudaMemcpyAsync(p.d_stage_c, c_host, p.N * cs, cudaMemcpyHostToDevice, st), "copy c");
    FL_CUDA(p.xi_mode ? run_forward_xi(p, p.d_stage_c, p.d_stage_f, st)
                      : forward_graphed(p, p.d_stage_c, p.d_stage_f, st),
            "fl_execute_host");
    if (p.M > 0)
        FL_CUDA(cudaMemcpyAsync(f_host, p.d_stage_f, p.M * cs, cudaMemcpyDeviceToHost, st), "copy f");
    FL_CUDA(cudaStreamSynchronize(st), "fl_execute_host: synchronise");
    return FL_OK;
}

fl_status fl_adjoint(fl_plan_t h, const void* r_dev, void* c_out_dev, void* stream) {
    if (!h || h->p.kind != 0) return fail(FL_EINVAL, "fl_adjoint: not a Fourier-Laplace plan");
    if (!c_out_dev || (h->p.M > 0 && !r_dev)) return fail(FL_EINVAL, "fl_adjoint: NULL buffer");
    if (h->p.batched) return fail(FL_EUNSUPPORTED, "fl_adjoint: batched plans are forward only");
    cudaError_t e = run_adjoint(h->p, r_dev, c_out_dev, (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(e, "fl_adjoint");
    return FL_OK;
}

fl_status fl_transposed(fl_plan_t h, const void* g_dev, void* out_dev, void* stream) {
    if (!h || h->p.kind != 0) return fail(FL_EINVAL, "fl_transposed: not a Fourier-Laplace plan");
    if (!out_dev || (h->p.M > 0 && !g_dev)) return fail(FL_EINVAL, "fl_transposed: NULL buffer");
    if (h->p.batched) return fail(FL_EUNSUPPORTED, "fl_transposed: batched plans are forward only");
    cudaError_t e = run_transposed(h->p, g_dev, out_dev, (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(e, "fl_transposed");
    return FL_OK;
}

fl_status fl_plan_xi(fl_plan_t* out, int64_t N, const double* xi_dev, int64_t M,
                     const double* nodes_dev, int q, double eps, fl_precision prec, void* stream) {
    g_err.clear();
    if (!out) return fail(FL_EINVAL, "fl_plan_xi: out is NULL");
    *out = nullptr;
    if (N < 1 || M < 0) return fail(FL_EINVAL, "fl_plan_xi: need N >= 1 and M >= 0");
    if (N > ((int64_t)1 << 22) || M > ((int64_t)1 << 31) - 1)
        return fail(FL_EUNSUPPORTED, "fl_plan_xi: N above 2^22 or M above 2^31 - 1");
    if (!(eps > 0.0 && eps < 1.0)) return fail(FL_EINVAL, "fl_plan_xi: eps must lie in (0, 1)");
    if (q < 0 || q > kMaxQ) return fail(FL_EINVAL, "fl_plan_xi: q must lie in [0, 40]");
    if (prec != FL_FP32 && prec != FL_FP64) return fail(FL_EINVAL, "fl_plan_xi: unknown precision");
    if (!xi_dev || (M > 0 && !nodes_dev)) return fail(FL_EINVAL, "fl_plan_xi: NULL argument");
    cudaStream_t st = (cudaStream_t)stream;
    std::vector<double> xh(N);
    FL_CUDA(cudaMemcpyAsync(xh.data(), xi_dev, N * sizeof(double), cudaMemcpyDeviceToHost, st), "copy xi");
    FL_CUDA(cudaStreamSynchronize(st), "fl_plan_xi: synchronise");
    std::vector<std::pair<double, int32_t>> order(N);
    for (int64_t k = 0; k < N; ++k) {
        if (!(xh[k] >= 1.0) || !std::isfinite(xh[k]))
            return fail(FL_EINVAL, "fl_plan_xi: every exponent must be finite and >= 1");
        order[k] = {xh[k], (int32_t)k};
    }
    std::stable_sort(order.begin(), order.end(),
                     [](const std::pair<double, int32_t>& a, const std::pair<double, int32_t>& b) {
                         return a.first < b.first;
                     });
    fl_plan_s* h = new (std::nothrow) fl_plan_s();
    if (!h) return fail(FL_ENOMEM, "fl_plan_xi: host allocation");
    Plan& p = h->p;
    p.kind = 0;
    p.prec = prec;
    p.eps = eps;
    p.route_mode = 1;
    p.xi_mode = true;
    p.h_xis.resize(N);
    std::vector<int32_t> perm(N);
    for (int64_t k = 0; k < N; ++k) {
        p.h_xis[k] = order[k].first;
        perm[k] = order[k].second;
    }
    auto bail = [&](fl_status s) {
        delete h;
        return s;
    };
    cudaError_t e = p.pool.bytes((void**)&p.d_xis, N * sizeof(double));
    if (e == cudaSuccess) e = p.pool.bytes((void**)&p.d_xperm, N * sizeof(int32_t));
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(p.d_xis, p.h_xis.data(), N * sizeof(double), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(p.d_xperm, perm.data(), N * sizeof(int32_t), cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return bail(cuda_fail(e, "fl_plan_xi: exponents"));
    fl_status s = plan_multi(p, 1, &N, &M, nodes_dev, q, false, st);
    if (s != FL_OK) return bail(s);
    e = build_xi_tables(p, st);
    if (e != cudaSuccess) return bail(cuda_fail(e, "fl_plan_xi: tables"));
    *out = h;
    return FL_OK;
}

fl_status fl_plan_batched(fl_plan_t* out, int B, const int64_t* N_host, const int64_t* M_host,
                          const double* nodes_dev, int q, double eps, fl_precision prec,
                          const fl_options* opt, void* stream) {
    g_err.clear();
    if (!out) return fail(FL_EINVAL, "fl_plan_batched: out is NULL");
    *out = nullptr;
    if (B < 1 || !N_host || !M_host) return fail(FL_EINVAL, "fl_plan_batched: need B >= 1 and sizes");
    int64_t Mtot = 0, Ntot = 0;
    for (int i = 0; i < B; ++i) {
        if (N_host[i] < 1 || M_host[i] < 0)
            return fail(FL_EINVAL, "fl_plan_batched: need N_i >= 1 and M_i >= 0");
        if (N_host[i] > ((int64_t)1 << 23)) return fail(FL_EUNSUPPORTED, "fl_plan_batched: N_i above 2^23");
        Ntot += N_host[i];
        Mtot += M_host[i];
    }
    if (Mtot > ((int64_t)1 << 31) - 1 || Ntot > ((int64_t)1 << 40))
        return fail(FL_EUNSUPPORTED, "fl_plan_batched: sum of M_i above 2^31 - 1");
    if (!(eps > 0.0 && eps < 1.0)) return fail(FL_EINVAL, "fl_plan_batched: eps must lie in (0, 1)");
    if (q < 0 || q > kMaxQ) return fail(FL_EINVAL, "fl_plan_batched: q must lie in [0, 40]");
    if (prec != FL_FP32 && prec != FL_FP64 && prec != FL_FP64_FF)
        return fail(FL_EINVAL, "fl_plan_batched: unknown precision");
    if (Mtot > 0 && !nodes_dev) return fail(FL_EINVAL, "fl_plan_batched: nodes is NULL");
    if (!options_valid(opt))
        return fail(FL_EINVAL, "fl_plan_batched: invalid options");
    const bool shared = opt && opt->shared_nodes;
    for (int i = 1; shared && i < B; ++i)
        if (M_host[i] != M_host[0])
            return fail(FL_EINVAL, "fl_plan_batched: shared nodes need every M_i equal to M_0");
    PlanSpec sp{B, N_host, M_host, nodes_dev, q, eps, prec, true, opt ? opt->route : 0,
                 opt ? opt->rhs_per_launch : 0, opt ? opt->use_graph >= 0 : true,
                 opt ? opt->variant : 0, opt ? opt->fuse_gather : 0, opt ? opt->oversampling : 0,
                 shared};
    const double bias = (opt && opt->direct_bias > 0.0) ? opt->direct_bias : 1.0;
    fl_plan_s* h = nullptr;
    fl_status s = build_plan_tuned(sp, bias, opt && opt->autotune, &h, (cudaStream_t)stream);
    if (s != FL_OK) return s;
    *out = h;
    return FL_OK;
}

fl_status fl_execute_batched(fl_plan_t h, const void* c_dev, void* f_dev, void* stream) {
    if (!h || h->p.kind != 0 || !h->p.batched)
        return fail(FL_EINVAL, "fl_execute_batched: not a batched Fourier-Laplace plan");
    if (h->p.M > 0 && (!c_dev || !f_dev)) return fail(FL_EINVAL, "fl_execute_batched: NULL buffer");
    cudaError_t e = forward_graphed(h->p, c_dev, f_dev, (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(e, "fl_execute_batched");
    return FL_OK;
}

fl_status fl_plan_batched_ptrs(fl_plan_t* out, int B, const int64_t* N_host, const int64_t* M_host,
                               const double* const* nodes_host, int q, double eps, fl_precision prec,
                               const fl_options* opt, void* stream) {
    g_err.clear();
    if (!out) return fail(FL_EINVAL, "fl_plan_batched_ptrs: out is NULL");
    *out = nullptr;
    if (B < 1 || !N_host || !M_host) return fail(FL_EINVAL, "fl_plan_batched_ptrs: need B >= 1 and sizes");
    if (opt && opt->shared_nodes)   // one node set: the first pointer
        return fl_plan_batched(out, B, N_host, M_host, nodes_host ? nodes_host[0] : nullptr, q, eps, prec,
                               opt, stream);
    int64_t Mtot = 0;
    for (int i = 0; i < B; ++i) {
        if (M_host[i] < 0) return fail(FL_EINVAL, "fl_plan_batched_ptrs: need M_i >= 0");
        if (M_host[i] > 0 && (!nodes_host || !nodes_host[i]))
            return fail(FL_EINVAL, "fl_plan_batched_ptrs: nodes of a transform with M_i > 0 is NULL");
        Mtot += M_host[i];
    }
    if (Mtot > ((int64_t)1 << 31) - 1) return fail(FL_EUNSUPPORTED, "fl_plan_batched_ptrs: sum of M_i above 2^31 - 1");
    cudaStream_t st = (cudaStream_t)stream;
    double* cat = nullptr;   // the node sets concatenated, for planning only
    if (Mtot > 0) {
        FL_CUDA(cudaMalloc(&cat, Mtot * 2 * sizeof(double)), "cudaMalloc nodes");
        int64_t off = 0;
        for (int i = 0; i < B; ++i) {
            if (M_host[i] > 0) {
                const cudaError_t e = cudaMemcpyAsync(cat + 2 * off, nodes_host[i], M_host[i] * 2 * sizeof(double),
                                                      cudaMemcpyDeviceToDevice, st);
                if (e != cudaSuccess) {
                    cudaFree(cat);
                    return cuda_fail(e, "fl_plan_batched_ptrs: copy nodes");
                }
            }
            off += M_host[i];
        }
    }
    fl_status s = fl_plan_batched(out, B, N_host, M_host, cat, q, eps, prec, opt, stream);
    if (cat) {
        const cudaError_t e = cudaStreamSynchronize(st);
        cudaFree(cat);
        if (e != cudaSuccess && s == FL_OK) {
            fl_destroy(*out);
            *out = nullptr;
            return cuda_fail(e, "fl_plan_batched_ptrs: synchronise");
        }
    }
    return s;
}

fl_status fl_execute_batched_ptrs(fl_plan_t h, const void* const* c_host, void* const* f_host, void* stream) {
    if (!h || h->p.kind != 0 || !h->p.batched)
        return fail(FL_EINVAL, "fl_execute_batched_ptrs: not a batched Fourier-Laplace plan");
    Plan& p = h->p;
    const int B = (int)p.inst.size();
    if (!c_host || (p.M > 0 && !f_host)) return fail(FL_EINVAL, "fl_execute_batched_ptrs: NULL pointer array");
    for (int i = 0; i < B; ++i) {
        if (!c_host[i]) return fail(FL_EINVAL, "fl_execute_batched_ptrs: NULL coefficients");
        if (p.inst[i].M > 0 && !f_host[i]) return fail(FL_EINVAL, "fl_execute_batched_ptrs: NULL result");
    }
    const size_t cs = p.prec != FL_FP32 ? 16 : 8;
    cudaStream_t st = (cudaStream_t)stream;
    if (!p.d_stage_c) FL_CUDA(cudaMalloc(&p.d_stage_c, p.N * cs), "cudaMalloc staging");
    if (!p.d_stage_f && p.M > 0) FL_CUDA(cudaMalloc(&p.d_stage_f, p.M * cs), "cudaMalloc staging");
    if (!p.d_boff) {   // instance offsets, fixed for the plan
        std::vector<int64_t> off(2 * (B + 1));
        for (int i = 0; i < B; ++i) {
            off[i] = p.inst[i].noff;
            off[B + 1 + i] = p.inst[i].moff;
        }
        off[B] = p.N;
        off[2 * B + 1] = p.M;
        FL_CUDA(cudaMalloc((void**)&p.d_boff, off.size() * sizeof(int64_t)), "cudaMalloc offsets");
        FL_CUDA(cudaMemcpy(p.d_boff, off.data(), off.size() * sizeof(int64_t), cudaMemcpyHostToDevice),
                "copy offsets");
        FL_CUDA(cudaMalloc((void**)&p.d_bptr, 2 * (size_t)B * sizeof(void*)), "cudaMalloc pointer table");
    }
    // the caller's pointers (pageable host memory: the copy is staged before
    // the call returns, so the arrays may be reused at once)
    std::vector<const void*> ptrs(2 * (size_t)B, nullptr);
    for (int i = 0; i < B; ++i) {
        ptrs[i] = c_host[i];
        ptrs[B + i] = p.M > 0 ? f_host[i] : nullptr;
    }
    FL_CUDA(cudaMemcpyAsync(p.d_bptr, ptrs.data(), ptrs.size() * sizeof(void*), cudaMemcpyHostToDevice, st),
            "copy pointer table");
    FL_CUDA(launch_batch_pack(p, cs, true, st), "fl_execute_batched_ptrs: gather coefficients");
    FL_CUDA(forward_graphed(p, p.d_stage_c, p.d_stage_f, st), "fl_execute_batched_ptrs");
    if (p.M > 0) FL_CUDA(launch_batch_pack(p, cs, false, st), "fl_execute_batched_ptrs: scatter results");
    return FL_OK;
}

fl_status fl_get_band_rhs(fl_plan_t h, int* rhs, int count) {
    if (!h || !rhs || count < 0 || count > FL_MAX_LEVELS) return fail(FL_EINVAL, "fl_get_band_rhs: invalid argument");
    const Plan& p = h->p;
    const int nb = p.kind == 0 && !p.inst.empty() ? p.inst[0].levels + 1 : 0;
    for (int b = 0; b < count; ++b)
        rhs[b] = b > 0 && b < nb && p.bands[b].dev.route == 1 ? p.bands[b].dev.nrhs : 0;
    return FL_OK;
}

fl_status fl_get_info(fl_plan_t h, fl_info* info) {
    if (!h || !info) return fail(FL_EINVAL, "fl_get_info: NULL argument");
    const Plan& p = h->p;
    memset(info, 0, sizeof(*info));
    info->kind = p.kind;
    info->precision = p.prec;
    info->N = p.N;
    info->M = p.M;
    info->eps = p.eps;
    info->eps_laplace = p.eps_K;
    info->eps_fourier = p.eps_A;
    info->q = p.q;
    info->levels = p.levels;
    info->m_w = p.mw;
    info->sigma = 2;
    info->y1 = p.y1;
    info->xi1 = p.xi1;
    info->z0_nodes = p.z0_nodes;
    info->batch = p.batched ? (int)p.inst.size() : 1;
    if (p.kind == 0) {   // bands of all transforms: routes counted over the batch
        for (const BandHost& bh : p.bands) {
            if (bh.local == 0 || bh.dev.parent >= 0) continue;   // sub-bands count with their band
            if (bh.dev.route == 1 || bh.leader >= 0) ++info->n_bands_fft;
            if (bh.dev.route == 2) ++info->n_bands_direct;
        }
    }
    const int nb_first = p.kind == 0 && !p.inst.empty() ? p.inst[0].levels + 1 : (int)p.bands.size();
    for (int b = 1; b < nb_first && b < (int)p.bands.size() && b < FL_MAX_LEVELS; ++b) {
        const BandHost& bh = p.bands[b];
        const BandDev& ev = p.kind == 0 && bh.leader >= 0 ? p.bands[bh.leader].dev : bh.dev;   // what evaluates it
        info->band_ell[b] = bh.ell;
        info->band_route[b] = ev.route;
        info->band_nodes[b] = bh.own;
        info->band_K[b] = bh.dev.K;
        info->band_n[b] = ev.n;
        info->band_parts[b] = ev.nsub > 0 ? ev.nsub : 1;
    }
    info->model_bytes = p.model_bytes;
    info->direct_bias = p.tuned_bias > 0 ? p.tuned_bias : p.direct_bias;
    info->scratch_bytes = p.scratch_bytes;
    info->variant = p.variant;
    info->kernel = p.kind == 1 ? p.lap_kernel : 0;
    info->n_bands_fused = (int)p.fused_bands;
    info->fused_entries = p.fused_entries;
    info->sigma_min = p.sigma_min;
    info->rhs_per_launch = p.rhs_per_launch;
    info->oversampling = p.sigma_mode;
    info->fuse_gather = p.fuse_mode;
    info->autotuned = p.tuned_rhs >= 0 ? 1 : 0;
    return FL_OK;
}

fl_status fl_set_timing(fl_plan_t h, int enable) {
    if (!h) return fail(FL_EINVAL, "fl_set_timing: NULL plan");
    Plan& p = h->p;
    for (Timer& t : p.timers) {
        cudaEventDestroy(t.start);
        cudaEventDestroy(t.stop);
    }
    p.timers.clear();
    p.timing = enable != 0;
    p.launches = 0;
    return FL_OK;
}

fl_status fl_get_timing(fl_plan_t h, fl_timing* out) {
    if (!h || !out) return fail(FL_EINVAL, "fl_get_timing: NULL argument");
    Plan& p = h->p;
    memset(out, 0, sizeof(*out));
    for (Timer& t : p.timers) {
        cudaError_t e = cudaEventSynchronize(t.stop);
        if (e != cudaSuccess) return cuda_fail(e, "fl_get_timing");
        float ms = 0.f;
        e = cudaEventElapsedTime(&ms, t.start, t.stop);
        if (e != cudaSuccess) return cuda_fail(e, "fl_get_timing");
        int slot = -1;
        for (int i = 0; i < out->n_kernels; ++i)
            if (t.name == out->name[i]) slot = i;
        if (slot < 0) {
            if (out->n_kernels >= FL_MAX_TIMED_KERNELS) continue;
            slot = out->n_kernels++;
            snprintf(out->name[slot], sizeof(out->name[slot]), "%s", t.name.c_str());
        }
        out->launches[slot] += 1;
        out->total_ms[slot] += ms;
        out->bytes[slot] += t.bytes;
    }
    out->total_launches = p.launches;
    return FL_OK;
}

void fl_destroy(fl_plan_t h) {
    if (!h) return;
    cudaDeviceSynchronize();
    delete h;
}

}  // extern "C"
