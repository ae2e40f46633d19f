// Swendsen-Wang sweep as a degenerate duality (Section 4.3).
//
// For a ferromagnetic Potts-type table exp(l_x [x_s = x_t]) with l_x >= 0 the
// dual variable of an edge is one bond bit: given x it is 1 with probability
// 1 - e^{-l_{x_s}} when x_s = x_t (never otherwise); given the bonds, the
// bonds' connected components (clusters) take one label each, cluster K
// label x with weight exp(sum_{v in K} u_v(x) + sum_{bonds in K} log(e^{l_x} - 1)).
//
// One sweep on the device, items (site or edge, chain) with the chain
// innermost so that a warp works on one site or edge for many chains.  Between
// sweeps every site is its own tree (parent[v][c] = v), its ban word is 0 and
// its weight row lw[v][c][.] is 0; a sweep touches only what its bonds reach
// and restores that state:
//   k_sw_bond     bond draws; each bond unions its endpoints' trees, adds its
//                 label weights to its source site's row and marks both
//                 endpoints bonded
//   k_sw_flatten  every bonded site records its root (the smallest site of its
//                 cluster) and adds its unaries and row into the root's row
//   k_sw_draw     every root (bonded or not) draws its cluster's label from
//                 its unaries plus its row
//   k_sw_assign   bonded non-roots copy the root's label; rows, parents and
//                 ban words of bonded sites are reset.
// Only about a fifth of the (edge, chain) items agree in their labels, 7 % are
// bonded and a third of the sites are bonded (ferromagnetic lattice, beta ~
// U[0, 1], 8 labels), at random lanes.  Each kernel therefore scans its items
// four chains per lane, and its warps collect the items that need the next
// step in a shared-memory queue and run it with full warps (WarpQueue).
// Weight rows keep the labels innermost, so that the 8 L bytes of a row are
// whole sectors.  Measured on 48^3, L = 8, 64 chains (us per sweep): bond and union
// 265 -> 94, flatten 194 -> 81, draw and assign 273 -> 149.
// Unaries enter as fixed-point values precomputed once per factor change.
// Higdon's partial Swendsen-Wang (k_hg_*) runs the same kernels with its own
// bond tables and per-chain potentials in place of the unaries; small models
// run whole Swendsen-Wang sweeps in one single-CTA launch (k_sw_small).
// The union-find is lock-free: a link always points from a root to a smaller
// site (atomicCAS on the root's entry), so every walk visits strictly
// decreasing sites and ends within N steps; a walk that exceeds that bound
// sets the error flag instead of looping (the host then resets the state).
// The forest of a chain is its own column of parent[][], so chains never
// contend.
#include "sweep_impl.cuh"   // draw_label

#include <algorithm>

namespace mrfk {

namespace {

__device__ __forceinline__ int64_t pidx(int32_t v, int32_t c, int32_t C) { return (int64_t)v * C + c; }

// Root of v, halving the path on the way (loads bypass L1: other threads
// rewrite entries meanwhile).  A halving store replaces a non-root's parent by
// one of its ancestors, so it never meets a link (links only rewrite roots)
// and any interleaving of halving stores leaves a forest with the same roots.
// Roots found by k_sw_flatten go to a separate array, not into parent[][]: a
// halving store landing after such a write would leave a non-root there.
// Returns -1 when the step bound is exceeded.
__device__ __forceinline__ int32_t sw_find(int32_t* __restrict__ par, int32_t v, int32_t c, int32_t C, int32_t N) {
    for (int32_t step = 0; step <= N; ++step) {
        const int32_t p = __ldcg(par + pidx(v, c, C));
        if (p == v) return v;
        const int32_t gp = __ldcg(par + pidx(p, c, C));
        if (gp != p) par[pidx(v, c, C)] = gp;
        v = gp;
    }
    return -1;
}

// Union of the trees of a and b: the larger root is linked to the smaller one.
// A failed link means that root was linked meanwhile; the retry starts from
// roots strictly smaller than before, so at most N retries happen.
__device__ __forceinline__ bool sw_union(int32_t* __restrict__ par, int32_t a, int32_t b, int32_t c, int32_t C,
                                         int32_t N) {
    for (int32_t step = 0; step <= N; ++step) {
        a = sw_find(par, a, c, C, N);
        b = sw_find(par, b, c, C, N);
        if (a < 0 || b < 0) return false;
        if (a == b) return true;
        if (a < b) { const int32_t t = a; a = b; b = t; }
        if (atomicCAS(par + pidx(a, c, C), a, b) == a) return true;
    }
    return false;
}

__device__ __forceinline__ void red_add_s64(int64_t* p, int64_t v) {
    atomicAdd(reinterpret_cast<unsigned long long*>(p), (unsigned long long)v);
}

}  // namespace

// sw_fix of a float32 value without float64 arithmetic: the value is
// m 2^(e - 150) with a 24-bit mantissa m, so its fixed-point form m 2^(e - 118)
// is a shift of m (rounded half away from zero when it drops bits; |f| < 2^30
// is guaranteed by the model check).
__device__ __forceinline__ int64_t fix_from_float(float f) {
    const uint32_t bits = __float_as_uint(f);
    const int e = (int)((bits >> 23) & 0xFFu);
    if (e == 0) return 0;                                          // zero and subnormals (|f| < 2^-126)
    const int64_t m = (int64_t)((bits & 0x7FFFFFu) | 0x800000u);
    const int sh = e - 118;
    int64_t v;
    if (sh >= 0) v = m << (sh < 38 ? sh : 38);
    else if (sh > -25) v = (m + ((int64_t)1 << (-sh - 1))) >> (-sh);
    else v = 0;
    return (bits >> 31) ? -v : v;
}

// Unary term of label x of item (v, c): the fixed-point unary, or the
// per-chain potential of Higdon's sweep.
template <int L>
__device__ __forceinline__ int64_t sw_unary(const SwArgs& a, int32_t v, int32_t c, int x) {
    return a.pot ? fix_from_float(a.pot[((int64_t)v * L + x) * a.C + c]) : __ldg(a.ufix + (int64_t)v * L + x);
}

// float of a fixed-point weight difference d <= 0 (two 32-bit conversions:
// GB300's 64-bit conversions run on its slow FP64 path).
__device__ __forceinline__ float sw_float(int64_t d) {
    return (float)(int32_t)(d >> 32) + (float)(uint32_t)d * (1.0f / 4294967296.0f);
}

// State between sweeps: parent[v][c] = v, ban[v][c] = 0, lw = 0 (the kernels
// below restore it); this kernel sets parent and ban, the host zeroes lw.
__global__ void __launch_bounds__(256) k_sw_reset(SwArgs a) {
    const int64_t n = (int64_t)a.N * a.C;
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < n; g += (int64_t)gridDim.x * blockDim.x) {
        a.parent[g] = (int32_t)a.fdC.div((uint32_t)g);
        a.ban[g] = 0u;
    }
}

// Per-warp queue of items in shared memory.  push() appends the lanes' flagged
// items; drain() hands them out 32 at a time to `fn(item, on)`, called by whole
// warps (lanes beyond the last item with on = false), until fewer than `keep`
// are left.
struct WarpQueue {
    uint32_t* q;
    int n;
    __device__ __forceinline__ void push(uint32_t item, bool flag) {
        const uint32_t bal = __ballot_sync(0xffffffffu, flag);
        if (flag) q[n + __popc(bal & ((1u << (threadIdx.x & 31)) - 1u))] = item;
        n += __popc(bal);
    }
    template <typename Fn>
    __device__ __forceinline__ void drain(int keep, Fn fn) {
        __syncwarp();
        while (n >= keep && n > 0) {
            const int lane = threadIdx.x & 31, take = n < 32 ? n : 32;
            n -= take;
            fn(lane < take ? q[n + lane] : 0u, lane < take);
            __syncwarp();
        }
    }
};

constexpr int kSwWarps = 8;                               // 256 threads

// Bond draws, items g = e C + c, V chains of one edge per lane (V = 4 when the
// chains are a multiple of 4).  Pairs of equal labels are queued, their draws
// (one Philox call each) decided 32 at a time, and the bonds queued again and
// united 32 at a time: each links its endpoints' trees, adds its label weights
// to its source site's row unless they are equal for every label (then they
// would shift all of a cluster's exact sums alike and leave its draw
// unchanged: Potts tables with one coupling per edge, every two-label table),
// and marks both endpoints bonded.  With Higdon's remainder (a.theta) a bond
// has no bits: its dual word, drawn before, is cleared.
template <int L, int V>
__global__ void __launch_bounds__(256) k_sw_bond(SwArgs a, int run) {
    __shared__ uint32_t s_q[kSwWarps][2][32 * V + 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t n = (uint32_t)(a.E * a.C);              // below 2^32 (host)
    const uint32_t t = (uint32_t)a.ctl->sweep, C = (uint32_t)a.C;
    const uint8_t* __restrict__ xin = a.x + (size_t)(t & 1) * a.N * a.C;
    WarpQueue same{s_q[warp][0], 0}, bonds{s_q[warp][1], 0};
    auto unite = [&](uint32_t g, bool on) {
        if (!on) return;
        const uint32_t e = a.fdC.div(g);
        const int32_t c = (int32_t)(g - e * C);
        const int32_t s = a.src[e], d = a.dst[e];
        if (a.theta) a.theta[g] = 0u;
        if (!sw_union(a.parent, s, d, c, a.C, a.N)) { atomicOr(a.err, 1u); return; }
        // every load before the first atomic (the compiler cannot move a
        // load above an atomic to a possibly aliasing address)
        int64_t wv[L];
#pragma unroll
        for (int x = 0; x < L; ++x) wv[x] = __ldg(a.lwe + (int64_t)e * L + x);
        bool uniform = wv[0] != kSwNoLabel;
#pragma unroll
        for (int x = 1; x < L; ++x) uniform &= wv[x] == wv[0];
        uint32_t flags = kSwBonded;
        if (!uniform) {
            flags |= kSwRow;
#pragma unroll
            for (int x = 0; x < L; ++x) {
                if (wv[x] == kSwNoLabel) flags |= 1u << x;
                else red_add_s64(a.lw + pidx(s, c, a.C) * L + x, wv[x]);
            }
        }
        atomicOr(a.ban + pidx(s, c, a.C), flags);
        atomicOr(a.ban + pidx(d, c, a.C), kSwBonded);
    };
    auto decide = [&](uint32_t g, bool on) {
        bool bond = false;
        if (on) {
            const uint32_t e = a.fdC.div(g), c = g - e * C;
            const uint32_t T = a.thr[(int64_t)e * L + xin[pidx(a.src[e], (int32_t)c, a.C)]];
            bond = T != 0u && (draw_rk(e, t, c, PH_BOND, 0, a.rk).x >> 9) < T;
        }
        bonds.push(g, bond);
        bonds.drain(32, unite);
    };
    const uint64_t first = ((uint64_t)blockIdx.x * kSwWarps + warp) * (32 * V * run);
    for (int k = 0; k < run; ++k) {
        const uint64_t g64 = first + (uint64_t)k * 32 * V + lane * V;
        uint32_t agree = 0;                                // bit j: item g + j has equal labels
        if (g64 < n) {
            const uint32_t e = a.fdC.div((uint32_t)g64);
            const int32_t c = (int32_t)((uint32_t)g64 - e * C), s = a.src[e];
            if (s >= 0) {
                const uint8_t* ps = xin + pidx(s, c, a.C);
                const uint8_t* pd = xin + pidx(a.dst[e], c, a.C);
                if constexpr (V == 4) {
                    const uint32_t eq = __vcmpeq4(*reinterpret_cast<const uint32_t*>(ps), *reinterpret_cast<const uint32_t*>(pd));
                    agree = (eq & 1u) | (eq >> 7 & 2u) | (eq >> 14 & 4u) | (eq >> 21 & 8u);
                } else {
                    agree = *ps == *pd;
                }
            }
        }
#pragma unroll
        for (int j = 0; j < V; ++j) same.push((uint32_t)g64 + j, (agree >> j) & 1u);
        same.drain(32, decide);
    }
    same.drain(1, decide);
    bonds.drain(1, unite);
}

// Scan of the ban words of the items that a warp owns, V of one site per lane:
// fn(g, words) for every lane and tile (items beyond the last: words 0).
template <int V, typename Fn>
__device__ __forceinline__ void sw_scan(const SwArgs& a, int run, Fn fn) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint64_t n = (uint64_t)a.N * a.C, first = ((uint64_t)blockIdx.x * kSwWarps + warp) * (32 * V * run);
    for (int k = 0; k < run; ++k) {
        const uint64_t g = first + (uint64_t)k * 32 * V + lane * V;
        uint32_t b[V];
#pragma unroll
        for (int j = 0; j < V; ++j) b[j] = 0u;
        if (g < n) {
            if constexpr (V == 4) {
                const uint4 q = *reinterpret_cast<const uint4*>(a.ban + g);
                b[0] = q.x; b[1] = q.y; b[2] = q.z; b[3] = q.w;
            } else {
                b[0] = a.ban[g];
            }
        }
        fn((uint32_t)g, g < n, b);
    }
}

// Bonded sites only (a site without a bond is its own cluster).  The forest
// is final once k_sw_bond has finished: every bonded site records its root
// (the smallest site of its cluster), and a non-root adds its unaries and the
// weights of the bonds it is the source of into its root's row.  Only roots'
// rows and ban words are written here, and only non-roots' are read.  The
// walks run one item per lane; the additions with the labels of an item on
// consecutive lanes, so that a row's loads and reductions are whole sectors.
template <int L, int V>
__global__ void __launch_bounds__(256) k_sw_flatten(SwArgs a, int run) {
    __shared__ uint32_t s_q[kSwWarps][32 * V + 32];
    const int lane = threadIdx.x & 31;
    const uint32_t C = (uint32_t)a.C;
    WarpQueue bonded{s_q[threadIdx.x >> 5], 0};
    auto flatten = [&](uint32_t g, bool on) {
        uint32_t b = 0u;
        int32_t v = 0, r = 0;
        if (on) {
            b = a.ban[g];
            v = (int32_t)a.fdC.div(g);
            r = sw_find(a.parent, v, (int32_t)(g - (uint32_t)v * C), a.C, a.N);
            if (r < 0) { atomicOr(a.err, 1u); on = false; }
            else a.root[g] = r;
        }
        on = on && r != v;
        const int32_t c = (int32_t)(g - (uint32_t)v * C);
        if (on && (b & kSwLabelMask)) atomicOr(a.ban + pidx(r, c, a.C), b & kSwLabelMask);
        if (a.pot) {                                       // per-chain unaries: consecutive chains on consecutive lanes
            if (!on) return;
            int64_t w[L];
#pragma unroll
            for (int x = 0; x < L; ++x) w[x] = sw_unary<L>(a, v, c, x);
            if (b & kSwRow) {
#pragma unroll
                for (int x = 0; x < L; ++x) w[x] += a.lw[(int64_t)g * L + x];
            }
#pragma unroll
            for (int x = 0; x < L; ++x) red_add_s64(a.lw + pidx(r, c, a.C) * L + x, w[x]);
            return;
        }
        const uint32_t act = __ballot_sync(0xffffffffu, on), rows = __ballot_sync(0xffffffffu, on && (b & kSwRow));
        const uint32_t gr = (uint32_t)pidx(r, c, a.C);     // the root's item, below 2^32
#pragma unroll
        for (int k = 0; k < L; ++k) {
            const int idx = k * 32 + lane, it = idx / L, x = idx - it * L;
            const int32_t vi = __shfl_sync(0xffffffffu, v, it);
            const uint32_t ri = __shfl_sync(0xffffffffu, gr, it), gi = __shfl_sync(0xffffffffu, g, it);
            if (!((act >> it) & 1u)) continue;
            int64_t w = __ldg(a.ufix + (int64_t)vi * L + x);
            if ((rows >> it) & 1u) w += a.lw[(int64_t)gi * L + x];
            red_add_s64(a.lw + (int64_t)ri * L + x, w);
        }
    };
    sw_scan<V>(a, run, [&](uint32_t g, bool, const uint32_t (&b)[V]) {
#pragma unroll
        for (int j = 0; j < V; ++j) bonded.push(g + j, (b[j] & kSwBonded) != 0u);
        bonded.drain(32, flatten);
    });
    bonded.drain(1, flatten);
}

// Float32 CDF of a site on its own (its unaries only), for the draw of
// unbonded sites: the same for every chain, so built once per factor change.
template <int L>
__global__ void k_sw_cdf(const int64_t* __restrict__ ufix, int N, float* __restrict__ cdf) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= N) return;
    int64_t w[L], mx = INT64_MIN;
#pragma unroll
    for (int x = 0; x < L; ++x) { w[x] = ufix[(int64_t)v * L + x]; mx = w[x] > mx ? w[x] : mx; }
    float s = 0.0f, c[L];
#pragma unroll
    for (int x = 0; x < L; ++x) { s += expf(sw_float(w[x] - mx)); c[x] = s; }
#pragma unroll
    for (int x = 0; x < L; ++x) cdf[(int64_t)v * L + x] = c[x] / s;
}

// Label of every cluster, drawn at its root r by the inverse CDF with the
// uniform of Philox(r, t, c, CLUSTER): weights are the root's unaries plus its
// row (bonded sites), the differences to the largest are exact in fixed point
// and then rounded to float for the softmax.  An unbonded site has the same
// weights in every chain: its draw compares u with the site's CDF (k_sw_cdf,
// within 3e-6 of the exact one, as draw_label's own), and only where a boundary
// is within 2^-16 is the draw computed in full.  Nothing but the label is
// written here: a store right behind the loads of the same row stalled the
// kernel several-fold, so k_sw_assign clears rows and ban words.
template <int L, int V>
__global__ void __launch_bounds__(256) k_sw_draw(SwArgs a, int run) {
    __shared__ uint32_t s_q[kSwWarps][32 * V + 32];
    const uint32_t t = (uint32_t)a.ctl->sweep, C = (uint32_t)a.C;
    uint8_t* __restrict__ xout = a.x + (size_t)((t + 1) & 1) * a.N * a.C;
    WarpQueue queue{s_q[threadIdx.x >> 5], 0};
    auto full = [&](uint32_t g, bool on) {
        if (!on) return;
        const int32_t v = (int32_t)a.fdC.div(g), c = (int32_t)(g - (uint32_t)v * C);
        const uint32_t b = a.ban[g];
        const bool bonded = (b & kSwBonded) != 0u;
        if (bonded && a.root[g] != v) {                    // labelled by k_sw_assign
            if (a.lpv) a.lpv[g] = 0.0f;
            return;
        }
        int64_t w[L];
#pragma unroll
        for (int x = 0; x < L; ++x) w[x] = sw_unary<L>(a, v, c, x);
        if (bonded) {
            const int64_t* row = a.lw + (int64_t)g * L;
            if constexpr (L % 2 == 0) {
#pragma unroll
                for (int x = 0; x < L; x += 2) {
                    const longlong2 q = *reinterpret_cast<const longlong2*>(row + x);
                    w[x] += q.x;
                    w[x + 1] += q.y;
                }
            } else {
#pragma unroll
                for (int x = 0; x < L; ++x) w[x] += row[x];
            }
        }
        int64_t mx = 0;
        bool any = false;
#pragma unroll
        for (int x = 0; x < L; ++x)
            if (!((b >> x) & 1u) && (!any || w[x] > mx)) { mx = w[x]; any = true; }
        float F[L];
#pragma unroll
        for (int x = 0; x < L; ++x)
            F[x] = ((b >> x) & 1u) ? -INFINITY : sw_float(w[x] - mx);
        xout[g] = (uint8_t)draw_label<L>(F, (uint32_t)v, (uint32_t)c, t, a.rk, PH_CLUSTER, nullptr, a.ctl,
                                         a.lpv ? a.lpv + g : nullptr);
    };
    const bool table = !a.pot && !a.lpv, fields = a.pot && !a.lpv;
    sw_scan<V>(a, run, [&](uint32_t g, bool in, const uint32_t (&b)[V]) {
        uint32_t rest = in ? (1u << V) - 1u : 0u;          // items that take the full draw
        uint32_t labels = 0;
        if (in && fields) {                                // Higdon: every chain has its own potentials
            const uint32_t v = a.fdC.div(g), c = g - v * C;
#pragma unroll 1
            for (int j = 0; j < V; ++j) {
                if (b[j] & kSwBonded) continue;
                float F[L];
#pragma unroll
                for (int x = 0; x < L; ++x) F[x] = a.pot[((int64_t)v * L + x) * a.C + c + j];
                const int lab = draw_label_fast<L>(F, uniform23(draw_rk(v, t, c + j, PH_CLUSTER, 0, a.rk).x));
                if (lab >= 0) { labels |= (uint32_t)lab << (8 * j); rest &= ~(1u << j); }
            }
        }
        if (in && table) {
            const uint32_t v = a.fdC.div(g), c = g - v * C;
            float cdf[L];
            if constexpr (L % 4 == 0) {
#pragma unroll
                for (int x = 0; x < L; x += 4) {
                    const float4 q = __ldg(reinterpret_cast<const float4*>(a.cdf + (int64_t)v * L + x));
                    cdf[x] = q.x; cdf[x + 1] = q.y; cdf[x + 2] = q.z; cdf[x + 3] = q.w;
                }
            } else {
#pragma unroll
                for (int x = 0; x < L; ++x) cdf[x] = __ldg(a.cdf + (int64_t)v * L + x);
            }
#pragma unroll
            for (int j = 0; j < V; ++j) {
                const float u = uniform23(draw_rk(v, t, c + j, PH_CLUSTER, 0, a.rk).x);
                float closest = INFINITY;
                int lab = 0;
#pragma unroll
                for (int x = 0; x < L; ++x) {
                    const float d = cdf[x] - u;
                    closest = fminf(closest, fabsf(d));
                    lab += d <= 0.0f ? 1 : 0;
                }
                if (!(b[j] & kSwBonded) && closest >= 0x1p-16f) rest &= ~(1u << j);
                labels |= (uint32_t)lab << (8 * j);
            }
        }
        if (in) {
            if (V == 4 && rest == 0u) {
                *reinterpret_cast<uint32_t*>(xout + g) = labels;
            } else {
#pragma unroll
                for (int j = 0; j < V; ++j)
                    if (!((rest >> j) & 1u)) xout[g + j] = (uint8_t)(labels >> (8 * j));
            }
        }
#pragma unroll
        for (int j = 0; j < V; ++j) queue.push(g + j, (rest >> j) & 1u);
        queue.drain(32, full);
    });
    queue.drain(1, full);
}

// Bonded sites return to the between-sweeps state: non-roots copy their
// root's label; a root's row (its cluster's sums) and a bond source's row are
// cleared (labels on consecutive lanes: whole sectors); parent and ban words
// are reset.
template <int L, int V>
__global__ void __launch_bounds__(256) k_sw_assign(SwArgs a, int run) {
    __shared__ uint32_t s_q[kSwWarps][32 * V + 32];
    const int lane = threadIdx.x & 31;
    const uint32_t t = (uint32_t)a.ctl->sweep, C = (uint32_t)a.C;
    uint8_t* __restrict__ xout = a.x + (size_t)((t + 1) & 1) * a.N * a.C;
    WarpQueue bonded{s_q[threadIdx.x >> 5], 0};
    auto assign = [&](uint32_t g, bool on) {
        bool clear = false;
        if (on) {
            const uint32_t b = a.ban[g];
            const int32_t v = (int32_t)a.fdC.div(g), c = (int32_t)(g - (uint32_t)v * C), r = a.root[g];
            if (r != v) xout[g] = xout[pidx(r, c, a.C)];
            clear = r == v || (b & kSwRow);
            a.parent[g] = v;
            a.ban[g] = 0u;
        }
        const uint32_t rows = __ballot_sync(0xffffffffu, clear);
#pragma unroll
        for (int k = 0; k < L; ++k) {
            const int idx = k * 32 + lane, it = idx / L;
            const uint32_t gi = __shfl_sync(0xffffffffu, g, it);
            if ((rows >> it) & 1u) a.lw[(int64_t)gi * L + (idx - it * L)] = 0;
        }
    };
    sw_scan<V>(a, run, [&](uint32_t g, bool, const uint32_t (&b)[V]) {
#pragma unroll
        for (int j = 0; j < V; ++j) bonded.push(g + j, (b[j] & kSwBonded) != 0u);
        bonded.drain(32, assign);
    });
    bonded.drain(1, assign);
}

// Small models: n_sweeps whole Swendsen-Wang sweeps in one launch of a single
// 1024-thread CTA (launch latency dominates there), the union-find state in
// shared memory: parent, root and ban words [N][C], weight rows [N][L][C].
// The same draws, exact sums and rules as the kernels above, phases separated
// by CTA barriers, hence the same chain bit for bit; marginal counts and the
// sweep counter are advanced here too.
__device__ __forceinline__ int32_t sws_find(volatile int32_t* par, int32_t v, int32_t c, int32_t C, int32_t N) {
    for (int32_t step = 0; step <= N; ++step) {
        const int32_t p = par[pidx(v, c, C)];
        if (p == v) return v;
        const int32_t gp = par[pidx(p, c, C)];
        if (gp != p) par[pidx(v, c, C)] = gp;
        v = gp;
    }
    return -1;
}

template <int L>
__global__ void __launch_bounds__(1024) k_sw_small(SwArgs a, int n_sweeps) {
    extern __shared__ int64_t s_lw[];                                  // [N][L][C]
    const int64_t nv = (int64_t)a.N * a.C, ne = a.E * a.C;
    int32_t* s_par = reinterpret_cast<int32_t*>(s_lw + nv * L);       // [N][C]
    int32_t* s_root = s_par + nv;                                     // [N][C]
    uint32_t* s_ban = reinterpret_cast<uint32_t*>(s_root + nv);       // [N][C]
    volatile int32_t* vpar = s_par;
    for (int64_t g = threadIdx.x; g < nv; g += blockDim.x) {
        s_par[g] = (int32_t)a.fdC.div((uint32_t)g);
        s_ban[g] = 0u;
    }
    for (int64_t i = threadIdx.x; i < nv * L; i += blockDim.x) s_lw[i] = 0;
    __syncthreads();
    uint32_t sweep = (uint32_t)a.ctl->sweep;
    const unsigned long long count_from = a.ctl->count_from;
    for (int it = 0; it < n_sweeps; ++it, ++sweep) {
        const uint8_t* xin = a.x + (size_t)(sweep & 1) * a.N * a.C;
        uint8_t* xout = a.x + (size_t)((sweep + 1) & 1) * a.N * a.C;
        // bonds and unions
        for (int64_t g = threadIdx.x; g < ne; g += blockDim.x) {
            const int64_t e = a.fdC.div((uint32_t)g);
            const int32_t c = (int32_t)(g - e * a.C);
            const int32_t s = a.src[e];
            if (s < 0) continue;
            const int32_t d = a.dst[e];
            const int xs = xin[pidx(s, c, a.C)];
            if (xs != xin[pidx(d, c, a.C)]) continue;
            const uint32_t T = a.thr[e * L + xs];
            if (T == 0u || (draw_rk((uint32_t)e, sweep, (uint32_t)c, PH_BOND, 0, a.rk).x >> 9) >= T) continue;
            int32_t ra = s, rb = d;
            bool linked = false;
            for (int32_t step = 0; step <= a.N && !linked; ++step) {
                ra = sws_find(vpar, ra, c, a.C, a.N);
                rb = sws_find(vpar, rb, c, a.C, a.N);
                if (ra < 0 || rb < 0) break;
                if (ra == rb) { linked = true; break; }
                if (ra < rb) { const int32_t t2 = ra; ra = rb; rb = t2; }
                linked = atomicCAS(s_par + pidx(ra, c, a.C), ra, rb) == ra;
            }
            if (!linked) { atomicOr(a.err, 1u); continue; }
            int64_t wv[L];
#pragma unroll
            for (int x = 0; x < L; ++x) wv[x] = __ldg(a.lwe + e * L + x);
            bool uniform = wv[0] != kSwNoLabel;
#pragma unroll
            for (int x = 1; x < L; ++x) uniform &= wv[x] == wv[0];
            uint32_t flags = kSwBonded;
            if (!uniform) {
                flags |= kSwRow;
#pragma unroll
                for (int x = 0; x < L; ++x) {
                    if (wv[x] == kSwNoLabel) flags |= 1u << x;
                    else atomicAdd(reinterpret_cast<unsigned long long*>(s_lw + ((int64_t)s * L + x) * a.C + c),
                                   (unsigned long long)wv[x]);
                }
            }
            atomicOr(s_ban + pidx(s, c, a.C), flags);
            atomicOr(s_ban + pidx(d, c, a.C), kSwBonded);
        }
        __syncthreads();
        // roots and cluster sums
        for (int64_t g = threadIdx.x; g < nv; g += blockDim.x) {
            const uint32_t b = s_ban[g];
            if (!(b & kSwBonded)) continue;
            const int32_t v = (int32_t)a.fdC.div((uint32_t)g), c = (int32_t)(g - (int64_t)v * a.C);
            const int32_t r = sws_find(vpar, v, c, a.C, a.N);
            if (r < 0) { atomicOr(a.err, 1u); s_root[g] = v; continue; }
            s_root[g] = r;
            if (r == v) continue;
#pragma unroll
            for (int x = 0; x < L; ++x) {
                int64_t w = __ldg(a.ufix + (int64_t)v * L + x);
                if (b & kSwRow) w += s_lw[((int64_t)v * L + x) * a.C + c];
                atomicAdd(reinterpret_cast<unsigned long long*>(s_lw + ((int64_t)r * L + x) * a.C + c),
                          (unsigned long long)w);
            }
            if (b & kSwLabelMask) atomicOr(s_ban + pidx(r, c, a.C), b & kSwLabelMask);
        }
        __syncthreads();
        // labels of the roots
        for (int64_t g = threadIdx.x; g < nv; g += blockDim.x) {
            const int32_t v = (int32_t)a.fdC.div((uint32_t)g), c = (int32_t)(g - (int64_t)v * a.C);
            const uint32_t b = s_ban[g];
            const bool bonded = (b & kSwBonded) != 0u;
            if (bonded && s_root[g] != v) continue;
            int64_t w[L];
#pragma unroll
            for (int x = 0; x < L; ++x) {
                w[x] = __ldg(a.ufix + (int64_t)v * L + x);
                if (bonded) w[x] += s_lw[((int64_t)v * L + x) * a.C + c];
            }
            int64_t mx = 0;
            bool any = false;
#pragma unroll
            for (int x = 0; x < L; ++x)
                if (!((b >> x) & 1u) && (!any || w[x] > mx)) { mx = w[x]; any = true; }
            float F[L];
#pragma unroll
            for (int x = 0; x < L; ++x) F[x] = ((b >> x) & 1u) ? -INFINITY : sw_float(w[x] - mx);
            xout[g] = (uint8_t)draw_label<L>(F, (uint32_t)v, (uint32_t)c, sweep, a.rk, PH_CLUSTER, nullptr, a.ctl);
        }
        __syncthreads();
        // labels of the other sites, state reset
        for (int64_t g = threadIdx.x; g < nv; g += blockDim.x) {
            const uint32_t b = s_ban[g];
            if (!(b & kSwBonded)) continue;
            const int32_t v = (int32_t)a.fdC.div((uint32_t)g), c = (int32_t)(g - (int64_t)v * a.C);
            const int32_t r = s_root[g];
            if (r != v) xout[g] = xout[pidx(r, c, a.C)];
            if (r == v || (b & kSwRow)) {
#pragma unroll
                for (int x = 0; x < L; ++x) s_lw[((int64_t)v * L + x) * a.C + c] = 0;
            }
            s_par[g] = v;
            s_ban[g] = 0u;
        }
        __syncthreads();
        if (sweep >= count_from) {
            for (int64_t v = threadIdx.x; v < a.N; v += blockDim.x) {
                uint32_t tot[L];
#pragma unroll
                for (int x = 0; x < L; ++x) tot[x] = 0;
                for (int c = 0; c < a.C; ++c) {
                    const int x = xout[v * a.C + c];
#pragma unroll
                    for (int y = 0; y < L; ++y) tot[y] += x == y ? 1u : 0u;
                }
#pragma unroll
                for (int x = 0; x < L; ++x) a.counts[v * L + x] += tot[x];
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) a.ctl->sweep = sweep;
}

// Higdon's partial Swendsen-Wang (Section 4.3): per edge and label a with
// coupling l (float64), alpha = rho (e^l - 1) and the remainder
// A = exp(l' [a = b]), l' = log(1 + (1 - rho)(e^l - 1)), dualised by
// entry_dual (diagonal layout, entry k = label k).  Written per edge: the bond
// threshold of rho (1 - e^{-l}), the bond weight log alpha - alpha1 - alpha2
// in fixed point, A's dual weights, thresholds and unary terms, and the
// edge's bound for the range check.
__global__ void k_hg_tables(const int32_t* __restrict__ src, const double* __restrict__ ell, int64_t E, int L,
                            double rho, HigdonTables t) {
    const int MP = pad4(L);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < E; e += (int64_t)gridDim.x * blockDim.x) {
        double bound_w = 0.0, bound_tau = 0.0;
        for (int x = 0; x < L; ++x) {
            const double l = src[e] >= 0 ? ell[e * L + x] : 0.0;
            const double alpha = rho * expm1(l);
            const double lp = log1p((1.0 - rho) * expm1(l));
            uint32_t T = 0;
            if (l > 0.0 && rho > 0.0) T = (uint32_t)ceil(rho * -expm1(-l) * 8388608.0 - 0.5);
            float tau_s = 0.0f;
            uint32_t word = 0;
            double a12 = 0.0;
            if (lp != 0.0) {
                const EntryDual d = entry_dual(lp);
                tau_s = d.tau_s; word = d.word; a12 = d.alpha1 + d.alpha2;
                t.fold[(e * 2 + 0) * L + x] = d.alpha1;
                t.fold[(e * 2 + 1) * L + x] = d.alpha2;
            } else {
                t.fold[(e * 2 + 0) * L + x] = 0.0;
                t.fold[(e * 2 + 1) * L + x] = 0.0;
            }
            int64_t lw = kSwNoLabel;
            if (alpha > 0.0) {
                const double w = log(alpha) - a12;
                lw = sw_fix(w);
                bound_w = fmax(bound_w, fabs(w));
            }
            bound_tau = fmax(bound_tau, fabs((double)tau_s));
            t.bond_thr[e * L + x] = T;
            t.bond_lw[e * L + x] = lw;
            t.tau[e * MP + x] = tau_s;
            t.thr[e * L + x] = word;
        }
        for (int x = L; x < MP; ++x) t.tau[e * MP + x] = 0.0f;
        t.bound[e] = src[e] >= 0 ? bound_w + 2.0 * bound_tau : 0.0;
    }
}

// out[0] += sum over sites of max_x |ut_v(x)| + sum over live edges of their bound.
__global__ void k_hg_check(const double* __restrict__ ut, int N, int L, const int32_t* __restrict__ src,
                           const double* __restrict__ bound, int64_t E, double* out) {
    double acc = 0.0;
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < N; v += (int64_t)gridDim.x * blockDim.x) {
        double m = 0.0;
        for (int x = 0; x < L; ++x) m = fmax(m, fabs(ut[v * L + x]));
        acc += m;
    }
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < E; e += (int64_t)gridDim.x * blockDim.x)
        if (src[e] >= 0) acc += bound[e];
    if (acc != 0.0) atomicAdd(out, acc);
}

// Small models, Higdon's sweep: n_sweeps whole sweeps in one single-CTA
// launch, the remainder's dual bits, the union-find state and the cluster
// rows in shared memory.  The bonds, bits (the dual contract of k_dual,
// decided by dual_bits), potentials (summed in the incidence order of the
// primal kernels, flushed every 32 incidences) and exact cluster sums are
// those of the launch-per-step path, hence the same chain bit for bit.
template <int L>
__global__ void __launch_bounds__(1024) k_hg_small(SweepArgs d, SwArgs a, int n_sweeps) {
    using En = Ent<L, MRF_LAYOUT_DIAG>;
    extern __shared__ int64_t s_lw[];                                  // [N][L][C]
    const int64_t nv = (int64_t)a.N * a.C, ne = a.E * a.C;
    int32_t* s_par = reinterpret_cast<int32_t*>(s_lw + nv * L);       // [N][C]
    int32_t* s_root = s_par + nv;                                     // [N][C]
    uint32_t* s_ban = reinterpret_cast<uint32_t*>(s_root + nv);       // [N][C]
    uint32_t* s_theta = s_ban + nv;                                   // [E][C] remainder's bits
    volatile int32_t* vpar = s_par;
    for (int64_t g = threadIdx.x; g < nv; g += blockDim.x) {
        s_par[g] = (int32_t)a.fdC.div((uint32_t)g);
        s_ban[g] = 0u;
    }
    for (int64_t i = threadIdx.x; i < nv * L; i += blockDim.x) s_lw[i] = 0;
    __syncthreads();
    uint32_t sweep = (uint32_t)a.ctl->sweep;
    const unsigned long long count_from = a.ctl->count_from;
    for (int it = 0; it < n_sweeps; ++it, ++sweep) {
        const uint8_t* xin = a.x + (size_t)(sweep & 1) * a.N * a.C;
        uint8_t* xout = a.x + (size_t)((sweep + 1) & 1) * a.N * a.C;
        // bonds (with their unions) or the remainder's bits, per (edge, chain)
        for (int64_t g = threadIdx.x; g < ne; g += blockDim.x) {
            const int64_t e = a.fdC.div((uint32_t)g);
            const int32_t c = (int32_t)(g - e * a.C);
            const int32_t s = a.src[e];
            s_theta[g] = 0u;
            if (s < 0) continue;
            const int32_t t = a.dst[e];
            const int xs = xin[pidx(s, c, a.C)], xt = xin[pidx(t, c, a.C)];
            bool bond = false;
            if (xs == xt) {
                const uint32_t T = a.thr[e * L + xs];
                bond = T != 0u && (draw_rk((uint32_t)e, sweep, (uint32_t)c, PH_BOND, 0, a.rk).x >> 9) < T;
            }
            if (!bond) {
                uint32_t bits[En::W];
                dual_bits<L, MRF_LAYOUT_DIAG>((uint32_t)e, (uint32_t)c, xs, xt, d.tpl + e * En::PW, d.thr + e * En::M,
                                              sweep, d.rk, bits);
                s_theta[g] = bits[0];
                continue;
            }
            int32_t ra = s, rb = t;
            bool linked = false;
            for (int32_t step = 0; step <= a.N && !linked; ++step) {
                ra = sws_find(vpar, ra, c, a.C, a.N);
                rb = sws_find(vpar, rb, c, a.C, a.N);
                if (ra < 0 || rb < 0) break;
                if (ra == rb) { linked = true; break; }
                if (ra < rb) { const int32_t t2 = ra; ra = rb; rb = t2; }
                linked = atomicCAS(s_par + pidx(ra, c, a.C), ra, rb) == ra;
            }
            if (!linked) { atomicOr(a.err, 1u); continue; }
            int64_t wv[L];
#pragma unroll
            for (int x = 0; x < L; ++x) wv[x] = __ldg(a.lwe + e * L + x);
            bool uniform = wv[0] != kSwNoLabel;
#pragma unroll
            for (int x = 1; x < L; ++x) uniform &= wv[x] == wv[0];
            uint32_t flags = kSwBonded;
            if (!uniform) {
                flags |= kSwRow;
#pragma unroll
                for (int x = 0; x < L; ++x) {
                    if (wv[x] == kSwNoLabel) flags |= 1u << x;
                    else atomicAdd(reinterpret_cast<unsigned long long*>(s_lw + ((int64_t)s * L + x) * a.C + c),
                                   (unsigned long long)wv[x]);
                }
            }
            atomicOr(s_ban + pidx(s, c, a.C), flags);
            atomicOr(s_ban + pidx(t, c, a.C), kSwBonded);
        }
        __syncthreads();
        // potentials of every site, moved into the rows of the cluster roots
        for (int64_t g = threadIdx.x; g < nv; g += blockDim.x) {
            const int32_t v = (int32_t)a.fdC.div((uint32_t)g), c = (int32_t)(g - (int64_t)v * a.C);
            float acc[L], hi[L], lo[L];
#pragma unroll
            for (int x = 0; x < L; ++x) { acc[x] = 0.0f; hi[x] = 0.0f; lo[x] = 0.0f; }
            int chunk = 0;
            bool flushed = false;
            for (int64_t p = d.inc_ptr[v]; p < d.inc_ptr[v + 1]; ++p) {
                const int2 ic = __ldg(&d.inc[p]);
                const int64_t e = ic.x >> 1;
                const uint32_t bits[En::W] = {s_theta[e * a.C + c]};
                add_side<L, MRF_LAYOUT_DIAG>(bits, d.tau + e * En::MP, ic.x & 1, acc);
                if (++chunk == 32) {
#pragma unroll
                    for (int x = 0; x < L; ++x) { two_sum_add(hi[x], lo[x], acc[x]); acc[x] = 0.0f; }
                    chunk = 0;
                    flushed = true;
                }
            }
            int64_t w[L];
            const float* uf = d.utf + (int64_t)v * L;
#pragma unroll
            for (int x = 0; x < L; ++x) {
                float F;
                if (flushed) { two_sum_add(hi[x], lo[x], acc[x]); F = __ldg(uf + x) + (hi[x] + lo[x]); }
                else F = __ldg(uf + x) + acc[x];
                w[x] = fix_from_float(F);
            }
            const uint32_t b = s_ban[g];
            int32_t r = v;
            if (b & kSwBonded) {
                r = sws_find(vpar, v, c, a.C, a.N);
                if (r < 0) { atomicOr(a.err, 1u); r = v; }
                s_root[g] = r;
                if (r != v && (b & kSwRow)) {
#pragma unroll
                    for (int x = 0; x < L; ++x) w[x] += s_lw[((int64_t)v * L + x) * a.C + c];
                }
                if (r != v && (b & kSwLabelMask)) atomicOr(s_ban + pidx(r, c, a.C), b & kSwLabelMask);
            }
#pragma unroll
            for (int x = 0; x < L; ++x)
                atomicAdd(reinterpret_cast<unsigned long long*>(s_lw + ((int64_t)r * L + x) * a.C + c),
                          (unsigned long long)w[x]);
        }
        __syncthreads();
        // labels of the roots
        for (int64_t g = threadIdx.x; g < nv; g += blockDim.x) {
            const int32_t v = (int32_t)a.fdC.div((uint32_t)g), c = (int32_t)(g - (int64_t)v * a.C);
            const uint32_t b = s_ban[g];
            if ((b & kSwBonded) && s_root[g] != v) continue;
            int64_t w[L];
#pragma unroll
            for (int x = 0; x < L; ++x) w[x] = s_lw[((int64_t)v * L + x) * a.C + c];
            int64_t mx = 0;
            bool any = false;
#pragma unroll
            for (int x = 0; x < L; ++x)
                if (!((b >> x) & 1u) && (!any || w[x] > mx)) { mx = w[x]; any = true; }
            float F[L];
#pragma unroll
            for (int x = 0; x < L; ++x) F[x] = ((b >> x) & 1u) ? -INFINITY : sw_float(w[x] - mx);
            xout[g] = (uint8_t)draw_label<L>(F, (uint32_t)v, (uint32_t)c, sweep, a.rk, PH_CLUSTER, nullptr, a.ctl);
        }
        __syncthreads();
        // labels of the other sites, state reset (every root's row holds sums now)
        for (int64_t g = threadIdx.x; g < nv; g += blockDim.x) {
            const int32_t v = (int32_t)a.fdC.div((uint32_t)g), c = (int32_t)(g - (int64_t)v * a.C);
            const uint32_t b = s_ban[g];
            const int32_t r = (b & kSwBonded) ? s_root[g] : v;
            if (r != v) xout[g] = xout[pidx(r, c, a.C)];
            if (r == v || (b & kSwRow)) {
#pragma unroll
                for (int x = 0; x < L; ++x) s_lw[((int64_t)v * L + x) * a.C + c] = 0;
            }
            s_par[g] = v;
            s_ban[g] = 0u;
        }
        __syncthreads();
        if (sweep >= count_from) {
            for (int64_t v = threadIdx.x; v < a.N; v += blockDim.x) {
                uint32_t tot[L];
#pragma unroll
                for (int x = 0; x < L; ++x) tot[x] = 0;
                for (int c = 0; c < a.C; ++c) {
                    const int x = xout[v * a.C + c];
#pragma unroll
                    for (int y = 0; y < L; ++y) tot[y] += x == y ? 1u : 0u;
                }
#pragma unroll
                for (int x = 0; x < L; ++x) a.counts[v * L + x] += tot[x];
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) a.ctl->sweep = sweep;
}

// Model check before the first Swendsen-Wang sweep after the factors change:
// out[0] = dual weights tau < 0 on live edges (antiferromagnetic entries; with
// two labels the one pivot entry's tau has the sign of l),
// out[1] = sum over live edges of max_x |log(e^{l_x} - 1)| over bondable labels,
// out[2] = sum over sites of max_x |u_v(x)| (the unaries the sweep uses).
// out[1] + out[2] bounds the magnitude of every partial sum of a cluster weight.
__global__ void k_sw_check(const int32_t* src, const float* tau, int64_t E, int M, const int64_t* lwe, int L,
                           const float* unary, const double* unary_d, int N, double* out) {
    double neg = 0.0, se = 0.0, su = 0.0;
    const int MP = pad4(M);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < E; e += (int64_t)gridDim.x * blockDim.x) {
        if (src[e] < 0) continue;
        double m = 0.0;
        for (int k = 0; k < M; ++k) neg += tau[e * MP + k] < 0.0f;
        for (int x = 0; x < L; ++x) {
            const int64_t w = lwe[e * L + x];
            if (w != kSwNoLabel) m = fmax(m, fabs((double)w / kSwFixScale));
        }
        se += m;
    }
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < N; v += (int64_t)gridDim.x * blockDim.x) {
        double m = 0.0;
        for (int x = 0; x < L; ++x) m = fmax(m, fabs(unary_d ? unary_d[v * L + x] : (double)unary[v * L + x]));
        su += m;
    }
    if (neg != 0.0) atomicAdd(out + 0, neg);
    if (se != 0.0) atomicAdd(out + 1, se);
    if (su != 0.0) atomicAdd(out + 2, su);
}

#define MRF_DISPATCH_LSW(L_, ...)                                                 \
    switch (L_) {                                                                 \
        case 2: { constexpr int LL = 2; __VA_ARGS__; } break;                     \
        case 3: { constexpr int LL = 3; __VA_ARGS__; } break;                     \
        case 4: { constexpr int LL = 4; __VA_ARGS__; } break;                     \
        case 5: { constexpr int LL = 5; __VA_ARGS__; } break;                     \
        case 6: { constexpr int LL = 6; __VA_ARGS__; } break;                     \
        case 7: { constexpr int LL = 7; __VA_ARGS__; } break;                     \
        case 8: { constexpr int LL = 8; __VA_ARGS__; } break;                     \
        case 9: { constexpr int LL = 9; __VA_ARGS__; } break;                     \
        case 10: { constexpr int LL = 10; __VA_ARGS__; } break;                   \
        case 11: { constexpr int LL = 11; __VA_ARGS__; } break;                   \
        case 12: { constexpr int LL = 12; __VA_ARGS__; } break;                   \
        case 13: { constexpr int LL = 13; __VA_ARGS__; } break;                   \
        case 14: { constexpr int LL = 14; __VA_ARGS__; } break;                   \
        case 15: { constexpr int LL = 15; __VA_ARGS__; } break;                   \
        case 16: { constexpr int LL = 16; __VA_ARGS__; } break;                   \
        default: return cudaErrorInvalidValue;                                    \
    }

static inline unsigned sw_blocks(int64_t n) {
    // grid-stride loops over at most 8 resident blocks of 256 threads per SM
    const int64_t b = (n + 255) / 256;
    return (unsigned)(b < 152 * 8 ? (b > 0 ? b : 1) : 152 * 8);
}

cudaError_t launch_sw_check(const int32_t* src, const float* tau, int64_t E, int M, const int64_t* lwe, int L,
                            const float* unary, const double* unary_d, int N, double* out, cudaStream_t s) {
    k_sw_check<<<sw_blocks(E > N ? E : N), 256, 0, s>>>(src, tau, E, M, lwe, L, unary, unary_d, N, out);
    return cudaGetLastError();
}

// Fixed-point unaries ufix[v][x] = sw_fix(u_v(x)) (once per factor change).
__global__ void k_sw_fix_unary(const float* unary, const double* unary_d, int64_t n, int64_t* ufix) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        ufix[i] = sw_fix(unary_d ? unary_d[i] : (double)unary[i]);
}

cudaError_t launch_hg_tables(const int32_t* src, const double* ell, int64_t E, int L, double rho, HigdonTables t,
                             cudaStream_t s) {
    if (E > 0) k_hg_tables<<<sw_blocks(E), 256, 0, s>>>(src, ell, E, L, rho, t);
    return cudaGetLastError();
}

cudaError_t launch_hg_check(const double* ut, int N, int L, const int32_t* src, const double* bound, int64_t E,
                            double* out, cudaStream_t s) {
    k_hg_check<<<sw_blocks(E > N ? E : N), 256, 0, s>>>(ut, N, L, src, bound, E, out);
    return cudaGetLastError();
}

// Also the CDF of every site on its own (k_sw_cdf).
cudaError_t launch_sw_fix_unary(const float* unary, const double* unary_d, int N, int L, int64_t* ufix, float* cdf,
                                cudaStream_t s) {
    const int64_t n = (int64_t)N * L;
    if (n <= 0) return cudaSuccess;
    k_sw_fix_unary<<<sw_blocks(n), 256, 0, s>>>(unary, unary_d, n, ufix);
    MRF_DISPATCH_LSW(L, (k_sw_cdf<LL><<<(unsigned)((N + 127) / 128), 128, 0, s>>>(ufix, N, cdf)));
    return cudaGetLastError();
}

cudaError_t launch_sw_reset(const SwArgs& a, cudaStream_t s) {
    const int64_t n = (int64_t)a.N * a.C;
    if (n > 0) {
        k_sw_reset<<<sw_blocks(n), 256, 0, s>>>(a);
        const cudaError_t e = cudaMemsetAsync(a.lw, 0, (size_t)n * a.L * sizeof(int64_t), s);
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

// Launch shape of a kernel that scans n items: four chains per lane from two
// blocks per SM on (below, one per lane spreads the items over more SMs), and
// as many tiles per warp, up to eight, as leave eight blocks per SM.
struct SwScan {
    int V, run;
    unsigned blocks;
    SwScan(int64_t n, int C) {
        V = C % 4 == 0 && n >= 32 * 4 * kSwWarps * 152 * 2 ? 4 : 1;
        const int64_t tile = 32ll * V * kSwWarps;
        run = (int)std::min<int64_t>(8, std::max<int64_t>(1, n / (tile * 152 * 8)));
        blocks = (unsigned)((n + tile * run - 1) / (tile * run));
    }
};
#define MRF_SW_SCAN(kernel, n)                                                                          \
    do {                                                                                                \
        const SwScan sc(n, a.C);                                                                        \
        if (sc.V == 4) {                                                                                \
            MRF_DISPATCH_LSW(a.L, (kernel<LL, 4><<<sc.blocks, 32 * kSwWarps, 0, s>>>(a, sc.run)));      \
        } else {                                                                                        \
            MRF_DISPATCH_LSW(a.L, (kernel<LL, 1><<<sc.blocks, 32 * kSwWarps, 0, s>>>(a, sc.run)));      \
        }                                                                                               \
    } while (0)

cudaError_t launch_sw_bond(const SwArgs& a, cudaStream_t s) {
    const int64_t n = a.E * a.C;
    if (n <= 0) return cudaSuccess;
    MRF_SW_SCAN(k_sw_bond, n);
    return cudaGetLastError();
}

cudaError_t launch_sw_flatten(const SwArgs& a, cudaStream_t s) {
    const int64_t n = (int64_t)a.N * a.C;
    if (n <= 0) return cudaSuccess;
    MRF_SW_SCAN(k_sw_flatten, n);
    return cudaGetLastError();
}

int64_t sw_small_smem(const SwArgs& a) { return (int64_t)a.N * a.C * (12 + 8 * a.L); }

cudaError_t launch_sw_small(const SwArgs& a, int n_sweeps, cudaStream_t s) {
    if (!a.counts || !a.ufix || !a.err || !a.ctl || !a.x || (a.E > 0 && (!a.src || !a.dst || !a.thr || !a.lwe)))
        return cudaErrorInvalidValue;
    const size_t smem = (size_t)sw_small_smem(a);
    MRF_DISPATCH_LSW(a.L, ({
        if (smem > 48 * 1024) {
            const cudaError_t e = cudaFuncSetAttribute(k_sw_small<LL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
        k_sw_small<LL><<<1, 1024, smem, s>>>(a, n_sweeps);
    }));
    return cudaGetLastError();
}

int64_t hg_small_smem(const SwArgs& a) { return (int64_t)a.N * a.C * (12 + 8 * a.L) + a.E * a.C * 4; }

cudaError_t launch_hg_small(const SweepArgs& d, const SwArgs& a, int n_sweeps, cudaStream_t s) {
    if (!a.counts || !a.ufix || !a.err || !a.ctl || !a.x || !d.utf || !d.inc_ptr ||
        (a.E > 0 && (!a.src || !a.dst || !a.thr || !a.lwe || !d.tau || !d.thr || !d.tpl || !d.inc)))
        return cudaErrorInvalidValue;
    const size_t smem = (size_t)hg_small_smem(a);
    MRF_DISPATCH_LSW(a.L, ({
        if (smem > 48 * 1024) {
            const cudaError_t e = cudaFuncSetAttribute(k_hg_small<LL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
        k_hg_small<LL><<<1, 1024, smem, s>>>(d, a, n_sweeps);
    }));
    return cudaGetLastError();
}

cudaError_t launch_sw_draw(const SwArgs& a, cudaStream_t s) {
    const int64_t n = (int64_t)a.N * a.C;
    if (n <= 0) return cudaSuccess;
    MRF_SW_SCAN(k_sw_draw, n);
    MRF_SW_SCAN(k_sw_assign, n);
    return cudaGetLastError();
}

}  // namespace mrfk
