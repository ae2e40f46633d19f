// The two half-steps of the primal-dual sweep (Section 5.1) for sm_103a.
//
//   dual step    theta_ek ~ Bernoulli(sigmoid(q + beta1 [x_s = i_k] + beta2 [x_t = j_k]))
//                for every edge slot e, dualised entry k and chain c    (k_dual)
//   primal step  x_v ~ softmax_a F_v(a),
//                F_v(a) = u~_v(a) + sum over incident edges of the beta terms of
//                the set dual bits whose entry row (source side) or column
//                (destination side) is a                                 (k_primal)
//   fused form   both in one vertex-centric kernel: each endpoint regenerates
//                the dual bits of its incident edges from the counter-based
//                RNG (identical at both ends), so theta is never stored
//
// Labels are stored chain-innermost, x[buf][v][c], so that lanes of a warp
// working on consecutive chains of one site or edge read consecutive bytes and
// share the edge's table row (one broadcast load per word for the warp).
// The dual bits of one (edge, chain) are packed into W = ceil(m/32) words,
// theta[e][c][w].  The kernels read the sweep index from device memory (Ctl),
// so one sweep can be captured once as a CUDA graph and replayed.
#pragma once
#include "common.cuh"

#include <algorithm>

namespace mrfk {

// ---------------------------------------------------------------------------- entry masks

// Bits [lo, hi) of a 32-bit word (lo, hi relative to the word, clipped).
__device__ __forceinline__ uint32_t range_mask(int lo, int hi) {
    lo = max(lo, 0);
    hi = min(hi, 32);
    if (hi <= lo) return 0u;
    const uint32_t upto = hi == 32 ? 0xFFFFFFFFu : ((1u << hi) - 1u);
    return upto & ~((1u << lo) - 1u);
}

// Word g of the PIVOT column-1 pattern: entries k = r (L-1), r = 0..L-2.
__host__ __device__ constexpr uint32_t col_pattern_word(int L, int g) {
    uint32_t w = 0;
    for (int r = 0; r < L - 1; ++r) {
        const int k = r * (L - 1) - 32 * g;
        if (k >= 0 && k < 32) w |= 1u << k;
    }
    return w;
}

__host__ __device__ constexpr uint32_t valid_word(int M, int g) {
    return M - 32 * g >= 32 ? 0xFFFFFFFFu : (M - 32 * g <= 0 ? 0u : ((1u << (M - 32 * g)) - 1u));
}

// Entries of group g whose row is label a (y = 1) and whose column is b (z = 1).
template <int L, int LAYOUT>
__device__ __forceinline__ uint32_t row_mask(int a, int g) {
    if (LAYOUT == MRF_LAYOUT_DIAG) return (a >> 5) == g ? (1u << (a & 31)) : 0u;
    if (a == 0) return 0u;
    const int lo = (a - 1) * (L - 1) - 32 * g;
    return range_mask(lo, lo + L - 1);
}

template <int L, int LAYOUT>
__device__ __forceinline__ uint32_t col_mask(int b, int g) {
    if (LAYOUT == MRF_LAYOUT_DIAG) return (b >> 5) == g ? (1u << (b & 31)) : 0u;
    if (b == 0) return 0u;
    const uint32_t hi = col_pattern_word(L, g);
    const uint32_t lo = g > 0 ? col_pattern_word(L, g - 1) : 0u;
    return __funnelshift_l(lo, hi, (unsigned)(b - 1));
}

// ---------------------------------------------------------------------------- blocked sweep

// Offset (ox, oy, oz) of the block grid of the current blocked sweep.
__device__ __forceinline__ void splash_offset(const Ctl* ctl, int& ox, int& oy, int& oz) {
    const uint32_t o = (uint32_t)ctl->splash_offset;
    ox = o & 0xFF; oy = (o >> 8) & 0xFF; oz = (o >> 16) & 0xFF;
}

// Lowest coordinate of the (clipped) 4-block containing coordinate x.
__device__ __forceinline__ int block_lo(int x, int o) { return max(0, ((x + o) >> 2) * 4 - o); }

// Is lattice edge slot e an edge of the comb forest of the current blocked
// sweep?  x-edges inside a block always are; y-edges when both ends have
// local x = 0; z-edges when both ends have local x = y = 0.
__device__ __forceinline__ bool is_tree_edge(const SweepArgs& a, uint32_t e) {
    int ox, oy, oz;
    splash_offset(a.ctl, ox, oy, oz);
    if (e < (uint64_t)a.nxe) {
        const uint32_t r = a.fdX1.div(e);
        const int x = (int)(e - r * (uint32_t)(a.grid_nx - 1));
        return ((x + ox) >> 2) == ((x + 1 + ox) >> 2);
    }
    if (e < (uint64_t)(a.nxe + a.nye)) {
        const uint32_t f = e - (uint32_t)a.nxe;
        const uint32_t r = a.fdX.div(f);
        const int x = (int)(f - r * (uint32_t)a.grid_nx);
        const uint32_t r2 = a.fdY1.div(r);
        const int y = (int)(r - r2 * (uint32_t)(a.grid_ny - 1));
        return x == block_lo(x, ox) && ((y + oy) >> 2) == ((y + 1 + oy) >> 2);
    }
    const uint32_t f = e - (uint32_t)(a.nxe + a.nye);
    const uint32_t r = a.fdX.div(f);
    const int x = (int)(f - r * (uint32_t)a.grid_nx);
    const uint32_t z = a.fdY.div(r);
    const int y = (int)(r - z * (uint32_t)a.grid_ny);
    return x == block_lo(x, ox) && y == block_lo(y, oy) && ((int(z) + oz) >> 2) == ((int(z) + 1 + oz) >> 2);
}

// ---------------------------------------------------------------------------- dual bits

// Row and column masks of the entries of a PIVOT table with at most 64
// entries as 64-bit words: entries (xs, j) and (i, xt).
template <int L>
__device__ __forceinline__ void pivot_masks64(int xs, int xt, uint64_t& Y, uint64_t& Z) {
    constexpr int R = L - 1;
    constexpr uint64_t row = (1ull << R) - 1ull;
    uint64_t col = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) col |= 1ull << (R * r);
    Y = xs ? row << (R * (xs - 1)) : 0ull;
    Z = xt ? col << (xt - 1) : 0ull;
}

// Dual bits of edge e, chain c, given the endpoint labels (xs, xt).
// Bit-sliced: the 8-bit prefixes of 32 uniforms arrive as 8 bit planes (two
// Philox calls per group of 32 entries; one call, two planes per word, when
// the table has at most 16 entries).  An entry's dual logit q + beta1 y +
// beta2 z sits at one of three levels, fixed by its sign s = [l < 0] and its
// case y = [x_s = i_k], z = [x_t = j_k]:
//   s = 0: level y + z,   s = 1: level z - y + 1   (0: -tau, 1: 0, 2: +tau)
// so with X = S ^ Y over a group's masks:
//   L0 = Act & ~Z & ~X,   L2 = Act & Z & X,   L1 = Act & ~(L0 | L2).
// Level 1 is p = 1/2 exactly (T = 2^23): its bit is the complement of the
// prefix's top bit.  For levels 0 and 2 the planes of the matching threshold
// prefix, t = B ^ (AB & L0) (k_build_planes), are compared with the random
// planes least significant first:
//   lt = (~r & t) | (~(r ^ t) & lt)        prefix <  threshold prefix
//   le = (~r & t) | (~(r ^ t) & le)        prefix <= threshold prefix
// Returns lt in bits, the ties le & ~lt (probability 1/256 per entry) in ties
// and the level-2 mask in lev2; a tie is decided by the low 16 bits of its
// uniform against the exact threshold of its level (resolve_tie).
// The Philox calls of the table's first two groups (draw_dual_words) do not
// depend on the labels and come as an argument.
// GLOBAL: the plane table is in global memory (read-only path); else in shared memory.
template <int L, int LAYOUT>
struct DualWords {
    static constexpr int GA = Ent<L, LAYOUT>::W < 2 ? Ent<L, LAYOUT>::W : 2;   // groups drawn together
    static constexpr int N = Ent<L, LAYOUT>::M <= 16 ? 1 : 2 * GA;
};

template <int L, int LAYOUT>
__device__ __forceinline__ void draw_dual_words(uint32_t e, uint32_t c, uint32_t sweep, const RoundKeys& key,
                                                uint4 (&R)[DualWords<L, LAYOUT>::N]) {
    // four calls of two groups share their first rounds and are in flight together
    if constexpr (DualWords<L, LAYOUT>::N == 1) R[0] = draw_rk(e, sweep, c, PH_DUAL, 0u, key);
    else draw_rk_subs<DualWords<L, LAYOUT>::N>(e, sweep, c, PH_DUAL, key, R);
}

template <int L, int LAYOUT, bool GLOBAL = true>
__device__ __forceinline__ void dual_prefix_bits(uint32_t e, uint32_t c, int xs, int xt,
                                                 const uint32_t* __restrict__ tpl_e, uint32_t sweep,
                                                 const RoundKeys& key, uint32_t (&bits)[Ent<L, LAYOUT>::W],
                                                 uint32_t (&ties)[Ent<L, LAYOUT>::W],
                                                 uint32_t (&lev2)[Ent<L, LAYOUT>::W],
                                                 const uint4 (&RA)[DualWords<L, LAYOUT>::N]) {
    using E = Ent<L, LAYOUT>;
    const uint4* tp = reinterpret_cast<const uint4*>(tpl_e);
    auto table = [](const uint4* q) { return GLOBAL ? __ldg(q) : *q; };
    if constexpr (E::M <= 16) {
        // one Philox call: word p = plane p (bits 0..15) and plane p + 4 (bits
        // 16..31); the low halves compare the prefix's high nibble, the high
        // halves its low nibble, combined at the end
        const uint4 r4 = RA[0];
        const uint32_t R[4] = {r4.x, r4.y, r4.z, r4.w};
        const uint4 qa = table(tp), qb = table(tp + 1);
        const uint32_t sa = GLOBAL ? __ldg(tpl_e + 8) : tpl_e[8];
        const uint32_t AB[4] = {qa.x, qa.y, qa.z, qa.w}, B[4] = {qb.x, qb.y, qb.z, qb.w};
        const uint32_t Y = row_mask<L, LAYOUT>(xs, 0), Z = col_mask<L, LAYOUT>(xt, 0);
        const uint32_t X = (sa & 0xFFFFu) ^ Y, act = sa >> 16;
        const uint32_t l0 = act & ~Z & ~X, l2 = act & Z & X, l02 = l0 | l2;
        const uint32_t L0 = l0 | (l0 << 16);
        uint32_t lt = 0u, le = 0xFFFFFFFFu;
#pragma unroll
        for (int p = 3; p >= 0; --p) {
            const uint32_t t = B[p] ^ (AB[p] & L0), r = R[p];
            lt = (~r & t) | (~(r ^ t) & lt);
            le = (~r & t) | (~(r ^ t) & le);
        }
        const uint32_t eq = le & ~lt;
        bits[0] = ((lt | (eq & (lt >> 16))) & l02) | (~R[0] & act & ~l02);
        ties[0] = eq & (eq >> 16) & l02;
        lev2[0] = l2;
        return;
    }
    constexpr bool M64 = LAYOUT == MRF_LAYOUT_PIVOT && E::M <= 64;
    uint64_t Y64 = 0, Z64 = 0;
    if constexpr (M64) pivot_masks64<L>(xs, xt, Y64, Z64);
    constexpr int GA = DualWords<L, LAYOUT>::GA;
#pragma unroll
    for (int g = 0; g < E::W; ++g) {
        uint4 r0, r1;
        if (g < GA) {
            r0 = RA[2 * (g < GA ? g : 0)];
            r1 = RA[2 * (g < GA ? g : 0) + 1];
        } else {
            r0 = draw_rk(e, sweep, c, PH_DUAL, 2u * g, key);
            r1 = draw_rk(e, sweep, c, PH_DUAL, 2u * g + 1u, key);
        }
        const uint32_t Rg[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
        const uint4* tg = tp + 5 * g;
        const uint4 sq = table(tg + 4);                    // {S, Act}
        uint32_t Y, Z;
        if constexpr (M64) {
            Y = (uint32_t)(Y64 >> (32 * g));
            Z = (uint32_t)(Z64 >> (32 * g));
        } else {
            Y = row_mask<L, LAYOUT>(xs, g);
            Z = col_mask<L, LAYOUT>(xt, g);
        }
        const uint32_t X = sq.x ^ Y;
        const uint32_t L0 = sq.y & ~Z & ~X, L2 = sq.y & Z & X, L02 = L0 | L2;
        uint32_t lt = 0u, le = 0xFFFFFFFFu;
#pragma unroll
        for (int h = 3; h >= 0; --h) {
            const uint4 q = table(tg + h);                 // {AB_2h, B_2h, AB_2h+1, B_2h+1}
            uint32_t t = q.w ^ (q.z & L0), r = Rg[2 * h + 1];
            lt = (~r & t) | (~(r ^ t) & lt);
            le = (~r & t) | (~(r ^ t) & le);
            t = q.y ^ (q.x & L0); r = Rg[2 * h];
            lt = (~r & t) | (~(r ^ t) & lt);
            le = (~r & t) | (~(r ^ t) & le);
        }
        bits[g] = (lt & L02) | (~Rg[0] & sq.y & ~L02);
        ties[g] = le & ~lt & L02;
        lev2[g] = L2;
    }
}

// Decision of a tie at entry k (its 8-bit prefix equals the prefix of the
// threshold T of its level): low 16 bits of the uniform < T - (prefix << 16).
__device__ __forceinline__ bool resolve_tie(uint32_t e, uint32_t c, bool lev2, int k, uint32_t thr_word,
                                            uint32_t sweep, const RoundKeys& key) {
    const uint32_t t = level_threshold(thr_word, lev2);
    const uint32_t rem = t - (threshold_prefix(t) << 16);      // in [0, 65536]
    return rem && dual_low16(e, sweep, c, k, key) < rem;
}

// Dual bits with the ties decided by the thread itself, one after another
// (thr_e in global memory, or both tables in shared memory).
template <int L, int LAYOUT, bool GLOBAL = true>
__device__ __forceinline__ void dual_bits(uint32_t e, uint32_t c, int xs, int xt, const uint32_t* __restrict__ tpl_e,
                                          const uint32_t* __restrict__ thr_e, uint32_t sweep, const RoundKeys& key,
                                          uint32_t (&bits)[Ent<L, LAYOUT>::W],
                                          const uint4 (&R)[DualWords<L, LAYOUT>::N]) {
    using E = Ent<L, LAYOUT>;
    uint32_t ties[E::W], lev2[E::W];
    dual_prefix_bits<L, LAYOUT, GLOBAL>(e, c, xs, xt, tpl_e, sweep, key, bits, ties, lev2, R);
#pragma unroll 1
    for (int g = 0; g < E::W; ++g) {
        uint32_t tg = ties[g];
        while (tg) {
            const int b = __ffs(tg) - 1;
            tg &= tg - 1u;
            const int k = 32 * g + b;
            if (resolve_tie(e, c, (lev2[g] >> b) & 1u, k, GLOBAL ? __ldg(thr_e + k) : thr_e[k], sweep, key)) bits[g] |= 1u << b;
        }
    }
}

template <int L, int LAYOUT>
__device__ __forceinline__ void dual_bits(uint32_t e, uint32_t c, int xs, int xt, const uint32_t* __restrict__ tpl_e,
                                          const uint32_t* __restrict__ thr_e, uint32_t sweep, const RoundKeys& key,
                                          uint32_t (&bits)[Ent<L, LAYOUT>::W]) {
    uint4 R[DualWords<L, LAYOUT>::N];
    draw_dual_words<L, LAYOUT>(e, c, sweep, key, R);
    dual_bits<L, LAYOUT, true>(e, c, xs, xt, tpl_e, thr_e, sweep, key, bits, R);
}

// ---------------------------------------------------------------------------- label draw

// The uniform of the top 23 bits of a Philox word: (U + 1/2) 2^-23, exact in float32.
__device__ __forceinline__ float uniform23(uint32_t word) {
    return __uint_as_float(0x3F800000u | (word >> 9)) - 0x1.fffffep-1f;
}

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0,%1;" : "=f"(y) : "f"(x));
    return y;
}

// First label a with u < cdf_a where the float32 inverse CDF below is sure to
// agree, -1 otherwise.  The unnormalised sums c_a of the hardware's 2^x
// (relative error 2^-22) are within 2e-6 s of the exact sums, and the CDF of
// the full computation (expf, division, L <= 16 additions) within 3e-6 of the
// exact one; so if every |c_a - u s| is at least 2^-16 s, both give the same
// label, and no boundary is within the 1e-6 that draw_label counts.  Takes 7
// instructions per label where the full computation takes 18; about one draw in
// 4,000 (L = 8) falls back to it.
// The rounding error of mb scales all the sums alike by 2^r, |r| up to half an
// ulp of mb: s is in [1, L] but for that.  From fields of 1.5e9 on it can pass the
// exponent range, where every term is 0 or infinite and the closeness test holds
// for any label, so sums outside [2^-32, 2^32] (fields of 5e8 and more, NaN and
// infinite fields) take the full computation.
template <int L>
__device__ __forceinline__ int draw_label_fast(const float (&F)[L], float u) {
    constexpr float kLog2e = 1.4426950408889634f;
    float mx = F[0];
#pragma unroll
    for (int a = 1; a < L; ++a) mx = fmaxf(mx, F[a]);
    const float mb = mx * kLog2e;
    float c[L], s = 0.0f;
#pragma unroll
    for (int a = 0; a < L; ++a) {
        s += ex2_approx(fmaf(F[a], kLog2e, -mb));
        c[a] = s;
    }
    const float us = u * s;
    float closest = INFINITY;
    int lab = 0;
#pragma unroll
    for (int a = 0; a < L; ++a) {
        const float d = c[a] - us;
        closest = fminf(closest, fabsf(d));
        lab += d <= 0.0f ? 1 : 0;
    }
    return s >= 0x1p-32f && s <= 0x1p32f && closest >= s * 0x1p-16f ? lab : -1;
}

// Draw x_v from exp(F)/Z by the inverse CDF with the 23-bit uniform u (exact in
// float32); optionally record log p.  Counts draws within 1e-6 of a CDF
// boundary.  lp_drawn (optional) receives log p of the drawn label.
template <int L>
__device__ __forceinline__ int draw_label_at(const float (&F)[L], float u, float* __restrict__ logp_out, Ctl* ctl,
                                             float* __restrict__ lp_drawn = nullptr) {
    if (!logp_out && !lp_drawn) {
        const int lab = draw_label_fast<L>(F, u);
        if (lab >= 0) return lab;
    }
    float mx = F[0];
#pragma unroll
    for (int a = 1; a < L; ++a) mx = fmaxf(mx, F[a]);
    float ex[L];
    float s = 0.0f;
#pragma unroll
    for (int a = 0; a < L; ++a) {
        ex[a] = expf(F[a] - mx);
        s += ex[a];
    }
    const float inv = 1.0f / s;
    if (logp_out) {
        const float ls = logf(s);
#pragma unroll
        for (int a = 0; a < L; ++a) logp_out[a] = (F[a] - mx) - ls;
    }
    float cdf = 0.0f;
    int lab = -1, last_pos = 0;
    bool near = false;
#pragma unroll
    for (int a = 0; a < L; ++a) {
        const float p = ex[a] * inv;
        cdf += p;
        if (p > 0.0f) last_pos = a;
        if (lab < 0 && u < cdf) lab = a;
        near |= fabsf(u - cdf) < 1e-6f;
    }
    if (near) atomicAdd(&ctl->boundary, 1ull);
    const int pick = lab < 0 ? last_pos : lab;
    if (lp_drawn) {
        float fp = F[0];
#pragma unroll
        for (int a = 1; a < L; ++a) fp = a == pick ? F[a] : fp;
        *lp_drawn = (fp - mx) - logf(s);
    }
    return pick;
}

// The same with the uniform of Philox phase `phase` for site v, chain c.
template <int L>
__device__ __forceinline__ int draw_label(const float (&F)[L], uint32_t v, uint32_t c, uint32_t sweep,
                                          const RoundKeys& key, uint32_t phase, float* __restrict__ logp_out, Ctl* ctl,
                                          float* __restrict__ lp_drawn = nullptr) {
    return draw_label_at<L>(F, uniform23(draw_rk(v, sweep, c, phase, 0, key).x), logp_out, ctl, lp_drawn);
}

// ---------------------------------------------------------------------------- kernels

// Dual step.  A warp takes NG consecutive groups of 32 (edge, chain) items
// (item g = e C + c, one item per lane).  A tie needs one more Philox call and
// a scattered threshold word; deciding it in the owning lane would hold the
// whole warp for a few lanes.  Instead the warp stages its dual words in
// shared memory and queues every nonzero tie word of a lane as one entry
// {group, lane, word | tie mask | level-2 mask}; after its NG groups the warp
// decides the queued entries with one entry per lane per round and ORs the
// won bits into the staged words, which are then stored.  Ties of a lane
// whose entry does not fit the queue are decided by the lane itself.
// PART: ng < NG groups per warp, where NG would leave SMs without a block
// (run_dual); an instance of its own, for the loop bound's sake (a variable
// bound for all cost 9 % on 447,262 edges of L = 5, 24 chains).
template <int M, int W>
struct DualTile {
    static constexpr int WARPS = 8;                                         // 256 threads
    static constexpr int NG = W >= 4 ? 2 : (M >= 32 ? 4 : (M >= 8 ? 8 : 16));
    // nonzero tie words expected per warp: NG 32 W (1 - (1 - 1/256)^32) <= NG 32 M / 256;
    // capacity twice that plus 32, in whole rounds of 32
    static constexpr int Q = ((NG * 32 * M * 2 / 256 + 32) + 31) / 32 * 32;
};

// FEW: the launch bounds of the form for fewer than 32 chains (run_dual).
template <int L, int LAYOUT, bool FEW = false, bool PART = false>
__global__ void __launch_bounds__(256, FEW ? 2 : 4) k_dual(SweepArgs a, int n_groups) {
    using E = Ent<L, LAYOUT>;
    using T = DualTile<E::M, E::W>;
    constexpr int W = E::W, NG = T::NG, Q = T::Q;
    const int ng = PART ? n_groups : NG;
    constexpr uint32_t FULL = 0xFFFFFFFFu;
    __shared__ uint32_t s_th[T::WARPS][NG * W][32];        // staged dual words, [group, word][lane]
    __shared__ uint4 s_q[T::WARPS][Q];                     // queued tie words
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t below = (1u << lane) - 1u;
    const uint64_t n_items = (uint64_t)a.E * a.C;          // < 2^32 (checked by the host)
    const uint64_t base = ((uint64_t)blockIdx.x * T::WARPS + warp) * (ng * 32);
    const uint32_t sweep = (uint32_t)a.ctl->sweep;
    const uint8_t* xin = a.x + (size_t)(sweep & 1) * a.N * a.C;
    int nq = 0;                                            // entries queued (warp-uniform)
#pragma unroll 1
    for (int j = 0; j < ng; ++j) {
        const uint64_t g64 = base + 32 * j + lane;
        const uint32_t g = (uint32_t)g64;
        const bool in_range = g64 < n_items;
        const uint32_t e = in_range ? a.fdC.div(g) : 0u;
        const uint32_t c = g - e * (uint32_t)a.C;
        uint32_t bits[W], ties[W], lev2[W];
        const int s = in_range ? a.src[e] : -1;
        if (s >= 0 && !(a.splash && is_tree_edge(a, e)) && !(a.skip && a.skip[e])) {
            const int t = a.dst[e];
            const int xs = xin[(int64_t)s * a.C + c], xt = xin[(int64_t)t * a.C + c];
            uint4 R[DualWords<L, LAYOUT>::N];
            draw_dual_words<L, LAYOUT>(e, c, sweep, a.rk, R);
            dual_prefix_bits<L, LAYOUT>(e, c, xs, xt, a.tpl + (int64_t)e * E::PW, sweep, a.rk, bits, ties, lev2, R);
        } else {
#pragma unroll
            for (int w = 0; w < W; ++w) { bits[w] = 0u; ties[w] = 0u; lev2[w] = 0u; }
        }
#pragma unroll
        for (int w = 0; w < W; ++w) {
            const bool has = ties[w] != 0u;
            const uint32_t bal = __ballot_sync(FULL, has);
            const int pos = nq + __popc(bal & below);
            nq += __popc(bal);
            if (has) {
                if (pos < Q) {
                    s_q[warp][pos] = make_uint4((uint32_t)(j * W + w) | ((uint32_t)lane << 8), ties[w], lev2[w] & ties[w], 0u);
                } else {
                    uint32_t tw = ties[w];                 // queue full: decide here
                    while (tw) {
                        const int b = __ffs(tw) - 1;
                        tw &= tw - 1u;
                        const int k = 32 * w + b;
                        if (resolve_tie(e, c, (lev2[w] >> b) & 1u, k, __ldg(a.thr + (int64_t)e * E::M + k), sweep, a.rk))
                            bits[w] |= 1u << b;
                    }
                }
            }
            s_th[warp][j * W + w][lane] = bits[w];
        }
    }
    __syncwarp();
    const int nres = nq < Q ? nq : Q;
#pragma unroll 1
    for (int r = lane; r < nres; r += 32) {
        const uint4 q = s_q[warp][r];
        const int jw = (int)(q.x & 0xFFu), l = (int)(q.x >> 8), j = jw / W, w = jw - j * W;
        const uint32_t g = (uint32_t)(base + 32 * j + l);
        const uint32_t e = a.fdC.div(g), c = g - e * (uint32_t)a.C;
        uint32_t tw = q.y, won = 0u;
        while (tw) {
            const int b = __ffs(tw) - 1;
            tw &= tw - 1u;
            const int k = 32 * w + b;
            if (resolve_tie(e, c, (q.z >> b) & 1u, k, __ldg(a.thr + (int64_t)e * E::M + k), sweep, a.rk)) won |= 1u << b;
        }
        if (won) atomicOr(&s_th[warp][jw][l], won);
    }
    __syncwarp();
#pragma unroll 1
    for (int j = 0; j < ng; ++j) {
        const uint64_t g64 = base + 32 * j + lane;
        if (g64 >= n_items) break;
        uint32_t* out = a.theta + g64 * W;
        if (W % 2 == 0) {
#pragma unroll
            for (int w = 0; w < W; w += 2)
                *reinterpret_cast<uint2*>(out + w) = make_uint2(s_th[warp][j * W + w][lane], s_th[warp][j * W + (w + 1 < W ? w + 1 : w)][lane]);
        } else {
#pragma unroll
            for (int w = 0; w < W; ++w) out[w] = s_th[warp][j * W + w][lane];
        }
    }
}

// Conditional additions of up to seven set dual bits, bits 0..n-1 of m.  A bit
// test and a predicated add per entry kept the ALU pipe of the primal step busy
// (two cycles per warp for a test); written as one block of bit tests followed
// by the adds, the tests of a block become one move of the word into the seven
// predicate registers.  49 entries took 65 ALU-pipe instructions before and
// take 17 (12 of them shifts and moves of the words).
#define MRF_BT1(M) "and.b32 a0," M ",1;setp.ne.u32 p0,a0,0;"
#define MRF_BT2(M) MRF_BT1(M) "and.b32 a1," M ",2;setp.ne.u32 p1,a1,0;"
#define MRF_BT3(M) MRF_BT2(M) "and.b32 a2," M ",4;setp.ne.u32 p2,a2,0;"
#define MRF_BT4(M) MRF_BT3(M) "and.b32 a3," M ",8;setp.ne.u32 p3,a3,0;"
#define MRF_BT5(M) MRF_BT4(M) "and.b32 a4," M ",16;setp.ne.u32 p4,a4,0;"
#define MRF_BT6(M) MRF_BT5(M) "and.b32 a5," M ",32;setp.ne.u32 p5,a5,0;"
#define MRF_BT7(M) MRF_BT6(M) "and.b32 a6," M ",64;setp.ne.u32 p6,a6,0;"
#define MRF_BR1 "@p0 add.f32 %0,%0,%2;"
#define MRF_BR2 MRF_BR1 "@p1 add.f32 %0,%0,%3;"
#define MRF_BR3 MRF_BR2 "@p2 add.f32 %0,%0,%4;"
#define MRF_BR4 MRF_BR3 "@p3 add.f32 %0,%0,%5;"
#define MRF_BR5 MRF_BR4 "@p4 add.f32 %0,%0,%6;"
#define MRF_BR6 MRF_BR5 "@p5 add.f32 %0,%0,%7;"
#define MRF_BR7 MRF_BR6 "@p6 add.f32 %0,%0,%8;"
#define MRF_BE1 "@p0 add.f32 %0,%0,%8;"
#define MRF_BE2 MRF_BE1 "@p1 add.f32 %1,%1,%9;"
#define MRF_BE3 MRF_BE2 "@p2 add.f32 %2,%2,%10;"
#define MRF_BE4 MRF_BE3 "@p3 add.f32 %3,%3,%11;"
#define MRF_BE5 MRF_BE4 "@p4 add.f32 %4,%4,%12;"
#define MRF_BE6 MRF_BE5 "@p5 add.f32 %5,%5,%13;"
#define MRF_BE7 MRF_BE6 "@p6 add.f32 %6,%6,%14;"
#define MRF_BITS_REGS "{.reg .pred p0,p1,p2,p3,p4,p5,p6;.reg .b32 a0,a1,a2,a3,a4,a5,a6;"
#define MRF_BITS_ROW(n)                                                                                        \
    if constexpr (N == n)                                                                                      \
        asm(MRF_BITS_REGS MRF_BT##n("%1") MRF_BR##n "}"                                                        \
            : "+f"(acc)                                                                                        \
            : "r"(m), "f"(t[0]), "f"(t[1]), "f"(t[2]), "f"(t[3]), "f"(t[4]), "f"(t[5]), "f"(t[6]))
#define MRF_BITS_EACH(n)                                                                                       \
    if constexpr (N == n)                                                                                      \
        asm(MRF_BITS_REGS MRF_BT##n("%7") MRF_BE##n "}"                                                        \
            : "+f"(r[0]), "+f"(r[1]), "+f"(r[2]), "+f"(r[3]), "+f"(r[4]), "+f"(r[5]), "+f"(r[6])               \
            : "r"(m), "f"(t[0]), "f"(t[1]), "f"(t[2]), "f"(t[3]), "f"(t[4]), "f"(t[5]), "f"(t[6]))

// acc += t[0..N-1] of the set bits, in order.
template <int N>
__device__ __forceinline__ void add_bits_row(uint32_t m, const float (&t)[7], float& acc) {
    MRF_BITS_ROW(1); MRF_BITS_ROW(2); MRF_BITS_ROW(3); MRF_BITS_ROW(4); MRF_BITS_ROW(5); MRF_BITS_ROW(6); MRF_BITS_ROW(7);
}

// acc[i] += t[i] for every set bit i < N.
template <int N>
__device__ __forceinline__ void add_bits_each(uint32_t m, const float (&t)[7], float* acc) {
    float r[7];
#pragma unroll
    for (int i = 0; i < 7; ++i) r[i] = i < N ? acc[i] : 0.0f;
    MRF_BITS_EACH(1); MRF_BITS_EACH(2); MRF_BITS_EACH(3); MRF_BITS_EACH(4); MRF_BITS_EACH(5); MRF_BITS_EACH(6);
    MRF_BITS_EACH(7);
#pragma unroll
    for (int i = 0; i < N; ++i) acc[i] = r[i];
}

// Entries [K0, K0 + N) of one table row: the dual words' bits K0.. as the low bits of a word.
template <int K0, int N, int W>
__device__ __forceinline__ uint32_t entry_bits(const uint32_t (&bits)[W]) {
    constexpr int g = K0 >> 5, sh = K0 & 31;
    if constexpr (sh == 0) return bits[g];
    else if constexpr (sh + N <= 32) return bits[g] >> sh;
    else return __funnelshift_r(bits[g], bits[g + 1 < W ? g + 1 : g], sh);
}

// Entries K0 .. K1-1 of one table row (PIVOT: row label i, first column label
// j0; DIAG: entries are labels), seven at a time, for CH chains.
template <int L, int LAYOUT, int CH, int K0, int K1>
__device__ __forceinline__ void add_span(const uint32_t (&bits)[CH][Ent<L, LAYOUT>::W],
                                         const float (&tv)[Ent<L, LAYOUT>::MP], int side, float (&acc)[CH][L]) {
    if constexpr (K0 < K1) {
        using E = Ent<L, LAYOUT>;
        constexpr int N = K1 - K0 < 7 ? K1 - K0 : 7;
        float t[7];
#pragma unroll
        for (int i = 0; i < 7; ++i) t[i] = i < N ? (side == 0 ? tv[K0 + (i < N ? i : 0)] : fabsf(tv[K0 + (i < N ? i : 0)])) : 0.0f;
#pragma unroll
        for (int h = 0; h < CH; ++h) {
            const uint32_t m = entry_bits<K0, N, E::W>(bits[h]);
            if (LAYOUT == MRF_LAYOUT_PIVOT && side == 0) add_bits_row<N>(m, t, acc[h][E::i(K0)]);
            else add_bits_each<N>(m, t, &acc[h][E::j(K0)]);
        }
        add_span<L, LAYOUT, CH, K0 + N, K1>(bits, tv, side, acc);
    }
}

template <int L, int LAYOUT, bool GLOBAL, int CH, int ROW>
__device__ __forceinline__ void add_rows(const uint32_t (&bits)[CH][Ent<L, LAYOUT>::W], const float4* __restrict__ t4,
                                         float (&tv)[Ent<L, LAYOUT>::MP], int side, float (&acc)[CH][L]) {
    using E = Ent<L, LAYOUT>;
    constexpr int R = LAYOUT == MRF_LAYOUT_PIVOT ? L - 1 : L;      // entries per table row
    if constexpr (ROW * R < E::M) {
        constexpr int q0 = (ROW * R + 3) / 4, q1 = ((ROW + 1) * R + 3) / 4;   // vectors not loaded by earlier rows
#pragma unroll
        for (int k4 = q0; k4 < q1; ++k4) {
            const float4 q = GLOBAL ? __ldg(t4 + k4) : t4[k4];
            tv[4 * k4] = q.x; tv[4 * k4 + 1] = q.y; tv[4 * k4 + 2] = q.z; tv[4 * k4 + 3] = q.w;
        }
        add_span<L, LAYOUT, CH, ROW * R, (ROW + 1) * R>(bits, tv, side, acc);
        add_rows<L, LAYOUT, GLOBAL, CH, ROW + 1>(bits, t4, tv, side, acc);
    }
}

// Accumulate the beta terms of edge e's set dual bits for one endpoint side
// (tau row loaded as 16-byte vectors; beta1 = tau_signed, beta2 = |tau_signed|),
// in entry order, for CH chains.
// GLOBAL: the row is in global memory (read-only path); else in shared memory.
template <int L, int LAYOUT, bool GLOBAL, int CH>
__device__ __forceinline__ void add_side_chains(const uint32_t (&bits)[CH][Ent<L, LAYOUT>::W],
                                                const float* __restrict__ tau_e, int side, float (&acc)[CH][L]) {
    const float4* t4 = reinterpret_cast<const float4*>(tau_e);
    float tv[Ent<L, LAYOUT>::MP];
    if (side == 0) add_rows<L, LAYOUT, GLOBAL, CH, 0>(bits, t4, tv, 0, acc);
    else add_rows<L, LAYOUT, GLOBAL, CH, 0>(bits, t4, tv, 1, acc);
}

// The same with a test and an add per entry, for the thread form (k_primal) of 3, 7
// to 10 and 12 to 15 labels: the grouped form holds a block's weights and predicates
// at once, and at 64 registers its sums spill from L = 9 on.  us per sweep, single /
// grouped: random graphs of degree 24, 5 chains, 79,992 edges: L = 9 76 / 78, L = 10
// 112 / 115, L = 12 170 / 175; a complete graph of 89 sites, 5 chains, L = 12 180 / 195;
// the primal step of two million lattice items: L = 3 0.85 to 1.0 times the grouped
// form's time, L = 7 0.93 to 0.97, L = 8 0.92 to 1.0; 36,000 sites, 18 chains: L = 14
// 145 / 159, L = 15 163 / 183.  L = 6 and 11 are even, L = 2, 4, 5 up to 1.1 and L = 16
// (466 / 381) better grouped.  The fused form: from 8 labels on (76,000 lattice sites, 2
// chains: L = 8 57 / 63, L = 10 90 / 102, L = 12 122 / 135, L = 16 256 / 284).
template <int L, int LAYOUT, bool FUSED>
constexpr bool kSingleAdds = LAYOUT == MRF_LAYOUT_PIVOT &&
                             (FUSED ? L >= 8 : L == 3 || (L >= 7 && L <= 15 && L != 11));

template <int L, int LAYOUT>
__device__ __forceinline__ void add_side_single(const uint32_t (&bits)[Ent<L, LAYOUT>::W], const float* __restrict__ tau_e,
                                                int side, float (&acc)[L]) {
    using E = Ent<L, LAYOUT>;
    const float4* t4 = reinterpret_cast<const float4*>(tau_e);
    if (side == 0) {
#pragma unroll
        for (int k4 = 0; k4 < E::MP / 4; ++k4) {
            const float4 q = __ldg(t4 + k4);
            const float tv[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = 4 * k4 + u;
                if (k < E::M && ((bits[k >> 5] >> (k & 31)) & 1u)) acc[E::i(k)] += tv[u];
            }
        }
    } else {
#pragma unroll
        for (int k4 = 0; k4 < E::MP / 4; ++k4) {
            const float4 q = __ldg(t4 + k4);
            const float tv[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = 4 * k4 + u;
                if (k < E::M && ((bits[k >> 5] >> (k & 31)) & 1u)) acc[E::j(k)] += fabsf(tv[u]);
            }
        }
    }
}

template <int L, int LAYOUT, bool GLOBAL = true>
__device__ __forceinline__ void add_side(const uint32_t (&bits)[Ent<L, LAYOUT>::W], const float* __restrict__ tau_e,
                                         int side, float (&acc)[L]) {
    add_side_chains<L, LAYOUT, GLOBAL, 1>(reinterpret_cast<const uint32_t(&)[1][Ent<L, LAYOUT>::W]>(bits), tau_e, side,
                                          reinterpret_cast<float(&)[1][L]>(acc));
}

// Compensated (two-sum) flush of a float32 partial sum into a hi/lo pair, used
// every 32 incident edges so that high-degree sites keep ~double precision.
__device__ __forceinline__ void two_sum_add(float& hi, float& lo, float x) {
    const float s = hi + x;
    const float bp = s - hi;
    lo += (hi - (s - bp)) + (x - bp);
    hi = s;
}

// FUSED = false: read theta written by k_dual.  FUSED = true: regenerate it.
// POT = true (blocked sweep): write the node potentials F to a.pot instead of
// drawing labels.
// Four blocks per SM even where the field arrays of wide tables spill at 64
// registers (L = 9: 354 B, L = 16: 702 B): fewer blocks measured slower (L = 8,
// one chain: 0.403 vs 0.386 ms; L = 10, 8 chains: 0.68 vs 0.60 ms; L = 12, 16
// chains: 0.39 vs 0.26 ms; L = 16, 8 chains: 2.22 vs 1.34 ms).
template <int L, int LAYOUT, bool FUSED, bool POT = false>
__global__ void __launch_bounds__(256, FUSED ? 2 : 4) k_primal(SweepArgs a) {
    using E = Ent<L, LAYOUT>;
    const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;     // N * C < 2^32 (checked by the host)
    if (g >= (uint64_t)a.N * a.C) return;
    const uint32_t v = a.fdC.div(g), c = g - v * (uint32_t)a.C;
    const uint32_t sweep = (uint32_t)a.ctl->sweep;
    const uint8_t* xin = a.x + (size_t)(sweep & 1) * a.N * a.C;
    uint8_t* xout = a.x + (size_t)((sweep + 1) & 1) * a.N * a.C;
    float acc[L], hi[L], lo[L];
#pragma unroll
    for (int x = 0; x < L; ++x) { acc[x] = 0.0f; hi[x] = 0.0f; lo[x] = 0.0f; }
    int xv = 0;
    if (FUSED) xv = xin[g];
    const int64_t p0 = a.inc_ptr[v], p1 = a.inc_ptr[v + 1];
    if (!FUSED && p1 - p0 > a.hub_deg) return;                    // k_primal_hub's
    int chunk = 0;
    bool flushed = false;
    // Incidences in batches of B: all incidence records and (plain form) all
    // theta words of a batch are loaded before any is used, so the dependent
    // loads of B edges are in flight together.
    constexpr int B = FUSED ? 1 : 4;
    for (int64_t base = p0; base < p1; base += B) {
        int2 ic[B];
        uint32_t bits[B][E::W];
#pragma unroll
        for (int u = 0; u < B; ++u) ic[u] = base + u < p1 ? __ldg(&a.inc[base + u]) : make_int2(-1, 0);
#pragma unroll
        for (int u = 0; u < B; ++u) {
            const int64_t e = ic[u].x >> 1;
            if (ic[u].x < 0) {
#pragma unroll
                for (int w = 0; w < E::W; ++w) bits[u][w] = 0;
            } else if (FUSED) {
                const int side = ic[u].x & 1;
                const int xn = xin[(int64_t)ic[u].y * a.C + c];
                dual_bits<L, LAYOUT>((uint32_t)e, c, side == 0 ? xv : xn, side == 0 ? xn : xv, a.tpl + e * E::PW,
                                     a.thr + e * E::M, sweep, a.rk, bits[u]);
            } else {
                const uint32_t* th = a.theta + (e * a.C + c) * E::W;
                if (E::W % 2 == 0) {
#pragma unroll
                    for (int w = 0; w < E::W; w += 2) {
                        const uint2 q = __ldcs(reinterpret_cast<const uint2*>(th + w));
                        bits[u][w] = q.x;
                        bits[u][w + 1 < E::W ? w + 1 : w] = q.y;
                    }
                } else {
#pragma unroll
                    for (int w = 0; w < E::W; ++w) bits[u][w] = __ldcs(th + w);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < B; ++u) {
            if (ic[u].x < 0) continue;
            if constexpr (kSingleAdds<L, LAYOUT, FUSED>) add_side_single<L, LAYOUT>(bits[u], a.tau + (ic[u].x >> 1) * (int64_t)E::MP, ic[u].x & 1, acc);
            else add_side<L, LAYOUT>(bits[u], a.tau + (ic[u].x >> 1) * (int64_t)E::MP, ic[u].x & 1, acc);
            if (++chunk == 32) {
#pragma unroll
                for (int x = 0; x < L; ++x) { two_sum_add(hi[x], lo[x], acc[x]); acc[x] = 0.0f; }
                chunk = 0;
                flushed = true;
            }
        }
    }
    float F[L];
    const float* uf = a.utf + (int64_t)v * L;
    if (flushed) {
#pragma unroll
        for (int x = 0; x < L; ++x) { two_sum_add(hi[x], lo[x], acc[x]); F[x] = __ldg(uf + x) + (hi[x] + lo[x]); }
    } else {
#pragma unroll
        for (int x = 0; x < L; ++x) F[x] = __ldg(uf + x) + acc[x];
    }
    if (POT) {
        float* pv = a.pot + (int64_t)v * L * a.C + c;
#pragma unroll
        for (int x = 0; x < L; ++x) pv[(int64_t)x * a.C] = F[x];
        return;
    }
    float* lp = a.logp ? a.logp + ((int64_t)c * a.N + v) * L : nullptr;
    xout[g] = (uint8_t)draw_label<L>(F, v, c, sweep, a.rk, PH_PRIMAL, lp, a.ctl, a.lpv ? a.lpv + g : nullptr);
}

// Thread form for sites of at most KB incidences: every incidence code, then
// every dual word of the site is loaded before any is used (two dependent loads
// where batches of four made four), and no two-sum pair is kept, since no sum
// reaches 32 incidences.  Keeps k_primal's order of additions (entry by entry: 0.92
// to 0.98 of the grouped form's time at L = 5).  151,951 sites of a lattice, L = 5,
// 24 chains: 120 -> 101 us with grouped additions, 0.95 of that with single ones.
template <int L, int LAYOUT, bool POT = false>
__global__ void __launch_bounds__(256, 4) k_primal_low(SweepArgs a) {
    using E = Ent<L, LAYOUT>;
    constexpr int W = E::W, KB = 8;
    static_assert(W <= 2, "the dual words of KB incidences are in registers");
    const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;     // N * C < 2^32 (checked by the host)
    if (g >= (uint64_t)a.N * a.C) return;
    const uint32_t v = a.fdC.div(g), c = g - v * (uint32_t)a.C;
    const int64_t p0 = a.inc_ptr[v];
    const int deg = (int)(a.inc_ptr[v + 1] - p0);
    int code[KB];
#pragma unroll
    for (int u = 0; u < KB; ++u) code[u] = u < deg ? __ldg(&a.inc[p0 + u].x) : -1;
    uint32_t bits[KB][W];
#pragma unroll
    for (int u = 0; u < KB; ++u) {
        if (code[u] < 0) continue;
        const uint32_t* th = a.theta + ((uint64_t)((uint32_t)code[u] >> 1) * (uint32_t)a.C + c) * W;
        if constexpr (W == 2) {
            const uint2 q = __ldcs(reinterpret_cast<const uint2*>(th));
            bits[u][0] = q.x;
            bits[u][1] = q.y;
        } else {
            bits[u][0] = __ldcs(th);
        }
    }
    float acc[L];
#pragma unroll
    for (int x = 0; x < L; ++x) acc[x] = 0.0f;
#pragma unroll
    for (int u = 0; u < KB; ++u)
        if (code[u] >= 0) {
            const float* tau = a.tau + (uint64_t)((uint32_t)code[u] >> 1) * E::MP;
            if constexpr (LAYOUT == MRF_LAYOUT_PIVOT) add_side_single<L, LAYOUT>(bits[u], tau, code[u] & 1, acc);
            else add_side<L, LAYOUT>(bits[u], tau, code[u] & 1, acc);
        }
    float F[L];
    const float* uf = a.utf + (int64_t)v * L;
#pragma unroll
    for (int x = 0; x < L; ++x) F[x] = __ldg(uf + x) + acc[x];
    if (POT) {
        float* pv = a.pot + (int64_t)v * L * a.C + c;
#pragma unroll
        for (int x = 0; x < L; ++x) pv[(int64_t)x * a.C] = F[x];
        return;
    }
    const uint32_t sweep = (uint32_t)a.ctl->sweep;
    uint8_t* xout = a.x + (size_t)((sweep + 1) & 1) * a.N * a.C;
    float* lp = a.logp ? a.logp + ((int64_t)c * a.N + v) * L : nullptr;
    xout[g] = (uint8_t)draw_label<L>(F, v, c, sweep, a.rk, PH_PRIMAL, lp, a.ctl, a.lpv ? a.lpv + g : nullptr);
}

// Warp-per-site form of the plain primal step (chains a multiple of 32, so a
// warp is one site and 32 of its chains).  BATCH (chosen by the host when no
// site has more than KB incidences, e.g. every lattice): one batch per site --
// the lanes load the incidence records in parallel, every lane issues the
// theta loads of all incidences at once, the incidences' tau rows are staged
// in shared memory (one row per incidence, shared by the 32 chains), then the
// field is summed.  Otherwise chunks of K incidences (same pattern, a two-sum
// flush of the partial sums every 32 incidences).  Both keep k_primal's order
// of additions.
template <int L, int LAYOUT>
struct PrimalWarp {
    static constexpr int MP = Ent<L, LAYOUT>::MP;
    static constexpr int W = Ent<L, LAYOUT>::W;
    static constexpr int K = 2;                          // incidences per chunk of the general path
    static constexpr int KB = W >= 8 ? 2 : (W >= 4 ? 4 : 8);   // one-batch path: degree <= KB
    static constexpr int WARPS = 8;                      // 256 threads
};

template <int L, int LAYOUT, bool POT = false, bool BATCH = false>
__global__ void __launch_bounds__(256, 4) k_primal_warp(SweepArgs a) {
    using E = Ent<L, LAYOUT>;
    using PW = PrimalWarp<L, LAYOUT>;
    constexpr int K = PW::K, KB = PW::KB, MP = PW::MP, Q = MP / 4;    // float4 per tau row
    constexpr uint32_t FULL = 0xFFFFFFFFu;
    __shared__ __align__(16) float4 s_tau[PW::WARPS][KB > K ? KB : K][Q];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;     // N * C < 2^32, C % 32 == 0 (host)
    if (g >= (uint64_t)a.N * a.C) return;                         // whole warps only
    const uint32_t v = a.fdC.div(g), c = g - v * (uint32_t)a.C;
    const uint32_t sweep = (uint32_t)a.ctl->sweep;
    uint8_t* xout = a.x + (size_t)((sweep + 1) & 1) * a.N * a.C;
    const int64_t p0 = a.inc_ptr[v], p1 = a.inc_ptr[v + 1];
    if (p1 - p0 > a.hub_deg) return;                              // k_primal_hub's
    const float4* tau4 = reinterpret_cast<const float4*>(a.tau);
    float F[L];
    const float* uf = a.utf + (int64_t)v * L;
    if constexpr (BATCH) {                                        // every site has at most KB incidences
        const int deg = (int)(p1 - p0);
        float acc[L];
#pragma unroll
        for (int x = 0; x < L; ++x) acc[x] = 0.0f;
        const int code_l = lane < deg ? __ldg(&a.inc[p0 + lane]).x : 0;
        uint32_t bits[KB][E::W];
#pragma unroll
        for (int u = 0; u < KB; ++u) {
            const int cu = __shfl_sync(FULL, code_l, u);
            if (u < deg) {
                const uint32_t* th = a.theta + ((int64_t)(cu >> 1) * a.C + c) * E::W;
                if (E::W % 2 == 0) {
#pragma unroll
                    for (int w = 0; w < E::W; w += 2) {
                        const uint2 q = __ldcs(reinterpret_cast<const uint2*>(th + w));
                        bits[u][w] = q.x;
                        bits[u][w + 1 < E::W ? w + 1 : w] = q.y;
                    }
                } else {
#pragma unroll
                    for (int w = 0; w < E::W; ++w) bits[u][w] = __ldcs(th + w);
                }
            }
        }
#pragma unroll
        for (int i0 = 0; i0 < KB * Q; i0 += 32) {
            const int i = i0 + lane;
            const int u = i / Q;
            const int cu = __shfl_sync(FULL, code_l, u < KB ? u : 0);
            if (i < KB * Q && u < deg) s_tau[warp][u][i - u * Q] = __ldg(tau4 + (int64_t)(cu >> 1) * Q + (i - u * Q));
        }
        __syncwarp();
#pragma unroll
        for (int u = 0; u < KB; ++u) {
            if (u >= deg) break;
            const int cu = __shfl_sync(FULL, code_l, u);
            add_side<L, LAYOUT, false>(bits[u], reinterpret_cast<const float*>(&s_tau[warp][u][0]), cu & 1, acc);
        }
#pragma unroll
        for (int x = 0; x < L; ++x) F[x] = __ldg(uf + x) + acc[x];
    } else {
        float acc[L], hi[L], lo[L];
    #pragma unroll
        for (int x = 0; x < L; ++x) { acc[x] = 0.0f; hi[x] = 0.0f; lo[x] = 0.0f; }
        int chunk = 0;
        bool flushed = false;
        for (int64_t base = p0; base < p1; base += K) {              // warp-uniform
            const int cnt = p1 - base < K ? (int)(p1 - base) : K;
            const int code_l = lane < cnt ? __ldg(&a.inc[base + lane]).x : 0;
            // tau rows of the chunk -> shared memory (uniform trip count; lanes split the float4s)
    #pragma unroll
            for (int i0 = 0; i0 < K * Q; i0 += 32) {
                const int i = i0 + lane;
                const int u = i / Q;
                const int cu = __shfl_sync(FULL, code_l, u < K ? u : 0);
                if (i < K * Q && u < cnt) s_tau[warp][u][i - u * Q] = __ldg(tau4 + (int64_t)(cu >> 1) * Q + (i - u * Q));
            }
            uint32_t bits[K][E::W];
            int code[K];
    #pragma unroll
            for (int u = 0; u < K; ++u) {
                code[u] = __shfl_sync(FULL, code_l, u);
                if (u < cnt) {
                    const uint32_t* th = a.theta + ((int64_t)(code[u] >> 1) * a.C + c) * E::W;
                    if (E::W % 2 == 0) {
    #pragma unroll
                        for (int w = 0; w < E::W; w += 2) {
                            const uint2 q = __ldcs(reinterpret_cast<const uint2*>(th + w));
                            bits[u][w] = q.x;
                            bits[u][w + 1 < E::W ? w + 1 : w] = q.y;
                        }
                    } else {
    #pragma unroll
                        for (int w = 0; w < E::W; ++w) bits[u][w] = __ldcs(th + w);
                    }
                }
            }
            __syncwarp();
    #pragma unroll
            for (int u = 0; u < K; ++u) {
                if (u >= cnt) break;
                add_side<L, LAYOUT, false>(bits[u], reinterpret_cast<const float*>(&s_tau[warp][u][0]), code[u] & 1, acc);
                if (++chunk == 32) {
    #pragma unroll
                    for (int x = 0; x < L; ++x) { two_sum_add(hi[x], lo[x], acc[x]); acc[x] = 0.0f; }
                    chunk = 0;
                    flushed = true;
                }
            }
            __syncwarp();                                              // rows consumed before the next chunk
        }
        if (flushed) {
    #pragma unroll
            for (int x = 0; x < L; ++x) { two_sum_add(hi[x], lo[x], acc[x]); F[x] = __ldg(uf + x) + (hi[x] + lo[x]); }
        } else {
    #pragma unroll
            for (int x = 0; x < L; ++x) F[x] = __ldg(uf + x) + acc[x];
        }
    }
    if (POT) {
        float* pv = a.pot + (int64_t)v * L * a.C + c;
#pragma unroll
        for (int x = 0; x < L; ++x) pv[(int64_t)x * a.C] = F[x];
        return;
    }
    float* lp = a.logp ? a.logp + ((int64_t)c * a.N + v) * L : nullptr;
    xout[g] = (uint8_t)draw_label<L>(F, v, c, sweep, a.rk, PH_PRIMAL, lp, a.ctl, a.lpv ? a.lpv + g : nullptr);
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}

// One-batch warp-per-site form with two chains per lane, for tables of one
// dual word and sites of at most KB incidences: lane l holds chains 2 l and
// 2 l + 1 of its warp's 64, so one 8-byte load brings both chains' dual words
// of an incidence, and every tau row, incidence code and unary row serves both.
// Small tables are bound by this bookkeeping and the label draws, not by the
// additions: 48^3, 64 chains, L = 2: 73 us (100 us with one chain per lane).
// Keeps k_primal's order of additions.
struct PrimalSite {
    static constexpr int KB = 8;
    static constexpr int WARPS = 4;                            // 128 threads
};

template <int L, int LAYOUT, bool POT = false>
__global__ void __launch_bounds__(128, L <= 6 ? 8 : 6) k_primal_site(SweepArgs a, FastDiv fdG) {
    using E = Ent<L, LAYOUT>;
    constexpr uint32_t FULL = 0xFFFFFFFFu;
    constexpr int MP = E::MP, KB = PrimalSite::KB;
    static_assert(E::W == 1 && MP <= 128, "one dual word; a tau row in one 16-byte copy per lane");
    __shared__ __align__(16) float s_tau[PrimalSite::WARPS][KB][MP];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t groups = fdG.d, un = blockIdx.x * PrimalSite::WARPS + warp;
    if (un >= (uint32_t)a.N * groups) return;                     // whole warps only
    const uint32_t v = fdG.div(un), c = (un - v * groups) * 64 + lane * 2;
    const int64_t p0 = a.inc_ptr[v];
    const int deg = (int)(a.inc_ptr[v + 1] - p0);
    const uint32_t code_l = lane < deg ? (uint32_t)__ldg(&a.inc[p0 + lane].x) : 0u;
    const uint32_t sweep = (uint32_t)a.ctl->sweep;
    uint8_t* xout = a.x + (size_t)((sweep + 1) & 1) * a.N * a.C;
    const uint32_t* const th0 = a.theta + c;
    const uint32_t st = (uint32_t)__cvta_generic_to_shared(&s_tau[warp][0][0]) + lane * 16;
    uint32_t bits[KB][2][1];
#pragma unroll
    for (int u = 0; u < KB; ++u) {
        if (u < deg) {
            const uint32_t e = __shfl_sync(FULL, code_l, u) >> 1;
            const uint2 q = __ldcs(reinterpret_cast<const uint2*>(th0 + (uint64_t)e * (uint32_t)a.C));
            bits[u][0][0] = q.x;
            bits[u][1][0] = q.y;
            if (lane * 4 < MP)
                cp_async16(st + u * MP * 4, reinterpret_cast<const uint8_t*>(a.tau) + (uint64_t)e * (MP * 4) + lane * 16);
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const float* uf = a.utf + (int64_t)v * L;
    float ut[L];
    if constexpr (L % 4 == 0) {
#pragma unroll
        for (int x = 0; x < L; x += 4) {
            const float4 q = __ldg(reinterpret_cast<const float4*>(uf + x));
            ut[x] = q.x; ut[x + 1] = q.y; ut[x + 2] = q.z; ut[x + 3] = q.w;
        }
    } else {
#pragma unroll
        for (int x = 0; x < L; ++x) ut[x] = __ldg(uf + x);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();
    float acc[2][L];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int x = 0; x < L; ++x) acc[h][x] = 0.0f;
#pragma unroll
    for (int u = 0; u < KB; ++u) {
        if (u >= deg) break;
        const int side = (int)(__shfl_sync(FULL, code_l, u) & 1u);
        add_side_chains<L, LAYOUT, false, 2>(bits[u], &s_tau[warp][u][0], side, acc);
    }
    const int64_t g = (int64_t)v * a.C + c;
    uint32_t out = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float F[L];
#pragma unroll
        for (int x = 0; x < L; ++x) F[x] = ut[x] + acc[h][x];
        if (POT) {
            float* pv = a.pot + (int64_t)v * L * a.C + c + h;
#pragma unroll
            for (int x = 0; x < L; ++x) pv[(int64_t)x * a.C] = F[x];
        } else {
            float* lp = a.logp ? a.logp + ((int64_t)(c + h) * a.N + v) * L : nullptr;
            out |= (uint32_t)draw_label<L>(F, v, c + h, sweep, a.rk, PH_PRIMAL, lp, a.ctl, a.lpv ? a.lpv + g + h : nullptr) << (8 * h);
        }
    }
    if (!POT) *reinterpret_cast<uint16_t*>(xout + g) = (uint16_t)out;
}

// Warp-per-site form with its loads in a pipeline, for sites of at most `kb`
// incidences (every lattice) and 32 CH chains per warp.  A persistent warp
// walks its (site, chain group) units; the theta rows and tau rows of the next
// unit's incidences and its unary row are on their way into the other half of
// the warp's shared-memory buffer (16-byte asynchronous copies) while the
// current unit is summed, the incidence codes of the unit after that are in a
// register and the incidence range of the next one too, so no dependent load
// is waited for.  CH = 2 chains per lane share every tau load and every
// incidence's bookkeeping.  Keeps k_primal's order of additions.
// Bound by instruction issue (73 % of the issue slots, 20 warps per SM): 128^3,
// L = 8, 64 chains: 760 instructions per 32 site updates (968 in the form that
// loaded a site's incidences when it came to it), 3.54 ms per sweep (4.35 ms).
template <int L, int LAYOUT, int CH>
struct PrimalPipe {
    using E = Ent<L, LAYOUT>;
    static constexpr int WARPS = 4;                            // 128 threads
    static constexpr int TH = 32 * CH * E::W * 4;              // bytes of a theta row (32 CH chains)
    static constexpr int TAU = E::MP * 4;                      // bytes of a tau row
    static constexpr int UT = 64;                              // bytes kept for the unary row
    static constexpr int BLOCKS = L <= 8 ? (CH == 2 ? 5 : 8) : 4;   // blocks per SM the registers allow
    __host__ __device__ static constexpr int stage(int kb) { return kb * (TH + TAU) + UT; }
    __host__ __device__ static constexpr int smem(int kb) { return WARPS * 2 * stage(kb); }
};

template <int L, int LAYOUT, int CH, bool POT = false>
__global__ void __launch_bounds__(128, PrimalPipe<L, LAYOUT, CH>::BLOCKS) k_primal_pipe(SweepArgs a, int kb, FastDiv fdG) {
    using E = Ent<L, LAYOUT>;
    using P = PrimalPipe<L, LAYOUT, CH>;
    constexpr uint32_t FULL = 0xFFFFFFFFu;
    constexpr int W = E::W;
    extern __shared__ __align__(16) uint8_t s_pipe[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t nw = gridDim.x * P::WARPS;
    const uint32_t groups = fdG.d, units = (uint32_t)a.N * groups;       // below 2^27: N C < 2^32 (host)
    const uint32_t first = blockIdx.x * P::WARPS + warp;
    if (first >= units) return;
    uint8_t* buf = s_pipe + (size_t)warp * 2 * P::stage(kb);
    const uint32_t sbuf = (uint32_t)__cvta_generic_to_shared(buf) + lane * 16;
    const uint32_t sweep = (uint32_t)a.ctl->sweep;
    uint8_t* xout = a.x + (size_t)((sweep + 1) & 1) * a.N * a.C;
    const uint8_t* const theta_l = reinterpret_cast<const uint8_t*>(a.theta) + lane * 16;
    const uint8_t* const tau_l = reinterpret_cast<const uint8_t*>(a.tau) + lane * 16;
    const uint32_t theta_edge = (uint32_t)a.C * (W * 4);

    auto range = [&](uint32_t un, int64_t& p, int& deg) {
        deg = 0;
        if (un < units) {
            const uint32_t v = fdG.div(un);
            p = a.inc_ptr[v];
            deg = (int)(a.inc_ptr[v + 1] - p);
        }
    };
    auto codes = [&](int64_t p, int deg) { return lane < deg ? __ldg(&a.inc[p + lane].x) : -1; };
    // copies of unit `un`, whose incidence codes the lanes hold, into buffer half `half`
    auto load = [&](uint32_t un, int code, int half) {
        if (un < units) {
            const uint32_t v = fdG.div(un), grp = un - v * groups;
            const int deg = __popc(__ballot_sync(FULL, code >= 0));
            const uint32_t eu = (uint32_t)code >> 1;
            const uint8_t* th = theta_l + grp * P::TH;
            uint32_t dst = sbuf + half * P::stage(kb), dtau = dst + kb * P::TH;
#pragma unroll 2
            for (int u = 0; u < deg; ++u, dst += P::TH, dtau += P::TAU) {
                const uint32_t e = __shfl_sync(FULL, eu, u);
                const uint8_t* src = th + (uint64_t)e * theta_edge;
                const uint8_t* tsrc = tau_l + (uint64_t)e * P::TAU;
#pragma unroll
                for (int o = 0; o < P::TH; o += 512)
                    if (o + 512 <= P::TH || o + lane * 16 < P::TH) cp_async16(dst + o, src + o);
#pragma unroll
                for (int o = 0; o < P::TAU; o += 512)
                    if (o + 512 <= P::TAU || o + lane * 16 < P::TAU) cp_async16(dtau + o, tsrc + o);
            }
            if (lane < L) cp_async4(sbuf - lane * 12 + half * P::stage(kb) + kb * (P::TH + P::TAU), a.utf + (int64_t)v * L + lane);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    int64_t p = 0;
    int deg;
    range(first, p, deg);
    int code = codes(p, deg);
    load(first, code, 0);
    range(first + nw, p, deg);
    int code1 = codes(p, deg);
    range(first + 2 * nw, p, deg);
    int half = 0;
    for (uint32_t un = first; un < units; un += nw, half ^= 1) {
        load(un + nw, code1, half ^ 1);
        const int code2 = codes(p, deg);
        range(un + 3 * nw, p, deg);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();
        const uint8_t* st = buf + (size_t)half * P::stage(kb);
        const int n = __popc(__ballot_sync(FULL, code >= 0));
        float acc[CH][L];
#pragma unroll
        for (int h = 0; h < CH; ++h)
#pragma unroll
            for (int x = 0; x < L; ++x) acc[h][x] = 0.0f;
        for (int u = 0; u < n; ++u) {
            const int side = __shfl_sync(FULL, code, u) & 1;
            uint32_t bits[CH][W];
#pragma unroll
            for (int h = 0; h < CH; ++h) {
                const uint32_t* th = reinterpret_cast<const uint32_t*>(st + u * P::TH) + (h * 32 + lane) * W;
                if constexpr (W % 4 == 0) {
#pragma unroll
                    for (int w = 0; w < W; w += 4) {
                        const uint4 q = *reinterpret_cast<const uint4*>(th + w);
                        bits[h][w] = q.x; bits[h][w + 1] = q.y; bits[h][w + 2] = q.z; bits[h][w + 3] = q.w;
                    }
                } else if constexpr (W % 2 == 0) {
#pragma unroll
                    for (int w = 0; w < W; w += 2) {
                        const uint2 q = *reinterpret_cast<const uint2*>(th + w);
                        bits[h][w] = q.x; bits[h][w + 1] = q.y;
                    }
                } else {
#pragma unroll
                    for (int w = 0; w < W; ++w) bits[h][w] = th[w];
                }
            }
            add_side_chains<L, LAYOUT, false, CH>(bits, reinterpret_cast<const float*>(st + kb * P::TH + u * P::TAU),
                                                  side, acc);
        }
        const uint32_t v = fdG.div(un), c0 = (un - v * groups) * 32 * CH + lane;
        const float* ut = reinterpret_cast<const float*>(st + kb * (P::TH + P::TAU));
#pragma unroll
        for (int h = 0; h < CH; ++h) {
            const uint32_t c = c0 + 32 * h;
            float F[L];
#pragma unroll
            for (int x = 0; x < L; ++x) F[x] = ut[x] + acc[h][x];
            if (POT) {
                float* pv = a.pot + (int64_t)v * L * a.C + c;
#pragma unroll
                for (int x = 0; x < L; ++x) pv[(int64_t)x * a.C] = F[x];
            } else {
                const int64_t g = (int64_t)v * a.C + c;
                float* lp = a.logp ? a.logp + ((int64_t)c * a.N + v) * L : nullptr;
                xout[g] = (uint8_t)draw_label<L>(F, v, c, sweep, a.rk, PH_PRIMAL, lp, a.ctl, a.lpv ? a.lpv + g : nullptr);
            }
        }
        __syncwarp();                                                    // this half is free for the unit after the next
        code = code1;
        code1 = code2;
    }
}

// Label-per-lane form for models that leave the thread form too few warps: G
// lanes (a power of two, at least L) share a (site, chain) item and lane x sums
// label x's field -- the entries of row x of an incidence where the site is the
// source, of column x where it is the destination, in entry order, two-sum
// flush every 32 incidences: the additions of k_primal into that label, bit for
// bit.  The first lane gathers the fields and draws.  A lane has L - 1 entries of
// an incidence instead of (L - 1)^2 and their weights are loaded side by side:
// 25,611 sites of degree 15, L = 8, one chain: 83 -> 34 us.
template <int L>
struct LabelLanes {
    static constexpr int G = L <= 8 ? 8 : 16;
};

template <int L, int LAYOUT, bool POT = false>
__global__ void __launch_bounds__(256) k_primal_labels(SweepArgs a) {
    using E = Ent<L, LAYOUT>;
    constexpr int G = LabelLanes<L>::G, W = E::W, MP = E::MP;
    constexpr int R = L - 1;                               // entries of a label per incidence
    static_assert(W <= 2 && LAYOUT == MRF_LAYOUT_PIVOT, "full tables of at most 64 entries");
    const uint64_t id = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    const uint64_t g64 = id / G;
    const int x = (int)(id % G);
    const bool item = g64 < (uint64_t)a.N * a.C;
    const uint32_t g = item ? (uint32_t)g64 : 0u;
    const uint32_t v = a.fdC.div(g), c = g - v * (uint32_t)a.C;
    const uint32_t sweep = (uint32_t)a.ctl->sweep;
    const int64_t p0 = a.inc_ptr[v];
    int64_t p1 = a.inc_ptr[v + 1];
    const bool active = item && p1 - p0 <= a.hub_deg;             // else k_primal_hub's
    const bool has = active && x < L && x > 0;                    // label 0 has no entries
    if (!has) p1 = p0;
    float acc = 0.0f, hi = 0.0f, lo = 0.0f;
    int chunk = 0;
    bool flushed = false;
    constexpr int B = 4;                                   // incidences whose words and weights are loaded together
    for (int64_t base = p0; base < p1; base += B) {
        int code[B];
        uint64_t bits[B];
#pragma unroll
        for (int u = 0; u < B; ++u) code[u] = base + u < p1 ? __ldg(&a.inc[base + u].x) : -1;
#pragma unroll
        for (int u = 0; u < B; ++u) {
            bits[u] = 0;
            if (code[u] >= 0) {
                const uint32_t* th = a.theta + ((int64_t)(code[u] >> 1) * a.C + c) * W;
                if constexpr (W == 2) {
                    const uint2 q = __ldg(reinterpret_cast<const uint2*>(th));
                    bits[u] = (uint64_t)q.y << 32 | q.x;
                } else {
                    bits[u] = __ldg(th);
                }
            }
        }
        float t[B][R];
        int first[B], step[B];
#pragma unroll
        for (int u = 0; u < B; ++u) {
            const bool dst = code[u] & 1;
            first[u] = dst ? x - 1 : (x - 1) * R;
            step[u] = dst ? R : 1;
            const float* tau = a.tau + (int64_t)(code[u] >= 0 ? code[u] >> 1 : 0) * MP;
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const float w = __ldg(tau + first[u] + i * step[u]);
                t[u][i] = dst ? fabsf(w) : w;
            }
        }
#pragma unroll
        for (int u = 0; u < B; ++u) {
            if (code[u] < 0) continue;
            const uint64_t b = bits[u] >> first[u];
#pragma unroll
            for (int i = 0; i < R; ++i)
                if ((b >> (i * step[u])) & 1u) acc += t[u][i];
            if (++chunk == 32) {
                two_sum_add(hi, lo, acc);
                acc = 0.0f;
                chunk = 0;
                flushed = true;
            }
        }
    }
    float f = 0.0f;
    if (active && x < L) {
        const float ut = __ldg(a.utf + (int64_t)v * L + x);
        // (an unflushed pair is zero: hi + lo = acc exactly)
        if (flushed) two_sum_add(hi, lo, acc);
        f = ut + (flushed ? hi + lo : acc);
        if (POT) a.pot[((int64_t)v * L + x) * a.C + c] = f;
    }
    if (POT) return;
    float F[L];
#pragma unroll
    for (int y = 0; y < L; ++y) F[y] = __shfl_sync(0xffffffffu, f, y, G);
    if (active && x == 0) {
        uint8_t* xout = a.x + (size_t)((sweep + 1) & 1) * a.N * a.C;
        float* lp = a.logp ? a.logp + ((int64_t)c * a.N + v) * L : nullptr;
        xout[g] = (uint8_t)draw_label<L>(F, v, c, sweep, a.rk, PH_PRIMAL, lp, a.ctl, a.lpv ? a.lpv + g : nullptr);
    }
}

// Sites of more than a.hub_deg incidences for the thread and warp forms above,
// which would sum such a site in one thread or warp while the rest of the GPU
// has finished (preferential attachment: a few sites of a thousand incidences
// among 50,000).  A CTA looks through its share of the sites (spread so that
// neighbouring hubs fall on different CTAs) and sums each hub with all its
// threads: CG = min(C, 32) chains (blockIdx.y: the groups of chains) by 512 / CG slices, a slice one run of 32
// incidences per round.  The forms above sum such a run from zero and then add
// it to the site's two-sum pair; here the runs are summed side by side and added
// to the pair in the same order, so the field is the same bit for bit.
// 50,000 sites, 5 edges per new site (largest degree 1,548), L = 4, 32 chains:
// potentials 355 -> 103 us; 10 chains 407 -> 84 us.
template <int L, int LAYOUT, bool POT>
__global__ void __launch_bounds__(512) k_primal_hub(SweepArgs a, int CG) {
    using E = Ent<L, LAYOUT>;
    constexpr int W = E::W, MAXH = 64;
    __shared__ float s_part[L][512];
    __shared__ int s_hub[MAXH];
    __shared__ int s_n;
    const int S = 512 / CG, lane = threadIdx.x % CG, slice = threadIdx.x / CG;
    const uint32_t sweep = (uint32_t)a.ctl->sweep;
    uint8_t* xout = a.x + (size_t)((sweep + 1) & 1) * a.N * a.C;
    for (int64_t v0 = blockIdx.x; v0 < a.N; v0 += (int64_t)gridDim.x * MAXH) {
        __syncthreads();
        if (threadIdx.x == 0) s_n = 0;
        __syncthreads();
        for (int i = threadIdx.x; i < MAXH; i += 512) {
            const int64_t v = v0 + (int64_t)i * gridDim.x;
            if (v < a.N && a.inc_ptr[v + 1] - a.inc_ptr[v] > a.hub_deg) s_hub[atomicAdd(&s_n, 1)] = (int)v;
        }
        __syncthreads();
        const int nh = s_n;
        for (int q = 0; q < nh; ++q) {
            const int v = s_hub[q];
            const int64_t p0 = a.inc_ptr[v];
            const int deg = (int)(a.inc_ptr[v + 1] - p0), runs = (deg + 31) / 32;
            for (int cb = (int)blockIdx.y * CG; cb < a.C; cb += CG * (int)gridDim.y) {
                const int c = cb + lane;
                float hi[L], lo[L], rest[L];
#pragma unroll
                for (int x = 0; x < L; ++x) { hi[x] = 0.0f; lo[x] = 0.0f; rest[x] = 0.0f; }
                for (int r0 = 0; r0 < runs; r0 += S) {
                    const int run = r0 + slice;
                    if (slice < S && c < a.C && run < runs) {
                        float acc[L];
#pragma unroll
                        for (int x = 0; x < L; ++x) acc[x] = 0.0f;
                        const int end = min(deg, run * 32 + 32);
                        constexpr int B = W <= 2 ? 4 : 2;  // incidences loaded together
                        for (int u0 = run * 32; u0 < end; u0 += B) {
                            int code[B];
                            uint32_t bits[B][W];
#pragma unroll
                            for (int u = 0; u < B; ++u) code[u] = u0 + u < end ? __ldg(&a.inc[p0 + u0 + u].x) : -1;
#pragma unroll
                            for (int u = 0; u < B; ++u) {
                                const uint32_t* th = a.theta + ((int64_t)(code[u] >> 1) * a.C + c) * W;
#pragma unroll
                                for (int w = 0; w < W; ++w) bits[u][w] = code[u] >= 0 ? __ldcs(th + w) : 0u;
                            }
#pragma unroll
                            for (int u = 0; u < B; ++u)
                                if (code[u] >= 0)
                                    add_side<L, LAYOUT>(bits[u], a.tau + (int64_t)(code[u] >> 1) * E::MP, code[u] & 1, acc);
                        }
#pragma unroll
                        for (int x = 0; x < L; ++x) s_part[x][threadIdx.x] = acc[x];
                    }
                    __syncthreads();
                    if (slice == 0 && c < a.C) {
                        for (int k = 0; k < S && r0 + k < runs; ++k) {
                            if ((r0 + k) * 32 + 32 <= deg) {
#pragma unroll
                                for (int x = 0; x < L; ++x) two_sum_add(hi[x], lo[x], s_part[x][k * CG + lane]);
                            } else {
#pragma unroll
                                for (int x = 0; x < L; ++x) rest[x] = s_part[x][k * CG + lane];
                            }
                        }
                    }
                    __syncthreads();
                }
                if (slice == 0 && c < a.C) {
                    float F[L];
                    const float* uf = a.utf + (int64_t)v * L;
#pragma unroll
                    for (int x = 0; x < L; ++x) { two_sum_add(hi[x], lo[x], rest[x]); F[x] = __ldg(uf + x) + (hi[x] + lo[x]); }
                    const int64_t g = (int64_t)v * a.C + c;
                    if (POT) {
                        float* pv = a.pot + (int64_t)v * L * a.C + c;
#pragma unroll
                        for (int x = 0; x < L; ++x) pv[(int64_t)x * a.C] = F[x];
                    } else {
                        float* lp = a.logp ? a.logp + ((int64_t)c * a.N + v) * L : nullptr;
                        xout[g] = (uint8_t)draw_label<L>(F, (uint32_t)v, (uint32_t)c, sweep, a.rk, PH_PRIMAL, lp, a.ctl,
                                                         a.lpv ? a.lpv + g : nullptr);
                    }
                }
            }
        }
    }
}

// CTA-per-site schedule of the plain primal step for high-degree sites: a CTA
// of 256 threads covers one site and CG = min(C, 32) chains; its CG x S threads
// (S = 256 / CG incidence slices) each sum a strided share of the incidence
// list for one chain, the S partial sums are combined in shared memory with
// the two-sum pair, and the first slice draws the labels.
template <int L, int LAYOUT>
__global__ void __launch_bounds__(256) k_primal_cta(SweepArgs a, int CG) {
    using E = Ent<L, LAYOUT>;
    __shared__ float red_hi[256][L];
    __shared__ float red_lo[256][L];
    const int S = 256 / CG;
    const int lane = threadIdx.x % CG, slice = threadIdx.x / CG;
    const int groups = (a.C + CG - 1) / CG;
    const uint32_t v = blockIdx.x / groups;
    const int c = (blockIdx.x % groups) * CG + lane;
    const bool active = slice < S && c < a.C;
    const uint32_t sweep = (uint32_t)a.ctl->sweep;
    float acc[L], hi[L], lo[L];
#pragma unroll
    for (int x = 0; x < L; ++x) { acc[x] = 0.0f; hi[x] = 0.0f; lo[x] = 0.0f; }
    if (active) {
        const int64_t p0 = a.inc_ptr[v], p1 = a.inc_ptr[v + 1];
        int chunk = 0;
        // B incidences of the slice per iteration, their records and theta words
        // loaded before any is added (same order of additions)
        // (8 for one word: 62 registers, 1.40 vs 1.12 ms at N = 4096; staging a site's records in
        // shared memory first: 1.14 ms, no gain)
        constexpr int B = E::W <= 2 ? 4 : 2;
        for (int64_t p = p0 + slice; p < p1; p += (int64_t)B * S) {
            int2 ic[B];
            uint32_t bits[B][E::W];
#pragma unroll
            for (int u = 0; u < B; ++u) ic[u] = p + (int64_t)u * S < p1 ? __ldg(&a.inc[p + (int64_t)u * S]) : make_int2(-1, 0);
#pragma unroll
            for (int u = 0; u < B; ++u) {
                const uint32_t* th = a.theta + ((int64_t)(ic[u].x >> 1) * a.C + c) * E::W;
#pragma unroll
                for (int w = 0; w < E::W; ++w) bits[u][w] = ic[u].x >= 0 ? __ldcs(th + w) : 0u;
            }
#pragma unroll
            for (int u = 0; u < B; ++u) {
                if (ic[u].x < 0) continue;
                add_side<L, LAYOUT>(bits[u], a.tau + (int64_t)(ic[u].x >> 1) * E::MP, ic[u].x & 1, acc);
                if (++chunk == 32) {
#pragma unroll
                    for (int x = 0; x < L; ++x) { two_sum_add(hi[x], lo[x], acc[x]); acc[x] = 0.0f; }
                    chunk = 0;
                }
            }
        }
#pragma unroll
        for (int x = 0; x < L; ++x) two_sum_add(hi[x], lo[x], acc[x]);
    }
#pragma unroll
    for (int x = 0; x < L; ++x) { red_hi[threadIdx.x][x] = hi[x]; red_lo[threadIdx.x][x] = lo[x]; }
    __syncthreads();
    if (slice == 0 && c < a.C) {
#pragma unroll
        for (int x = 0; x < L; ++x) {
            float h = 0.0f, l = 0.0f;
            for (int q = 0; q < S; ++q) {
                two_sum_add(h, l, red_hi[q * CG + lane][x]);
                l += red_lo[q * CG + lane][x];
            }
            hi[x] = h; lo[x] = l;
        }
        float F[L];
        const float* uf = a.utf + (int64_t)v * L;
#pragma unroll
        for (int x = 0; x < L; ++x) F[x] = __ldg(uf + x) + (hi[x] + lo[x]);
        uint8_t* xout = a.x + (size_t)((sweep + 1) & 1) * a.N * a.C;
        float* lp = a.logp ? a.logp + ((int64_t)c * a.N + v) * L : nullptr;
        xout[(int64_t)v * a.C + c] = (uint8_t)draw_label<L>(F, v, (uint32_t)c, sweep, a.rk, PH_PRIMAL, lp, a.ctl,
                                                            a.lpv ? a.lpv + (int64_t)v * a.C + c : nullptr);
    }
}

// ---------------------------------------------------------------------------- few chains, many entries

// Plain sweep for few chains (C <= 4) and tables with more than 16 entries,
// where a thread per (site, chain) would read every incident entry's weight
// row on its own.  After the dual step (k_dual), one warp per edge reads the
// edge's signed weights once (lane b: entries k = 32 g + b, coalesced) and,
// per chain, its dual bit words, and writes the edge's two partial fields:
// over the set bits, the row sums of the signed weights (source side, beta1)
// and the column sums of their magnitudes (destination side, beta2), each in
// entry order.  The primal step (k_primal_partial) then adds the partial
// fields of a site's incidences in incidence order (two-sum flush every 32,
// as k_primal) and draws the label.
template <int L, int LAYOUT>
__global__ void __launch_bounds__(256) k_edge_partial(SweepArgs a) {
    using E = Ent<L, LAYOUT>;
    constexpr int M = E::M, W = E::W, MP = E::MP;
    static_assert(M > 16 && L <= 16, "edge-partial form: more than 16 entries, at most 16 labels");
    __shared__ float s_t[8][W * 32];                       // weights of the set bits, per warp
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t e = blockIdx.x * 8ll + warp;
    if (e >= a.E || a.src[e] < 0) return;                  // whole warps; a free slot has no incidences
    const int C = a.C;
    float tv[W];
#pragma unroll
    for (int g = 0; g < W; ++g) {
        const int k = 32 * g + lane;
        tv[g] = k < M ? __ldg(a.tau + e * MP + k) : 0.0f;
    }
    for (int c = 0; c < C; ++c) {
        const uint32_t* th = a.theta + (e * C + c) * W;
        uint32_t bw[W];
        if constexpr (W % 4 == 0) {                        // the edge-chain's words in 16-byte loads
#pragma unroll
            for (int g = 0; g < W; g += 4) {
                const uint4 q = __ldcs(reinterpret_cast<const uint4*>(th + g));
                bw[g] = q.x; bw[g + 1] = q.y; bw[g + 2] = q.z; bw[g + 3] = q.w;
            }
        } else {
#pragma unroll
            for (int g = 0; g < W; ++g) bw[g] = __ldcs(th + g);
        }
#pragma unroll
        for (int g = 0; g < W; ++g) s_t[warp][32 * g + lane] = ((bw[g] >> lane) & 1u) ? tv[g] : 0.0f;
        __syncwarp();
        float* pe = a.part + ((e * C + c) * 2) * L;
        if (lane < L) {                                    // row `lane`: source side
            float sum = 0.0f;
            if (LAYOUT == MRF_LAYOUT_PIVOT) {
                if (lane >= 1)
#pragma unroll
                    for (int jj = 1; jj < L; ++jj) sum += s_t[warp][(lane - 1) * (L - 1) + (jj - 1)];
            } else {
                sum = s_t[warp][lane];
            }
            pe[lane] = sum;
        } else if (lane >= 16 && lane < 16 + L) {          // column `lane - 16`: destination side
            const int x = lane - 16;
            float sum = 0.0f;
            if (LAYOUT == MRF_LAYOUT_PIVOT) {
                if (x >= 1)
#pragma unroll
                    for (int ii = 1; ii < L; ++ii) sum += fabsf(s_t[warp][(ii - 1) * (L - 1) + (x - 1)]);
            } else {
                sum = fabsf(s_t[warp][x]);
            }
            pe[L + x] = sum;
        }
        __syncwarp();
    }
}

template <int L>
__global__ void __launch_bounds__(256, 3) k_primal_partial(SweepArgs a) {
    const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;     // N * C < 2^32 (checked by the host)
    if (g >= (uint64_t)a.N * a.C) return;
    const uint32_t v = a.fdC.div(g), c = g - v * (uint32_t)a.C;
    const uint32_t sweep = (uint32_t)a.ctl->sweep;
    uint8_t* xout = a.x + (size_t)((sweep + 1) & 1) * a.N * a.C;
    float acc[L], hi[L], lo[L];
#pragma unroll
    for (int x = 0; x < L; ++x) { acc[x] = 0.0f; hi[x] = 0.0f; lo[x] = 0.0f; }
    const int64_t p0 = a.inc_ptr[v], p1 = a.inc_ptr[v + 1];
    int chunk = 0;
    bool flushed = false;
    constexpr int B = 4;                                   // incidence records loaded together
    for (int64_t base = p0; base < p1; base += B) {
        int code[B];
#pragma unroll
        for (int u = 0; u < B; ++u) code[u] = base + u < p1 ? __ldg(&a.inc[base + u]).x : -1;
#pragma unroll
        for (int u = 0; u < B; ++u) {
            if (code[u] < 0) continue;
            const float* pe = a.part + (((int64_t)(code[u] >> 1) * a.C + c) * 2 + (code[u] & 1)) * L;
            if constexpr (L % 4 == 0) {
#pragma unroll
                for (int x4 = 0; x4 < L / 4; ++x4) {
                    const float4 q = __ldcs(reinterpret_cast<const float4*>(pe) + x4);
                    acc[4 * x4] += q.x; acc[4 * x4 + 1] += q.y; acc[4 * x4 + 2] += q.z; acc[4 * x4 + 3] += q.w;
                }
            } else {
#pragma unroll
                for (int x = 0; x < L; ++x) acc[x] += __ldcs(pe + x);
            }
            if (++chunk == 32) {
#pragma unroll
                for (int x = 0; x < L; ++x) { two_sum_add(hi[x], lo[x], acc[x]); acc[x] = 0.0f; }
                chunk = 0;
                flushed = true;
            }
        }
    }
    float F[L];
    const float* uf = a.utf + (int64_t)v * L;
    if (flushed) {
#pragma unroll
        for (int x = 0; x < L; ++x) { two_sum_add(hi[x], lo[x], acc[x]); F[x] = __ldg(uf + x) + (hi[x] + lo[x]); }
    } else {
#pragma unroll
        for (int x = 0; x < L; ++x) F[x] = __ldg(uf + x) + acc[x];
    }
    float* lp = a.logp ? a.logp + ((int64_t)c * a.N + v) * L : nullptr;
    xout[g] = (uint8_t)draw_label<L>(F, v, c, sweep, a.rk, PH_PRIMAL, lp, a.ctl, a.lpv ? a.lpv + g : nullptr);
}

template <int L, int LAYOUT>
cudaError_t run_sweep_partial(const SweepArgs& a, int step, cudaStream_t s) {
    if constexpr (Ent<L, LAYOUT>::M > 16) {
        const int64_t n = (int64_t)a.N * a.C;
        if (step == 0 && a.E > 0) k_edge_partial<L, LAYOUT><<<(unsigned)((a.E + 7) / 8), 256, 0, s>>>(a);
        if (step == 1 && n > 0) k_primal_partial<L><<<(unsigned)((n + 255) / 256), 256, 0, s>>>(a);
        return cudaGetLastError();
    } else {
        return cudaErrorInvalidValue;
    }
}

// ---------------------------------------------------------------------------- small models

// Barrier of a thread-block cluster: what its threads wrote before is seen by
// its threads after (loads that may have been cached go to L2).
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ void cluster_barrier() { cluster_arrive(); cluster_wait(); }

// Dual words of one (edge, chain), written by a CTA of the cluster (L2).
template <int W>
__device__ __forceinline__ void load_words(const uint32_t* th, uint32_t (&bits)[W]) {
    if constexpr (W % 2 == 0) {
#pragma unroll
        for (int w = 0; w < W; w += 2) {
            const uint2 q = __ldcg(reinterpret_cast<const uint2*>(th + w));
            bits[w] = q.x;
            bits[w + 1] = q.y;
        }
    } else {
#pragma unroll
        for (int w = 0; w < W; ++w) bits[w] = __ldcg(th + w);
    }
}

// Additions of one incidence in the one-launch kernels: grouped (add_side), or entry
// by entry where that is faster (PIVOT, single over grouped, median of sites of
// degree 24 and more: L = 5 1.02, L = 6 0.92 in clusters and 1.07 in one CTA, L = 7
// 0.83 and 0.90, L = 8 0.80 to 0.89, L = 10 0.83, L = 16 0.82).
template <int L, int LAYOUT, bool CLUSTER>
__device__ __forceinline__ void add_side_small(const uint32_t (&bits)[Ent<L, LAYOUT>::W], const float* __restrict__ tau_e,
                                               int side, float (&acc)[L]) {
    if constexpr (LAYOUT == MRF_LAYOUT_PIVOT && L >= (CLUSTER ? 6 : 7)) add_side_single<L, LAYOUT>(bits, tau_e, side, acc);
    else add_side<L, LAYOUT>(bits, tau_e, side, acc);
}

// n_sweeps whole plain sweeps of a small model in one launch (sizes where
// launches and latency, not work, set the time).  Chains are independent, so
// a cluster of CTAs takes nc chains and no cluster waits for another; within
// it the items of a half-step are spread over all its threads, labels and
// dual bits go through L2, and the half-steps are separated by cluster
// barriers only.  Counts are reductions to memory from the label draw.  The
// draws and the order of every addition are those of k_dual / k_primal, so
// the chain is the same bit for bit.  The sweep index is read from device
// memory by every thread and advanced by the last cluster to finish.
// Bound by latency (two barriers and their dependent L2 round trips).  50 x 50
// Ising grid, 10 chains, 10 sweeps: 990 us in one CTA with all chains, 62 us here.
// CLUSTER = false: one CTA per group of chains, labels through its L1 and dual
// words in shared memory (no barrier's acquire drops the lines of its tables
// either); the words of the last sweep are stored.  Up to 10 labels 1,024
// threads, whose 64 registers hold the sums of 512 threads' 128 nearly as well:
// 512 threads take 1.1 to 1.4 times as long on 512 to 5,120 items, from L = 11
// on 0.9 times.
template <int L, int LAYOUT, bool CLUSTER>
__global__ void __launch_bounds__(CLUSTER ? 512 : small_one_cta_threads(L)) k_sweep_small(SweepArgs a, int n_sweeps, FastDiv fdn) {
    using E = Ent<L, LAYOUT>;
    constexpr int W = E::W;
    extern __shared__ __align__(16) uint32_t s_theta[];    // one CTA: [E][nc][W]
    uint32_t rank = 0, size = 1;
    if (CLUSTER) {
        asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
        asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(size));
    }
    auto label = [](const uint8_t* p) -> int { return CLUSTER ? __ldcg(p) : *p; };
    auto barrier = [] { if (CLUSTER) cluster_barrier(); else __syncthreads(); };
    const uint32_t nc = fdn.d, cluster = blockIdx.x / size;
    const uint32_t c0 = cluster * nc;
    const uint32_t tid = rank * blockDim.x + threadIdx.x, T = size * blockDim.x;
    const uint32_t ne = (uint32_t)a.E * nc, nv = (uint32_t)a.N * nc, C = (uint32_t)a.C;
    uint32_t sweep = (uint32_t)a.ctl->sweep;
    const unsigned long long count_from = a.ctl->count_from;
    for (int it = 0; it < n_sweeps; ++it, ++sweep) {
        const uint8_t* xin = a.x + (size_t)(sweep & 1) * a.N * a.C;
        uint8_t* xout = a.x + (size_t)((sweep + 1) & 1) * a.N * a.C;
        for (uint32_t i = tid; i < ne; i += T) {
            const uint32_t e = fdn.div(i), c = c0 + (i - e * nc);
            if (c >= C) continue;
            uint32_t bits[W];
            const int s = a.src[e];
            if (s >= 0) {
                const int t = a.dst[e];
                dual_bits<L, LAYOUT>(e, c, label(xin + (int64_t)s * C + c), label(xin + (int64_t)t * C + c),
                                     a.tpl + (int64_t)e * E::PW, a.thr + (int64_t)e * E::M, sweep, a.rk, bits);
            } else {
#pragma unroll
                for (int w = 0; w < W; ++w) bits[w] = 0;
            }
            uint32_t* out = a.theta + ((int64_t)e * C + c) * W;
            if (CLUSTER || it + 1 == n_sweeps) {
#pragma unroll
                for (int w = 0; w < W; ++w) out[w] = bits[w];
            }
            if (!CLUSTER) {
#pragma unroll
                for (int w = 0; w < W; ++w) s_theta[i * W + w] = bits[w];
            }
        }
        barrier();
        for (uint32_t i = tid; i < nv; i += T) {
            const uint32_t v = fdn.div(i), c = c0 + (i - v * nc);
            if (c >= C) continue;
            float acc[L], hi[L], lo[L];
#pragma unroll
            for (int x = 0; x < L; ++x) { acc[x] = 0.0f; hi[x] = 0.0f; lo[x] = 0.0f; }
            int chunk = 0;
            bool flushed = false;
            const int64_t p0 = a.inc_ptr[v], p1 = a.inc_ptr[v + 1];
            constexpr int B = W <= 2 ? 4 : 2;              // incidences whose dual words are loaded together
            for (int64_t base = p0; base < p1; base += B) {
                int code[B];
                uint32_t bits[B][W];
#pragma unroll
                for (int u = 0; u < B; ++u) code[u] = base + u < p1 ? __ldg(&a.inc[base + u].x) : -1;
#pragma unroll
                for (int u = 0; u < B; ++u) {
                    if (code[u] < 0) continue;
                    if (CLUSTER) load_words<W>(a.theta + ((int64_t)(code[u] >> 1) * C + c) * W, bits[u]);
                    else {
                        const uint32_t* th = s_theta + ((uint32_t)(code[u] >> 1) * nc + (c - c0)) * W;
#pragma unroll
                        for (int w = 0; w < W; ++w) bits[u][w] = th[w];
                    }
                }
#pragma unroll
                for (int u = 0; u < B; ++u) {
                    if (code[u] < 0) continue;
                    add_side_small<L, LAYOUT, CLUSTER>(bits[u], a.tau + (int64_t)(code[u] >> 1) * E::MP, code[u] & 1, acc);
                    if (++chunk == 32) {
#pragma unroll
                        for (int x = 0; x < L; ++x) { two_sum_add(hi[x], lo[x], acc[x]); acc[x] = 0.0f; }
                        chunk = 0;
                        flushed = true;
                    }
                }
            }
            float F[L];
            const float* uf = a.utf + (int64_t)v * L;
            if (flushed) {
#pragma unroll
                for (int x = 0; x < L; ++x) { two_sum_add(hi[x], lo[x], acc[x]); F[x] = __ldg(uf + x) + (hi[x] + lo[x]); }
            } else {
#pragma unroll
                for (int x = 0; x < L; ++x) F[x] = __ldg(uf + x) + acc[x];
            }
            float* lp = a.logp ? a.logp + ((int64_t)c * a.N + v) * L : nullptr;
            const int lab = draw_label<L>(F, v, c, sweep, a.rk, PH_PRIMAL, lp, a.ctl);
            xout[(int64_t)v * C + c] = (uint8_t)lab;
            if (sweep >= count_from) atomicAdd(a.counts + (int64_t)v * L + lab, 1u);
        }
        barrier();
    }
    // after the last barrier every thread of the cluster has read the index
    if (rank == 0 && threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&a.ctl->done, 1u) + 1u == gridDim.x / size) {
            a.ctl->done = 0u;
            a.ctl->sweep = sweep;
        }
    }
}

// The same for models small enough that every thread of a cluster owns at
// most one (edge, chain) and one (site, chain) item: everything the sweeps read
// stays on the SMs.  Every CTA keeps all labels of the cluster's chains, and
// the dual words of its own sites' incidences at their (edge, chain) place; a
// label is stored into every CTA's copy and a dual word into the copies of the
// two endpoints' owners (distributed shared memory), so that all loads of a
// half-step are local and its only wait is the barrier.  The plane and
// threshold words of a thread's edge and the weights of its site's first
// incidences are staged in shared memory, the edge's endpoints and those
// incidences' codes in registers (a barrier's acquire drops the L1 lines, so a
// table word read from memory would be an L2 round trip in every sweep), and
// the random words of the next half-step are drawn between a barrier's arrival
// and its wait.  Bound by the latency of the two barriers and of the dual ->
// label -> dual chain: 32 x 32 Ising grid, one chain: 1.9 us per sweep (4.9 us in
// one CTA; 4.6 us in k_sweep_small); 50 x 50, 10 chains: 3.4 us (99 us).
template <int L, int LAYOUT>
struct SmallResident {
    using E = Ent<L, LAYOUT>;
    static constexpr int KT = small_row_incidences(E::M);
    static constexpr int TAU = small_row_tau(E::M);
    static constexpr int ROW = small_row_words(E::M);
};

__device__ __forceinline__ uint32_t cluster_address(uint32_t shared_address, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0,%1,%2;" : "=r"(r) : "r"(shared_address), "r"(rank));
    return r;
}

template <int L, int LAYOUT>
__global__ void __launch_bounds__(640) k_sweep_resident(SweepArgs a, int n_sweeps, FastDiv fdn) {
    using E = Ent<L, LAYOUT>;
    using S = SmallResident<L, LAYOUT>;
    constexpr int W = E::W, KI = 4;                        // incidences kept in registers
    extern __shared__ __align__(16) uint8_t s_small[];
    uint32_t rank, size;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(size));
    const uint32_t nc = fdn.d, c0 = blockIdx.x / size * nc, C = (uint32_t)a.C;
    const uint32_t i = rank * blockDim.x + threadIdx.x;    // this thread's edge item and site item
    const uint32_t ne = (uint32_t)a.E * nc, nv = (uint32_t)a.N * nc;
    const uint32_t lab_bytes = (nv + 15u) / 16u * 16u;
    uint8_t* s_lab = s_small;                              // [2][N][nc]
    uint32_t* s_th = reinterpret_cast<uint32_t*>(s_small + 2 * lab_bytes);     // [E][nc][W]
    uint32_t* s_row = s_th + (ne * W + 3u) / 4u * 4u + threadIdx.x * S::ROW;   // this thread's table row
    const uint32_t lab_addr = (uint32_t)__cvta_generic_to_shared(s_lab);
    const uint32_t th_addr = (uint32_t)__cvta_generic_to_shared(s_th);
    uint32_t sweep = (uint32_t)a.ctl->sweep;
    const unsigned long long count_from = a.ctl->count_from;
    const uint8_t* x0 = a.x + (size_t)(sweep & 1) * a.N * a.C;
    for (uint32_t j = threadIdx.x; j < nv; j += blockDim.x) {
        const uint32_t v = fdn.div(j), c = c0 + (j - v * nc);
        s_lab[(sweep & 1) * lab_bytes + j] = c < C ? x0[(int64_t)v * C + c] : 0;
    }
    // edge item
    const uint32_t e = fdn.div(i), ec = c0 + (i - e * nc);
    const bool edge_item = i < ne && ec < C, has_edge = edge_item && a.src[e] >= 0;
    uint32_t ls = 0, lt = 0, th_s = 0, th_t = 0;           // label places of the endpoints, dual words in their owners' copies
    if (has_edge) {
        ls = (uint32_t)a.src[e] * nc + (ec - c0);
        lt = (uint32_t)a.dst[e] * nc + (ec - c0);
        th_s = cluster_address(th_addr + i * W * 4, ls / blockDim.x);
        th_t = cluster_address(th_addr + i * W * 4, lt / blockDim.x);
        for (int k = 0; k < E::PW; ++k) s_row[k] = __ldg(a.tpl + (int64_t)e * E::PW + k);
        for (int k = 0; k < E::M; ++k) s_row[E::PW + k] = __ldg(a.thr + (int64_t)e * E::M + k);
    }
    // site item
    const uint32_t v = fdn.div(i), vc = c0 + (i - v * nc);
    const bool has_site = i < nv && vc < C;
    int64_t p0 = 0;
    int deg = 0;
    int code[KI];
    if (has_site) { p0 = a.inc_ptr[v]; deg = (int)(a.inc_ptr[v + 1] - p0); }
#pragma unroll
    for (int u = 0; u < KI; ++u) code[u] = u < deg ? __ldg(&a.inc[p0 + u].x) : -1;
    float ut[L];
#pragma unroll
    for (int x = 0; x < L; ++x) ut[x] = has_site ? __ldg(a.utf + (int64_t)v * L + x) : 0.0f;
    if constexpr (S::KT > 0) {
#pragma unroll
        for (int u = 0; u < S::KT; ++u)
            if (code[u] >= 0)
                for (int k = 0; k < E::MP; ++k)
                    s_row[S::TAU + u * E::MP + k] = __float_as_uint(__ldg(a.tau + (int64_t)(code[u] >> 1) * E::MP + k));
    }
    int lab = 0;
    auto arrive = [&] { if (size > 1) cluster_arrive(); };
    auto wait = [&] { if (size > 1) cluster_wait(); else __syncthreads(); };
    arrive();
    uint4 R[DualWords<L, LAYOUT>::N];
    if (has_edge) draw_dual_words<L, LAYOUT>(e, ec, sweep, a.rk, R);
    wait();                                                // labels in place; every CTA of the cluster has started
    for (int it = 0; it < n_sweeps; ++it, ++sweep) {
        if (has_edge) {
            uint32_t bits[W];
            const uint8_t* x = s_lab + (sweep & 1) * lab_bytes;
            dual_bits<L, LAYOUT, false>(e, ec, x[ls], x[lt], s_row, s_row + E::PW, sweep, a.rk, bits, R);
#pragma unroll
            for (int w = 0; w < W; ++w) {
                asm volatile("st.shared::cluster.u32 [%0],%1;" ::"r"(th_s + 4 * w), "r"(bits[w]) : "memory");
                if (th_t != th_s) asm volatile("st.shared::cluster.u32 [%0],%1;" ::"r"(th_t + 4 * w), "r"(bits[w]) : "memory");
            }
            if (it + 1 == n_sweeps) {                      // the last sweep's words are kept (mrf_debug_theta)
#pragma unroll
                for (int w = 0; w < W; ++w) a.theta[((int64_t)e * C + ec) * W + w] = bits[w];
            }
        } else if (edge_item && it + 1 == n_sweeps) {      // a free slot has none
#pragma unroll
            for (int w = 0; w < W; ++w) a.theta[((int64_t)e * C + ec) * W + w] = 0u;
        }
        // the random words of the next half-step are drawn while the barrier completes
        arrive();
        float uni = 0.0f;
        if (has_site) uni = uniform23(draw_rk(v, sweep, vc, PH_PRIMAL, 0, a.rk).x);
        wait();
        if (has_site) {
            float acc[L], hi[L], lo[L];
#pragma unroll
            for (int x = 0; x < L; ++x) { acc[x] = 0.0f; hi[x] = 0.0f; lo[x] = 0.0f; }
            int chunk = 0;
            bool flushed = false;
            auto words = [&](int cd, uint32_t (&bits)[W]) {
                const uint32_t* th = s_th + ((uint32_t)(cd >> 1) * nc + (vc - c0)) * W;
#pragma unroll
                for (int w = 0; w < W; ++w) bits[w] = th[w];
            };
            auto flush = [&] {
                if (++chunk == 32) {
#pragma unroll
                    for (int x = 0; x < L; ++x) { two_sum_add(hi[x], lo[x], acc[x]); acc[x] = 0.0f; }
                    chunk = 0;
                    flushed = true;
                }
            };
#pragma unroll
            for (int u = 0; u < KI; ++u) {
                if (code[u] < 0) continue;
                uint32_t bits[W];
                words(code[u], bits);
                if constexpr (S::KT > 0)
                    add_side<L, LAYOUT, false>(bits, reinterpret_cast<const float*>(s_row + S::TAU + u * E::MP), code[u] & 1, acc);
                else
                    add_side_small<L, LAYOUT, true>(bits, a.tau + (int64_t)(code[u] >> 1) * E::MP, code[u] & 1, acc);
                flush();
            }
            for (int u = KI; u < deg; ++u) {
                const int cd = __ldg(&a.inc[p0 + u].x);
                uint32_t bits[W];
                words(cd, bits);
                add_side_small<L, LAYOUT, true>(bits, a.tau + (int64_t)(cd >> 1) * E::MP, cd & 1, acc);
                flush();
            }
            float F[L];
            if (flushed) {
#pragma unroll
                for (int x = 0; x < L; ++x) { two_sum_add(hi[x], lo[x], acc[x]); F[x] = ut[x] + (hi[x] + lo[x]); }
            } else {
#pragma unroll
                for (int x = 0; x < L; ++x) F[x] = ut[x] + acc[x];
            }
            float* lp = a.logp ? a.logp + ((int64_t)vc * a.N + v) * L : nullptr;
            lab = draw_label_at<L>(F, uni, lp, a.ctl);
            const uint32_t place = lab_addr + ((sweep + 1) & 1) * lab_bytes + i;
            for (uint32_t r = 0; r < size; ++r)
                asm volatile("st.shared::cluster.u8 [%0],%1;" ::"r"(cluster_address(place, r)), "r"(lab) : "memory");
        }
        arrive();
        if (has_edge) draw_dual_words<L, LAYOUT>(e, ec, sweep + 1, a.rk, R);
        if (has_site && sweep >= count_from) atomicAdd(a.counts + (int64_t)v * L + lab, 1u);
        wait();
    }
    if (has_site) {                                        // the last labels and, in the other half, those before
        const int64_t g = (int64_t)v * C + vc;
        a.x[(size_t)(sweep & 1) * a.N * a.C + g] = (uint8_t)lab;
        a.x[(size_t)((sweep + 1) & 1) * a.N * a.C + g] = s_lab[((sweep + 1) & 1) * lab_bytes + i];
    }
    if (rank == 0 && threadIdx.x == 0) {                   // see k_sweep_small
        __threadfence();
        if (atomicAdd(&a.ctl->done, 1u) + 1u == gridDim.x / size) {
            a.ctl->done = 0u;
            a.ctl->sweep = sweep;
        }
    }
}

// ---------------------------------------------------------------------------- EM and mean field

// Theta-update of Section 5.3's primal-dual EM / mean field for one incident
// edge: with eta_y,k and eta_z,k the (expected) indicators of the entry's row
// and column labels, pi_k = sigmoid(q_k + beta1 eta_y + beta2 eta_z),
// q = -max(tau, 0), beta1 = tau, beta2 = |tau| (tau signed), and its beta pi
// is added to the field of this endpoint (row i_k on the source side, column
// j_k on the destination side).  ey / ez give eta for label a of the source /
// destination endpoint.
template <int L, int LAYOUT, typename EtaS, typename EtaT>
__device__ __forceinline__ void add_side_mean(const float* __restrict__ tau_e, int side, EtaS ey, EtaT ez,
                                              float (&acc)[L]) {
    using E = Ent<L, LAYOUT>;
    const float4* t4 = reinterpret_cast<const float4*>(tau_e);
#pragma unroll
    for (int k4 = 0; k4 < E::MP / 4; ++k4) {
        const float4 qv = __ldg(t4 + k4);
        const float tv[4] = {qv.x, qv.y, qv.z, qv.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int k = 4 * k4 + u;
            if (k >= E::M) continue;
            const float ts = tv[u], b2 = fabsf(ts);
            const float logit = -fmaxf(ts, 0.0f) + ts * ey(E::i(k)) + b2 * ez(E::j(k));
            const float pi = 1.0f / (1.0f + expf(-logit));
            if (side == 0) acc[E::i(k)] += ts * pi;
            else acc[E::j(k)] += b2 * pi;
        }
    }
}

// EM (local MAP): x' = argmax of the field of the expected duals given x.
template <int L, int LAYOUT>
__global__ void __launch_bounds__(256) k_em(SweepArgs a, const uint8_t* __restrict__ xin, uint8_t* __restrict__ xout) {
    const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= (uint64_t)a.N * a.C) return;
    const uint32_t v = a.fdC.div(g), c = g - v * (uint32_t)a.C;
    const int xv = xin[g];
    float acc[L];
#pragma unroll
    for (int x = 0; x < L; ++x) acc[x] = 0.0f;
    for (int64_t p = a.inc_ptr[v]; p < a.inc_ptr[v + 1]; ++p) {
        const int2 ic = __ldg(&a.inc[p]);
        const int side = ic.x & 1;
        const int xu = xin[(int64_t)ic.y * a.C + c];
        const int xs = side == 0 ? xv : xu, xt = side == 0 ? xu : xv;
        add_side_mean<L, LAYOUT>(a.tau + (int64_t)(ic.x >> 1) * Ent<L, LAYOUT>::MP, side,
                                 [&](int i) { return xs == i ? 1.0f : 0.0f; }, [&](int j) { return xt == j ? 1.0f : 0.0f; }, acc);
    }
    const float* uf = a.utf + (int64_t)v * L;
    int best = 0;
    float fb = __ldg(uf) + acc[0];
#pragma unroll
    for (int x = 1; x < L; ++x) {
        const float f = __ldg(uf + x) + acc[x];
        if (f > fb) { fb = f; best = x; }
    }
    xout[g] = (uint8_t)best;
}

// Blocked EM, potentials: F_v = u~_v + the beta pi of the expected duals of
// v's incident non-tree edges (the comb forest of the current block offset),
// written to a.pot ([N][L][C]) for the tree MAP.
template <int L, int LAYOUT>
__global__ void __launch_bounds__(256) k_em_pot(SweepArgs a, const uint8_t* __restrict__ xin) {
    const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= (uint64_t)a.N * a.C) return;
    const uint32_t v = a.fdC.div(g), c = g - v * (uint32_t)a.C;
    const int xv = xin[g];
    float acc[L];
#pragma unroll
    for (int x = 0; x < L; ++x) acc[x] = 0.0f;
    for (int64_t p = a.inc_ptr[v]; p < a.inc_ptr[v + 1]; ++p) {
        const int2 ic = __ldg(&a.inc[p]);
        if (is_tree_edge(a, (uint32_t)(ic.x >> 1))) continue;
        const int side = ic.x & 1;
        const int xu = xin[(int64_t)ic.y * a.C + c];
        const int xs = side == 0 ? xv : xu, xt = side == 0 ? xu : xv;
        add_side_mean<L, LAYOUT>(a.tau + (int64_t)(ic.x >> 1) * Ent<L, LAYOUT>::MP, side,
                                 [&](int i) { return xs == i ? 1.0f : 0.0f; }, [&](int j) { return xt == j ? 1.0f : 0.0f; }, acc);
    }
    const float* uf = a.utf + (int64_t)v * L;
    float* pv = a.pot + (int64_t)v * L * a.C + c;
#pragma unroll
    for (int x = 0; x < L; ++x) pv[(int64_t)x * a.C] = __ldg(uf + x) + acc[x];
}

// Mean field: q' = softmax of the field of the expected duals given the site
// marginals q ([N][L][C], chain innermost).
template <int L, int LAYOUT>
__global__ void __launch_bounds__(256) k_mf(SweepArgs a, const float* __restrict__ qin, float* __restrict__ qout) {
    const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= (uint64_t)a.N * a.C) return;
    const uint32_t v = a.fdC.div(g), c = g - v * (uint32_t)a.C;
    const int64_t C = a.C;
    float qv[L], acc[L];
#pragma unroll
    for (int x = 0; x < L; ++x) { qv[x] = qin[((int64_t)v * L + x) * C + c]; acc[x] = 0.0f; }
    for (int64_t p = a.inc_ptr[v]; p < a.inc_ptr[v + 1]; ++p) {
        const int2 ic = __ldg(&a.inc[p]);
        const int side = ic.x & 1;
        float qu[L];
#pragma unroll
        for (int x = 0; x < L; ++x) qu[x] = qin[((int64_t)ic.y * L + x) * C + c];
        const float* tau_e = a.tau + (int64_t)(ic.x >> 1) * Ent<L, LAYOUT>::MP;
        if (side == 0)
            add_side_mean<L, LAYOUT>(tau_e, 0, [&](int i) { return qv[i]; }, [&](int j) { return qu[j]; }, acc);
        else
            add_side_mean<L, LAYOUT>(tau_e, 1, [&](int i) { return qu[i]; }, [&](int j) { return qv[j]; }, acc);
    }
    const float* uf = a.utf + (int64_t)v * L;
    float F[L], mx = -INFINITY;
#pragma unroll
    for (int x = 0; x < L; ++x) { F[x] = __ldg(uf + x) + acc[x]; mx = fmaxf(mx, F[x]); }
    float s = 0.0f;
#pragma unroll
    for (int x = 0; x < L; ++x) { F[x] = expf(F[x] - mx); s += F[x]; }
    const float inv = 1.0f / s;
#pragma unroll
    for (int x = 0; x < L; ++x) qout[((int64_t)v * L + x) * C + c] = F[x] * inv;
}

// Blocked (tree) mean field, potentials: F_v = u~_v + the beta pi of the
// expected duals of v's incident non-forest edges given the site marginals q
// ([N][L][C]), written to a.pot for the forest's sum-product pass.
template <int L, int LAYOUT>
__global__ void __launch_bounds__(256) k_mf_pot(SweepArgs a, const float* __restrict__ qin) {
    const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= (uint64_t)a.N * a.C) return;
    const uint32_t v = a.fdC.div(g), c = g - v * (uint32_t)a.C;
    const int64_t C = a.C;
    float qv[L], acc[L];
#pragma unroll
    for (int x = 0; x < L; ++x) { qv[x] = qin[((int64_t)v * L + x) * C + c]; acc[x] = 0.0f; }
    for (int64_t p = a.inc_ptr[v]; p < a.inc_ptr[v + 1]; ++p) {
        const int2 ic = __ldg(&a.inc[p]);
        if (is_tree_edge(a, (uint32_t)(ic.x >> 1))) continue;
        const int side = ic.x & 1;
        float qu[L];
#pragma unroll
        for (int x = 0; x < L; ++x) qu[x] = qin[((int64_t)ic.y * L + x) * C + c];
        const float* tau_e = a.tau + (int64_t)(ic.x >> 1) * Ent<L, LAYOUT>::MP;
        if (side == 0)
            add_side_mean<L, LAYOUT>(tau_e, 0, [&](int i) { return qv[i]; }, [&](int j) { return qu[j]; }, acc);
        else
            add_side_mean<L, LAYOUT>(tau_e, 1, [&](int i) { return qu[i]; }, [&](int j) { return qv[j]; }, acc);
    }
    const float* uf = a.utf + (int64_t)v * L;
    float* pv = a.pot + (int64_t)v * L * C + c;
#pragma unroll
    for (int x = 0; x < L; ++x) pv[(int64_t)x * C] = __ldg(uf + x) + acc[x];
}

static inline unsigned blocks_for(int64_t n, int threads) { return (unsigned)((n + threads - 1) / threads); }

template <int L, int LAYOUT>
cudaError_t run_primal_cta(const SweepArgs& a, cudaStream_t s) {
    const int CG = a.C >= 32 ? 32 : a.C;
    const int64_t blocks = (int64_t)a.N * ((a.C + CG - 1) / CG);
    if (blocks > 0) k_primal_cta<L, LAYOUT><<<(unsigned)blocks, 256, 0, s>>>(a, CG);
    return cudaGetLastError();
}

template <int L, int LAYOUT>
cudaError_t run_dual(const SweepArgs& a, cudaStream_t s) {
    using T = DualTile<Ent<L, LAYOUT>::M, Ent<L, LAYOUT>::W>;
    const int64_t n = a.E * a.C;
    if (n <= 0) return cudaSuccess;
    // few chains and wide tables (two groups per warp): 128 registers and two blocks per SM; at 64
    // registers the 8-word form spills (224 B); with one chain on 25.2 M edges of L = 16 (the
    // 2,000-graph batch's largest class) it measured 5.14 vs 4.12 ms per sweep
    // groups per warp: NG where it leaves two blocks per SM (the variable bound costs up to 9 %), else the
    // largest power of two that leaves four blocks per SM (199,852 edges of L = 2, one chain: 16 groups per
    // warp are 49 blocks, 33 us; one group 9 us), two for two and three dual words, one for wide tables.
    // Other counts leave the last blocks to some SMs: 605,694 items of L = 6, one chain, in 1 / 2 / 3 / 4 / 8
    // groups 22.4 / 19.7 / 22.8 / 18.9 / 22.5 us; 226,688 items of L = 8, 32 chains, in 1 / 2 / 4 12.4 / 11.4 / 12.4;
    // 302,400 items in 3 13.8, in 4 12.3; 102,060 items of L = 14 in 1 / 2 27 / 24.
    const int64_t per_sm = Ent<L, LAYOUT>::W >= 4 ? 1 : (Ent<L, LAYOUT>::W >= 2 ? 2 : 4);
    int ng = T::NG;
    if (n < 32ll * T::WARPS * T::NG * 152 * 2)
        while (ng > 1 && n < 32ll * T::WARPS * ng * 152 * per_sm) ng /= 2;
    const unsigned blocks = blocks_for(n, 32 * ng * T::WARPS);
    if (a.C < 32 && T::NG <= 2) {
        if (ng < T::NG) k_dual<L, LAYOUT, (T::NG <= 2), true><<<blocks, 32 * T::WARPS, 0, s>>>(a, ng);
        else k_dual<L, LAYOUT, (T::NG <= 2)><<<blocks, 32 * T::WARPS, 0, s>>>(a, ng);
    } else if (ng < T::NG) {
        k_dual<L, LAYOUT, false, true><<<blocks, 32 * T::WARPS, 0, s>>>(a, ng);
    } else {
        k_dual<L, LAYOUT><<<blocks, 32 * T::WARPS, 0, s>>>(a, ng);
    }
    return cudaGetLastError();
}

// The pipelined warp form where its buffers leave at least two blocks per SM; false if not.
template <int L, int LAYOUT, int CH, bool POT>
bool try_primal_pipe(const SweepArgs& a, cudaStream_t s, cudaError_t& e) {
    using P = PrimalPipe<L, LAYOUT, CH>;
    if (a.C % (32 * CH) || a.max_deg >= 32) return false;
    const int kb = a.max_deg > 0 ? a.max_deg : 1, smem = P::smem(kb);
    if (smem > 100 * 1024) return false;
    if (smem > 48 * 1024) {
        e = cudaFuncSetAttribute(k_primal_pipe<L, LAYOUT, CH, POT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return true;
    }
    const int64_t blocks = ((int64_t)a.N * (a.C / (32 * CH)) + P::WARPS - 1) / P::WARPS;
    const int64_t resident = 152 * std::min<int64_t>(P::BLOCKS, 227 * 1024 / (smem + 1024));
    k_primal_pipe<L, LAYOUT, CH, POT><<<(unsigned)std::min(blocks, resident), 32 * P::WARPS, smem, s>>>(
        a, kb, FastDiv::make((uint32_t)(a.C / (32 * CH))));
    e = cudaGetLastError();
    return true;
}

// Chains a multiple of 32: the warp form by table width, degree and chains.
// us per launch on a 48^3 lattice (degree 6), measured one against the other:
//   one dual word, L <= 8, 64 chains: two chains per lane (k_primal_site) 73 / 98 / 114 / 127 for
//     L = 2 / 4 / 5 / 6 against 100 / 118 / 134 / 149 with one chain per lane (k_primal_warp);
//     with 16 labels on the diagonal 194 against 170, so one chain per lane there
//   PIVOT, L = 7 ... 12, 64 chains: pipelined, two chains per lane 165 / 191 / 252 / 284 / 366 / 409 (L = 8: 191)
//     against 189 / 215 / 268 / 310 / 506 / 546
//   PIVOT, L = 11 ... 14, 32 chains: pipelined, one chain per lane 199 / 221 / - / 329 against
//     260 / 282 / - / 375; for L <= 10 it is slower (L = 8: 135 against 115), L = 16 even (527 and 525)
template <int L, int LAYOUT, bool POT>
cudaError_t run_primal_warps(const SweepArgs& a, cudaStream_t s) {
    const int64_t n = (int64_t)a.N * a.C;
    cudaError_t e = cudaSuccess;
    if constexpr (Ent<L, LAYOUT>::W == 1 && L <= 8) {
        if (a.C % 64 == 0 && a.max_deg <= PrimalSite::KB) {
            k_primal_site<L, LAYOUT, POT><<<blocks_for(n, 64 * PrimalSite::WARPS), 32 * PrimalSite::WARPS, 0, s>>>(
                a, FastDiv::make((uint32_t)(a.C / 64)));
            return cudaGetLastError();
        }
    }
    if constexpr (LAYOUT == MRF_LAYOUT_PIVOT && L >= 7 && L <= 12)
        if (try_primal_pipe<L, LAYOUT, 2, POT>(a, s, e)) return e;
    if constexpr (LAYOUT == MRF_LAYOUT_PIVOT && L >= 11 && L <= 14)
        if (try_primal_pipe<L, LAYOUT, 1, POT>(a, s, e)) return e;
    if (a.max_deg <= PrimalWarp<L, LAYOUT>::KB)
        k_primal_warp<L, LAYOUT, POT, true><<<blocks_for(n, 256), 256, 0, s>>>(a);
    else
        k_primal_warp<L, LAYOUT, POT><<<blocks_for(n, 256), 256, 0, s>>>(a);
    return cudaGetLastError();
}

// Where k_primal_low beats the thread form (time over the thread form's, 100,000 to two
// million items of 2-d and 3-d lattices, 1 to 40 chains): L = 9 0.89 to 1.0, at 20,000
// items up to 1.17; L = 8 1.0 to 1.2, L = 7 0.91 to 1.05; L = 6 0.88 to 1.02 from a million items, up to 1.18 below; L = 5
// 0.83 to 1.0 from 300,000, up to 1.04 below; L = 2 to 4 only with many chains, whose
// lanes share the codes and weights, and six incidences: 0.86 to 1.0, else up to 1.2.
// Diagonal tables 0.77 to 1.0, L = 3 and 4 below 300,000 items up to 1.1.
template <int L, int LAYOUT>
bool low_form_wins(const SweepArgs& a, int64_t n) {
    constexpr int64_t kSome = 300000, kMany = 1 << 20;
    if (LAYOUT == MRF_LAYOUT_DIAG) return L >= 8 || n >= kSome;
    if (L >= 7) return L == 9 && n >= 65536;
    if (L >= 5) return n >= (L == 6 ? kMany : kSome);
    return n >= kSome && a.C >= 16 && a.max_deg >= 5;
}

// Thread or warp form of the plain primal step or its potentials.  A graph
// with hubs leaves them to a second launch; where the largest degree may
// change between launches (a batch's edit queue) there is none.
template <int L, int LAYOUT, bool POT>
cudaError_t run_field(const SweepArgs& args, cudaStream_t s) {
    const int64_t n = (int64_t)args.N * args.C;
    if (n <= 0) return cudaSuccess;
    SweepArgs a = args;
    const int hub_deg = hub_degree(n);
    const bool hubs = a.max_deg != 0x7FFFFFFF && a.max_deg > std::max(hub_deg, hub_min_degree(a.C)) &&
                      2 * a.E * a.C <= a.max_deg * kHubHidden;
    if (hubs) a.hub_deg = hub_deg;
    cudaError_t e = cudaSuccess;
    bool labels = false;
    if constexpr (LAYOUT == MRF_LAYOUT_PIVOT && L >= 5 && L <= 9) {
        // Few items: a lane per label.  us per launch, thread form / label lanes, lattices of L = 8:
        // 1,728 items 16 / 8, 13,824 18 / 11, 20,480 17 / 14, 32,768 17 / 17, 69,120 17 / 27; 25,611
        // sites of degree 15: 83 / 34; L = 4: no gain.  With a multiple of 32 chains the warp form is
        // faster (16,384 items: 8 / 12).  The limits are where the two meet on lattices (degree 4 to 6):
        // the thread form gains with the chains, whose lanes share a table row, and L = 9 pays for the
        // seven idle lanes of its sixteen (lane form over thread form, 1 / 5 / 16 chains: L = 5 at
        // 16,000 items 1.0 / 1.06 / 1.13; L = 7 at 32,000 0.95 / 0.97 / 1.15; L = 9 at 16,000
        // 0.81 / 1.03 / 1.14, at 32,000 1.3 / 1.7 / 1.9).
        constexpr int few = L == 9 ? 20480 : (L >= 7 ? 32768 : 16384);
        constexpr int many = L == 9 ? 13312 : (L == 8 ? 32768 : (L == 7 ? 24576 : (L == 6 ? 16384 : 12288)));
        labels = a.C % 32 != 0 && n <= (a.C < 4 ? few : many);
        if (labels) {
            k_primal_labels<L, LAYOUT, POT><<<blocks_for(n * LabelLanes<L>::G, 256), 256, 0, s>>>(a);
            e = cudaGetLastError();
        }
    }
    if (labels) {
        // done
    } else if (a.C % 32 == 0) {
        e = run_primal_warps<L, LAYOUT, POT>(a, s);
    } else {
        bool low = false;
        if constexpr (Ent<L, LAYOUT>::W <= 2) {
            low = a.max_deg <= 8 && low_form_wins<L, LAYOUT>(a, n);
            if (low) k_primal_low<L, LAYOUT, POT><<<blocks_for(n, 256), 256, 0, s>>>(a);
        }
        if (!low) k_primal<L, LAYOUT, false, POT><<<blocks_for(n, 256), 256, 0, s>>>(a);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess || !hubs) return e;
    const unsigned blocks = (unsigned)std::min<int64_t>(a.N, 152 * 2);
    // A CTA per 32 chains (one CTA taking them in turn: 200,000 sites, L = 4, 96 chains 1,024 us, now 925).
    const int cg = std::min(a.C, 32), groups = std::min((a.C + cg - 1) / cg, 32);
    k_primal_hub<L, LAYOUT, POT><<<dim3(blocks, (unsigned)groups), 512, 0, s>>>(a, cg);
    return cudaGetLastError();
}

template <int L, int LAYOUT, bool FUSED>
cudaError_t run_primal(const SweepArgs& a, cudaStream_t s) {
    if constexpr (!FUSED) return run_field<L, LAYOUT, false>(a, s);
    const int64_t n = (int64_t)a.N * a.C;
    if (n > 0) k_primal<L, LAYOUT, true><<<blocks_for(n, 256), 256, 0, s>>>(a);
    return cudaGetLastError();
}

template <int L, int LAYOUT>
cudaError_t run_potential(const SweepArgs& a, cudaStream_t s) { return run_field<L, LAYOUT, true>(a, s); }

template <int L, int LAYOUT>
cudaError_t run_em(const SweepArgs& a, const uint8_t* xin, uint8_t* xout, cudaStream_t s) {
    const int64_t n = (int64_t)a.N * a.C;
    if (n > 0) k_em<L, LAYOUT><<<blocks_for(n, 256), 256, 0, s>>>(a, xin, xout);
    return cudaGetLastError();
}

template <int L, int LAYOUT>
cudaError_t run_mf(const SweepArgs& a, const float* qin, float* qout, cudaStream_t s) {
    const int64_t n = (int64_t)a.N * a.C;
    if (n > 0) k_mf<L, LAYOUT><<<blocks_for(n, 256), 256, 0, s>>>(a, qin, qout);
    return cudaGetLastError();
}

template <int L, int LAYOUT>
cudaError_t run_sweep_small(const SweepArgs& a, int n_sweeps, const SmallPlan& p, cudaStream_t s) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)((a.C + p.nc - 1) / p.nc) * p.size);
    cfg.blockDim = dim3((unsigned)p.threads);
    cfg.dynamicSmemBytes = (size_t)p.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = p.size;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = p.size > 1 ? 1 : 0;
    const FastDiv fdn = FastDiv::make((uint32_t)p.nc);
    auto launch = [&](auto kernel) {
        if (p.smem > 48 * 1024) {
            const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smem);
            if (e != cudaSuccess) return e;
        }
        return cudaLaunchKernelEx(&cfg, kernel, a, n_sweeps, fdn);
    };
    if (p.form == SmallPlan::kResident) return launch(k_sweep_resident<L, LAYOUT>);
    if (p.form == SmallPlan::kCluster) return launch(k_sweep_small<L, LAYOUT, true>);
    if (p.form == SmallPlan::kOneCta) return launch(k_sweep_small<L, LAYOUT, false>);
    return cudaErrorInvalidValue;
}

template <int L, int LAYOUT>
cudaError_t run_mf_pot(const SweepArgs& a, const float* qin, cudaStream_t s) {
    const int64_t n = (int64_t)a.N * a.C;
    if (n > 0) k_mf_pot<L, LAYOUT><<<blocks_for(n, 256), 256, 0, s>>>(a, qin);
    return cudaGetLastError();
}

template <int L, int LAYOUT>
cudaError_t run_em_pot(const SweepArgs& a, const uint8_t* xin, cudaStream_t s) {
    const int64_t n = (int64_t)a.N * a.C;
    if (n > 0) k_em_pot<L, LAYOUT><<<blocks_for(n, 256), 256, 0, s>>>(a, xin);
    return cudaGetLastError();
}

#define MRF_INSTANTIATE_SWEEP(L)                                                                 \
    template cudaError_t run_mf_pot<L, MRF_LAYOUT_PIVOT>(const SweepArgs&, const float*, cudaStream_t); \
    template cudaError_t run_mf_pot<L, MRF_LAYOUT_DIAG>(const SweepArgs&, const float*, cudaStream_t);  \
    template cudaError_t run_em_pot<L, MRF_LAYOUT_PIVOT>(const SweepArgs&, const uint8_t*, cudaStream_t); \
    template cudaError_t run_em_pot<L, MRF_LAYOUT_DIAG>(const SweepArgs&, const uint8_t*, cudaStream_t);  \
    template cudaError_t run_sweep_small<L, MRF_LAYOUT_PIVOT>(const SweepArgs&, int, const SmallPlan&, cudaStream_t); \
    template cudaError_t run_sweep_small<L, MRF_LAYOUT_DIAG>(const SweepArgs&, int, const SmallPlan&, cudaStream_t);  \
    template cudaError_t run_em<L, MRF_LAYOUT_PIVOT>(const SweepArgs&, const uint8_t*, uint8_t*, cudaStream_t); \
    template cudaError_t run_em<L, MRF_LAYOUT_DIAG>(const SweepArgs&, const uint8_t*, uint8_t*, cudaStream_t);  \
    template cudaError_t run_mf<L, MRF_LAYOUT_PIVOT>(const SweepArgs&, const float*, float*, cudaStream_t);     \
    template cudaError_t run_mf<L, MRF_LAYOUT_DIAG>(const SweepArgs&, const float*, float*, cudaStream_t);      \
    template cudaError_t run_primal_cta<L, MRF_LAYOUT_PIVOT>(const SweepArgs&, cudaStream_t);     \
    template cudaError_t run_primal_cta<L, MRF_LAYOUT_DIAG>(const SweepArgs&, cudaStream_t);      \
    template cudaError_t run_potential<L, MRF_LAYOUT_PIVOT>(const SweepArgs&, cudaStream_t);      \
    template cudaError_t run_potential<L, MRF_LAYOUT_DIAG>(const SweepArgs&, cudaStream_t);       \
    template cudaError_t run_sweep_partial<L, MRF_LAYOUT_PIVOT>(const SweepArgs&, int, cudaStream_t); \
    template cudaError_t run_sweep_partial<L, MRF_LAYOUT_DIAG>(const SweepArgs&, int, cudaStream_t);  \
    template cudaError_t run_dual<L, MRF_LAYOUT_PIVOT>(const SweepArgs&, cudaStream_t);           \
    template cudaError_t run_dual<L, MRF_LAYOUT_DIAG>(const SweepArgs&, cudaStream_t);            \
    template cudaError_t run_primal<L, MRF_LAYOUT_PIVOT, false>(const SweepArgs&, cudaStream_t);  \
    template cudaError_t run_primal<L, MRF_LAYOUT_DIAG, false>(const SweepArgs&, cudaStream_t);   \
    template cudaError_t run_primal<L, MRF_LAYOUT_PIVOT, true>(const SweepArgs&, cudaStream_t);   \
    template cudaError_t run_primal<L, MRF_LAYOUT_DIAG, true>(const SweepArgs&, cudaStream_t);

}  // namespace mrfk
