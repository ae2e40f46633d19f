// Factor decomposition of Sections 4.1-4.2 on the device (setup and edits).
//
// For every edge e with log-table w (L x L, row = label of the source):
//  * PIVOT layout: l(i,j) = w(i,j) - w(i,0) - w(0,j) + w(0,0) for i, j >= 1;
//    offsets w(a,0) - w(0,0) fold into the source unary, w(0,b) - w(0,0) into
//    the destination unary, w(0,0) into the log constant.
//  * DIAG layout (Potts-type tables, Section 4.2): l(a,a) = w(a,a), no offsets.
// Every entry with l != 0 gets one dual bit (Section 4.2: none for 1-entries).
// Its one-hot 2x2 factor [[1,1],[1,e^l]] factors as in Lemmas 2-4 and Theorem 2;
// in closed form, with tau = 2 arccosh(e^{|l|/2}) evaluated stably as
// tau = |l| + 2 log1p(sqrt(-expm1(-|l|))):
//    l > 0:  q = -tau, beta1 = beta2 = tau, alpha1 = alpha2 = (l - tau)/2
//    l < 0:  q = 0, beta1 = -tau, beta2 = tau, alpha1 = (l + tau)/2, alpha2 = (l - tau)/2
// so the dual logit q + beta1 y + beta2 z takes one of {-tau, 0, +tau}.
//
// Stored per entry: tau_signed (= beta1; beta2 = |tau_signed|) as float, and a
// packed threshold word: T+ = ceil(sigmoid(tau) 2^24 - 1/2) in bits 0..24,
// d = T+ + T- - (2^24 - 1) in bits 25..26 (T- from sigmoid(-tau)), the sign of
// l in bit 31; 0 marks an entry without a dual bit.  A draw with 24-bit
// integer uniform U sets theta iff U < T for the case's threshold, which is
// exactly u = (U + 1/2) / 2^24 < p.  All of this runs in float64.
#include "common.cuh"

#include <algorithm>
#include <cmath>

namespace mrfk {

__global__ void k_check_finite(const float* p, int64_t n, unsigned long long* bad) {
    unsigned long long cnt = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        cnt += !isfinite(p[i]);
    if (cnt) atomicAdd(bad, cnt);
}

// One row of a table per thread, one atomic per block (one per thread held
// every table with off-diagonal values up on a single address: 153,040 tables of
// 5 x 5 took 209 us for 15 MB).
__global__ void k_count_offdiag(const float* pair, int64_t n_edges, int L, FastDiv fdL, unsigned long long* nz) {
    const int64_t rows = n_edges * L;
    unsigned long long cnt = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < rows; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e0 = i < 0xFFFFFFFFll ? (int64_t)fdL.div((uint32_t)i) : i / L;
        const int r = (int)(i - e0 * L);
        for (int c = 0; c < L; ++c) cnt += (r != c) && (pair[i * L + c] != 0.0f);
    }
    __shared__ unsigned long long s_cnt;
    if (threadIdx.x == 0) s_cnt = 0ull;
    __syncthreads();
    cnt = __reduce_add_sync(0xffffffffu, (unsigned)cnt);   // a thread's share is far below 2^27
    if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(&s_cnt, cnt);
    __syncthreads();
    if (threadIdx.x == 0 && s_cnt) atomicAdd(nz, s_cnt);
}

// A block takes `eb` edges.  Their entries are spread over its threads (the
// float64 transcendentals of entry_dual are the kernel's time, so every lane
// has one, and few edges still fill the GPU: 1,470 new edges of 225 entries in
// a thread per edge took 1.53 ms, 0.10 ms here); the entries' terms meet in
// shared memory, where a thread per row or column sums them in entry order.
constexpr int kDecompItems = 512;                          // entries of a block
__global__ void __launch_bounds__(128) k_decompose(DecompArgs a, int eb) {
    __shared__ double s_a1[kDecompItems], s_a2[kDecompItems], s_ln[kDecompItems];
    __shared__ double s_f[kDecompItems * 2];               // folded rows and columns of the block's edges
    __shared__ double s_row[kDecompItems];             // log-constant terms per row
    const int64_t n = a.n_dev && *a.n_dev < a.n ? *a.n_dev : a.n;
    const int64_t i0 = (int64_t)blockIdx.x * eb;
    if (i0 >= n || (a.status && (*a.status & kQFatal))) return;
    const int L = a.L, M = a.M, MP = pad4(M), ne = (int)(n - i0 < eb ? n - i0 : eb), tid = threadIdx.x;
    const bool pivot = a.layout == MRF_LAYOUT_PIVOT;
    auto slot = [&](int q) { return a.slots ? a.slots[i0 + q] : a.first_slot + i0 + q; };
    auto table = [&](int q) { return a.pair + (a.pair_off ? a.pair_off[i0 + q] : (i0 + q) * L * L); };
    for (int it = tid; it < ne * M; it += 128) {
        const int q = it / M, k = it - q * M;
        const float* w = table(q);
        double l;
        if (pivot) {
            const int r = k / (L - 1), ii = 1 + r, jj = 1 + k - r * (L - 1);
            l = (double)w[ii * L + jj] - (double)w[ii * L] - (double)w[jj] + (double)w[0];
        } else {
            l = (double)w[k * L + k];
        }
        EntryDual d{};
        if (l != 0.0) d = entry_dual(l);
        s_a1[it] = d.alpha1; s_a2[it] = d.alpha2; s_ln[it] = d.log_norm;   // -log(1 + e^q)
        const int64_t e = slot(q);
        a.tau[e * MP + k] = d.tau_s;
        a.thr[e * M + k] = d.word;
        if (k < MP - M) a.tau[e * MP + M + k] = 0.0f;      // the row's padding (at most 3, M = 1: see below)
        if (M == 1) { a.tau[e * MP + 2] = 0.0f; a.tau[e * MP + 3] = 0.0f; }
    }
    __syncthreads();
    // entries of row x (source side) or column x (destination side), in entry order
    for (int j = tid; j < ne * 2 * L; j += 128) {
        const int q = j / (2 * L), sd = j - q * 2 * L, side = sd >= L, x = sd - side * L;
        const float* w = table(q);
        double f = 0.0, ln = 0.0;
        if (pivot) {
            f = (double)w[side ? x : x * L] - (double)w[0];
            if (x > 0)
                for (int y = 0; y < L - 1; ++y) {
                    const int k = q * M + (side ? y * (L - 1) + x - 1 : (x - 1) * (L - 1) + y);
                    f += side ? s_a2[k] : s_a1[k];
                    if (!side) ln += s_ln[k];
                }
        } else {
            f += side ? s_a2[q * M + x] : s_a1[q * M + x];
            ln = s_ln[q * M + x];
        }
        s_f[j] = f;
        if (!side) s_row[q * L + x] = ln;
        a.fold[slot(q) * 2 * L + sd] = f;
    }
    __syncthreads();
    for (int q = tid; q < ne; q += 128) {
        double cst = pivot ? (double)table(q)[0] : 0.0;
        for (int x = 0; x < L; ++x) cst += s_row[q * L + x];
        a.cst[slot(q)] = cst;
    }
    if (a.sw_thr && (!pivot || L == 2)) {
        // Swendsen-Wang tables (Section 4.3): the table as
        // c + f(a) + g(b) + l_a [a = b] -- diagonal tables: l_x = w(x,x), f = g = 0;
        // two labels: l = (w00 + w11 - w01 - w10) / 2 for both labels,
        // f(1) = w10 - w00 + l, g(1) = w01 - w00 + l (folded into the SW unaries).
        // Per label x: bond probability 1 - e^{-l_x} as the exact 23-bit threshold
        // T = ceil(p 2^23 - 1/2) (a draw U bonds iff U < T, i.e. (U + 1/2) / 2^23 < p),
        // and the bond's label weight log(e^{l_x} - 1) in fixed point (sw_fix);
        // l <= 0: no bond (T = 0) and the label is excluded when bonded (kSwNoLabel).
        for (int j = tid; j < ne * L; j += 128) {
            const int q = j / L, x = j - q * L;
            const float* w = table(q);
            const int64_t e = slot(q);
            double l;
            if (L == 2) {
                l = 0.5 * ((double)w[0] + (double)w[3] - (double)w[1] - (double)w[2]);
                if (a.sw_fold) {
                    a.sw_fold[(e * 2 + 0) * 2 + x] = x ? (double)w[2] - (double)w[0] + l : 0.0;
                    a.sw_fold[(e * 2 + 1) * 2 + x] = x ? (double)w[1] - (double)w[0] + l : 0.0;
                }
            } else {
                l = (double)w[x * L + x];
            }
            uint32_t T = 0;
            int64_t lw = kSwNoLabel;
            if (l > 0.0) {
                T = (uint32_t)ceil(-expm1(-l) * 8388608.0 - 0.5);
                lw = sw_fix(log(expm1(l)));
            }
            a.sw_thr[e * L + x] = T;
            a.sw_lw[e * L + x] = lw;
            if (a.sw_ell) a.sw_ell[e * L + x] = l;
        }
    }
    if (a.resid) {
        // exact pairwise potential in the folded representation (tree edges of
        // the blocked sweep): w(a,b) - fold_s(a) - fold_t(b)
        for (int j = tid; j < ne * L * L; j += 128) {
            const int q = j / (L * L), xy = j - q * L * L, x = xy / L, y = xy - x * L;
            a.resid[slot(q) * L * L + xy] =
                (float)((double)table(q)[xy] - s_f[q * 2 * L + x] - s_f[q * 2 * L + L + y]);
        }
    }
}

// Threshold prefix planes of the bit-sliced dual draw, per edge and group of
// 32 entries (entry 32g + b at bit b).  An entry's dual logit is at one of
// three levels: 0 (-tau, threshold T-), 1 (logit 0, T = 2^23) or 2 (+tau, T+);
// which one depends on its sign and its case (see dual_prefix_bits).  Stored:
// the 8 bit planes of the 8-bit prefix of T+ (B_p: bit 7 - p of the prefix),
// the planes of the difference between the prefixes of T- and T+
// (AB_p = A_p ^ B_p, A_p the planes of T-'s prefix), the sign mask and the mask
// of entries with a dual bit:
//   uint4 {AB_p, B_p, AB_p+1, B_p+1} for p = 0, 2, 4, 6,   uint4 {S, Act, 0, 0}
// 20 words per group.  A chain whose level-0 entries are L0 reads its
// threshold plane as B_p ^ (AB_p & L0).  Tables with at most 16 entries pack
// two planes per word (plane p in bits 0..15, plane p + 4 in bits 16..31), 12
// words per edge:
//   uint4 {AB_0|AB_4<<16, .., AB_3|AB_7<<16}, uint4 {B likewise}, uint4 {S | Act << 16, 0, 0, 0}.
__global__ void k_build_planes(const uint32_t* thr, int64_t n, const int64_t* slots, int64_t first_slot, int M,
                               uint32_t* tpl, const int64_t* n_dev, const uint32_t* status) {
    const int G = (M + 31) / 32;
    const int64_t gid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (gid >= n * G) return;
    const int64_t i = gid / G;
    if ((n_dev && i >= *n_dev) || (status && (*status & kQFatal))) return;
    const int g = (int)(gid % G);
    const int64_t e = slots ? slots[i] : first_slot + i;
    uint32_t A[8] = {0, 0, 0, 0, 0, 0, 0, 0}, B[8] = {0, 0, 0, 0, 0, 0, 0, 0}, S = 0, Act = 0;
    for (int b = 0; b < 32; ++b) {
        const int k = 32 * g + b;
        if (k >= M) break;
        const uint32_t w = thr[e * M + k];
        const uint32_t pa = threshold_prefix(level_threshold(w, false));
        const uint32_t pb = threshold_prefix(level_threshold(w, true));
        for (int p = 0; p < 8; ++p) {
            A[p] |= ((pa >> (7 - p)) & 1u) << b;
            B[p] |= ((pb >> (7 - p)) & 1u) << b;
        }
        S |= (w >> 31) << b;
        Act |= (w != 0u ? 1u : 0u) << b;
    }
    uint4* out = reinterpret_cast<uint4*>(tpl + e * (int64_t)plane_words(M) + 20 * g);
    for (int p = 0; p < 8; ++p) A[p] ^= B[p];
    if (M <= 16) {
        out[0] = make_uint4(A[0] | A[4] << 16, A[1] | A[5] << 16, A[2] | A[6] << 16, A[3] | A[7] << 16);
        out[1] = make_uint4(B[0] | B[4] << 16, B[1] | B[5] << 16, B[2] | B[6] << 16, B[3] | B[7] << 16);
        out[2] = make_uint4(S | Act << 16, 0u, 0u, 0u);
        return;
    }
    for (int p = 0; p < 8; p += 2) out[p / 2] = make_uint4(A[p], B[p], A[p + 1], B[p + 1]);
    out[4] = make_uint4(S, Act, 0u, 0u);
}

// A thread per (site, label): the incidences' terms in order, float64.
__global__ void k_fold_unary(const float* unary, const double* unary_d, const double* fold, const int64_t* inc_ptr,
                             const int2* inc, int N, int L, FastDiv fdL, double* ut, float* utf) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= (int64_t)N * L) return;
    const int64_t v = i < 0xFFFFFFFFll ? (int64_t)fdL.div((uint32_t)i) : i / L;
    const int x = (int)(i - v * L);
    double acc = unary_d ? unary_d[i] : (double)unary[i];
    for (int64_t p = inc_ptr[v]; p < inc_ptr[v + 1]; ++p) acc += fold[(int64_t)inc[p].x * L + x];   // code = 2 edge + side
    ut[i] = acc;
    if (utf) utf[i] = (float)acc;
}

__global__ void __launch_bounds__(256) k_sum_double(const double* __restrict__ p, int64_t n, double* __restrict__ out) {
    __shared__ double s_sum[256];
    double acc = 0.0;
    for (int64_t i = blockIdx.x * 256ll + threadIdx.x; i < n; i += gridDim.x * 256ll) acc += p[i];
    s_sum[threadIdx.x] = acc;
    for (int o = 128; o > 0; o >>= 1) {
        __syncthreads();
        if (threadIdx.x < o) s_sum[threadIdx.x] += s_sum[threadIdx.x + o];
    }
    if (threadIdx.x == 0) out[blockIdx.x] = s_sum[0];
}

cudaError_t launch_sum_double(const double* p, int64_t n, double* out, cudaStream_t s) {
    k_sum_double<<<kSumBlocks, 256, 0, s>>>(p, n, out);
    return cudaGetLastError();
}

cudaError_t launch_check_finite(const float* p, int64_t n, unsigned long long* bad, cudaStream_t s) {
    if (n > 0) k_check_finite<<<1216, 256, 0, s>>>(p, n, bad);
    return cudaGetLastError();
}

cudaError_t launch_count_offdiag(const float* pair, int64_t n_edges, int L, unsigned long long* nz, cudaStream_t s) {
    if (n_edges > 0) k_count_offdiag<<<1216, 256, 0, s>>>(pair, n_edges, L, FastDiv::make((uint32_t)L), nz);
    return cudaGetLastError();
}

cudaError_t launch_decompose(const DecompArgs& a, cudaStream_t s) {
    if (a.n <= 0) return cudaSuccess;
    // up to 512 entries (and 512 row sums) per block, fewer while the blocks do not fill the GPU
    const int most = std::max(1, kDecompItems / std::max(a.M, a.L));
    const int eb = (int)std::min<int64_t>(most, std::max<int64_t>(std::max(1, 128 / a.M), (a.n + 152 * 8 - 1) / (152 * 8)));
    k_decompose<<<(unsigned)((a.n + eb - 1) / eb), 128, 0, s>>>(a, eb);
    return cudaGetLastError();
}

cudaError_t launch_fold_unary(const float* unary, const double* fold, const int64_t* inc_ptr, const int2* inc,
                              int N, int L, double* ut, float* utf, cudaStream_t s, const double* unary_d) {
    const int64_t n = (int64_t)N * L;
    if (n > 0)
        k_fold_unary<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(unary, unary_d, fold, inc_ptr, inc, N, L,
                                                                 FastDiv::make((uint32_t)L), ut, utf);
    return cudaGetLastError();
}

cudaError_t launch_build_planes(const uint32_t* thr, int64_t n, const int64_t* slots, int64_t first_slot, int M,
                                uint32_t* tpl, cudaStream_t s, const int64_t* n_dev, const uint32_t* status) {
    const int64_t work = n * ((M + 31) / 32);
    if (work > 0)
        k_build_planes<<<(unsigned)((work + 127) / 128), 128, 0, s>>>(thr, n, slots, first_slot, M, tpl, n_dev, status);
    return cudaGetLastError();
}

}  // namespace mrfk
