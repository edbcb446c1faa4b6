// Stage 3: pivot selection (Eq. 4) on the O2Graph.
//
// P = the min(K1, |E+|) edges (i < j, W_ij > 0) of largest weight, ties at
// the threshold weight alpha broken by the lowest (i, j) (row-major linear
// index), listed in (W desc, i asc, j asc) order.  With the learned
// proposal the competing weight is floor(W_ij p_i p_j) (pivot_weight).
//
// Exact radix-style selection; the selected set, and so the pivots, do not
// depend on the order in which blocks run:
//   hist    histogram of edge weights (built by the SC^2 pass; by a pass of its
//           own for the learned weights and for a caller's matrix, there with
//           the row maxima)
//   select  alpha = K1-th largest weight, c_gt = #{W > alpha}, m = K1' - c_gt
//           ties still needed (K1' = min(K1, |E+|)): every count block for
//           one problem, else one block per problem of the select launch
//   count   blocks of eight row pairs (i, n-1-i): #{j : W_ij > alpha} and
//           #{j : W_ij == alpha}; rows with such edges join the active list
//           (rows whose largest weight, recorded by the SC^2 pass, is below
//           alpha are skipped without reading W)
//   emit    blocks over the active rows: W > alpha edges take slots from one
//           atomic per row (the rank pass orders them); ties get global tie
//           ranks (tie prefix over the active rows above) + rank-in-row
//           (column order) and ranks < m are kept
//   rank    candidate keys (W << 32 | ~(i*n+j)) are unique; each pivot's
//           position is the number of larger keys.  In the registration
//           pipeline the clique search computes these ranks itself (one warp
//           per selected edge); rank_kernel serves the allocation-free
//           selection entry point.
#include "tr_common.cuh"
#include "tr_problem.h"
#include "tr_select.cuh"

namespace tr {

namespace {

constexpr int kHistSmemMaxBins = 24576;   // 96 KB of shared bins; larger N uses global atomics
constexpr int kCountThreads = 256;
constexpr int kCountPairs = 8;            // row pairs per count block

__device__ __forceinline__ uint64_t edge_key(int w, int i, int j, int n)
{
    const uint32_t lin = static_cast<uint32_t>(i) * static_cast<uint32_t>(n) + static_cast<uint32_t>(j);
    return (static_cast<uint64_t>(w) << 32) | static_cast<uint64_t>(0xFFFFFFFFu - lin);
}

// Largest learned pivot weight a row can hold, before truncation: every entry
// of row i has floor(W_ij p_i p_j) with W_ij <= rowmax_i and p_j <= max p, and
// correctly rounded products of non-negative factors are monotonic, so
// fl(fl(W_ij p_i) p_j) <= fl(fl(rowmax_i p_i) pmax).  Infinite when no bound
// is available (plain weights, or no row maxima).
__device__ __forceinline__ float learned_row_bound(const ProbView& v, int i)
{
    if (v.prob == nullptr || v.rowmax == nullptr) return __int_as_float(0x7f800000);
    const float pmax = __uint_as_float(__ldcg(&v.ctl->pmax_bits));
    return __fmul_rn(__fmul_rn(static_cast<float>(__ldcg(v.rowmax + i)), __ldcg(v.prob + i)), pmax);
}

// Zero the weights of a 16-byte chunk (8 entries, columns 8c .. 8c+7) outside
// the row's upper part (row, n): only a row's first and last chunks have any.
__device__ __forceinline__ uint4 mask_chunk(uint4 q, int c, int row, int n)
{
    const int lo = row + 1 - c * 8, hi = n - c * 8;   // keep entries e with lo <= e < hi
    if (lo <= 0 && hi >= 8) return q;
    uint32_t wd[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int e = 0; e < 8; ++e)
        if (e < lo || e >= hi) wd[e >> 1] &= (e & 1) ? 0x0000FFFFu : 0xFFFF0000u;
    return make_uint4(wd[0], wd[1], wd[2], wd[3]);
}

// Eight row pairs (p, n-1-p) of a block, whose upper-triangle parts hold about
// n/8 16-byte chunks per pair, so that every group has about the same span of
// rows; entry k: pair 8 g + k / 2, side k % 2.
struct RowGroup {
    int row[16], c0[16], off[17];   // row, its first chunk, first chunk number in the group
};

// Row of entry t (< 16) of group g; false when the entry holds no edge.
__device__ __forceinline__ bool group_row(int g, int t, int n, int& row)
{
    const int p = g * kCountPairs + (t >> 1);
    row = (t & 1) ? n - 1 - p : p;
    return t < 16 && p < (n + 1) / 2 && !((t & 1) && row == p) && row + 1 < n;
}

// The group's chunk numbering over its rows marked `act`, by one warp (lane t < 32).
__device__ __forceinline__ void group_offsets(RowGroup& sg, int t, int row, bool act, int n)
{
    const int c0 = (row + 1) >> 3;
    const int len = act ? ((n - 1) >> 3) - c0 + 1 : 0;
    int incl = len;
#pragma unroll
    for (int off = 1; off < 16; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, off);
        if (t >= off) incl += y;
    }
    if (t < 16) {
        sg.row[t] = row;
        sg.c0[t] = c0;
        sg.off[t] = incl - len;
    }
    if (t == 15) sg.off[16] = incl;
}

// The group's chunks spread over T threads (this one is number t), eight
// 16-byte loads in flight each: f(k, row, c, weights) for chunk c of entry k,
// entries outside the upper part zeroed.
template <int T = kCountThreads, typename F>
__device__ __forceinline__ void for_group_chunks(const ProbView& v, const RowGroup& sg, int t, F&& f)
{
    const int tot = sg.off[16];
    for (int base = t; base < tot; base += 8 * T) {
        uint4 q[8];
        int kk[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int x = base + u * T;
            int k = 0;   // the last entry that begins at or before chunk x
#pragma unroll
            for (int m = 8; m >= 1; m >>= 1) k += sg.off[k + m] <= x ? m : 0;
            kk[u] = k;
            q[u] = x < tot ? *reinterpret_cast<const uint4*>(v.w + (size_t)sg.row[k] * v.n_pad +
                                                             (size_t)(sg.c0[k] + x - sg.off[k]) * 8)
                           : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int x = base + u * T;
            if (x >= tot) break;
            const int k = kk[u];
            const int row = sg.row[k], c = sg.c0[k] + x - sg.off[k];
            f(k, row, c, mask_chunk(q[u], c, row, v.n));
        }
    }
}

// floor of a learned weight fl(fl(W p_i) p_j), the integer pivot_weight takes:
// added to 2^23 toward zero, the floor is the low bits (0 <= W p_i p_j < 2^15;
// a NaN counts as 0, as the conversion has it).
__device__ __forceinline__ uint32_t learned_weight(uint32_t w, float pi, float pj)
{
    const float x = __fmul_rn(__fmul_rn(__uint_as_float(0x4B000000u | w) - 8388608.f, pi), pj);
    return __float_as_uint(__fadd_rz(fmaxf(x, 0.f), 8388608.f)) & 0x7FFFFFu;
}

// Histogram of the learned weights: the groups of row pairs of the count pass.
// Most rows hold only zeros (their bound is below 1) and are skipped, so the
// chunks of the others are spread over the whole block (a warp per row pair
// took 144 us instead of 99 for 32 problems: one or two warps of a block had
// all its rows).
template <bool kSmem>
__global__ void __launch_bounds__(kCountThreads, 3) learned_hist_kernel(ManyViews vs)
{
    int lb;
    const ProbView v = vs.get(ST_HIST, blockIdx.x, lb);   // launch descriptors: before the wait
    extern __shared__ uint32_t sh[];
    __shared__ RowGroup sg;
    const int n = v.n, t = threadIdx.x;
    if (kSmem)
        for (int q = t; q <= n; q += kCountThreads) sh[q] = 0;
    pdl_wait();
    pdl_release();
    uint32_t* const bins = kSmem ? sh : v.hist;
    const int groups = count_groups(n), stride = hist_blocks(n);
    for (int g = lb; g < groups; g += stride) {
        __syncthreads();   // the bins are cleared; the previous group's list is consumed
        if (t < 32) {
            int row;
            const bool act = group_row(g, t, n, row) && learned_row_bound(v, row) >= 1.f;
            group_offsets(sg, t, row, act, n);
        }
        __syncthreads();
        for_group_chunks(v, sg, t, [&](int, int row, int c, uint4 q) {
            if ((q.x | q.y | q.z | q.w) == 0u) return;
            const uint32_t wd[4] = {q.x, q.y, q.z, q.w};
            const float pi = __ldcg(v.prob + row);
            // (n_pad is a multiple of 256: the probabilities of a whole chunk can be read)
            const float4 pa = __ldcg(reinterpret_cast<const float4*>(v.prob + c * 8));
            const float4 pb = __ldcg(reinterpret_cast<const float4*>(v.prob + c * 8 + 4));
            const float pj[8] = {pa.x, pa.y, pa.z, pa.w, pb.x, pb.y, pb.z, pb.w};
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const uint32_t w = (wd[e >> 1] >> ((e & 1) * 16)) & 0xFFFFu;
                const uint32_t pw = w != 0u ? learned_weight(w, pi, pj[e]) : 0u;
                if (pw != 0u) atomicAdd(bins + pw, 1u);
            }
        });
    }
    if (kSmem) {
        __syncthreads();
        for (int q = t; q <= n; q += kCountThreads)
            if (sh[q]) atomicAdd(&v.hist[q], sh[q]);
    }
}

// Histogram of a caller's matrix (n <= 8192: the bins fit in shared memory),
// one block per SM.  The chunks of a row pair (p, n-1-p), about n/8 together,
// are cut into windows of 256, and the warps of the grid take windows, eight
// 16-byte loads per lane in flight.  It reads the upper triangle once; the
// entries of a chunk are counted by predicated additions without branches.  One
// block per SM because every block adds its bins to the same few hundred
// global ones.  At n = 5000: 15.0 us; with 313 blocks of a warp per pair 20.4, 625
// of two 22.4; with the chunks of 16 rows spread over a block, each looking up
// its row and checking every entry, 24.7; with a warp per row, two loads in
// flight and 64 rows per block 196 (the whole selection then 231 us, now 35).
// A weight above n - 2 (no SC^2 count can be larger; the bins end at n) is not
// counted: it sets TR_ERR_BAD_WEIGHT, and nothing is selected then.  The row
// maxima (cleared before) are recorded, so that the count pass skips rows.
constexpr int kWindow = 256;
// windows per pair, whose two rows hold at most n / 8 + 3 chunks (both round outwards)
__host__ __device__ inline int caller_windows(int n) { return (n / 8 + 3 + kWindow - 1) / kWindow; }

__global__ void __launch_bounds__(1024, 1) caller_hist_kernel(OneView vs)
{
    int lb;
    const ProbView v = vs.get(ST_HIST, blockIdx.x, lb);
    extern __shared__ uint32_t sh[];
    const int n = v.n, t = threadIdx.x, lane = t & 31;
    for (int q = t; q <= n; q += 1024) sh[q] = 0;
    pdl_wait();
    pdl_release();
    __syncthreads();   // the bins are cleared
    const int c1 = (n - 1) >> 3, nw = caller_windows(n), items = (n + 1) / 2 * nw;
    const uint32_t wmax = static_cast<uint32_t>(max(n - 2, 0));
    bool bad = false;
    for (int it = (t >> 5) * static_cast<int>(gridDim.x) + lb; it < items; it += 32 * static_cast<int>(gridDim.x)) {
        const int p = it / nw, x0 = (it - p * nw) * kWindow + lane;
        const int ra = p, rb = n - 1 - p;   // (one row when they meet)
        const int ca = (ra + 1) >> 3, cb = (rb + 1) >> 3;
        const int la = ra + 1 < n ? c1 - ca + 1 : 0, lt = la + (rb > ra && rb + 1 < n ? c1 - cb + 1 : 0);
        const uint16_t *wa = v.w + (size_t)ra * v.n_pad, *wb = v.w + (size_t)rb * v.n_pad;
        uint4 q[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int x = x0 + 32 * u;
            q[u] = x < lt ? *reinterpret_cast<const uint4*>(x < la ? wa + (ca + x) * 8 : wb + (cb + x - la) * 8)
                          : make_uint4(0u, 0u, 0u, 0u);
        }
        uint32_t ma = 0u, mb = 0u;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int x = x0 + 32 * u;
            const bool in_a = x < la;
            const uint4 qm = mask_chunk(q[u], in_a ? ca + x : cb + x - la, in_a ? ra : rb, n);
            const uint32_t wd[4] = {qm.x, qm.y, qm.z, qm.w};
            const uint32_t m2 = __vmaxu2(__vmaxu2(wd[0], wd[1]), __vmaxu2(wd[2], wd[3]));
            const uint32_t m = max(m2 & 0xFFFFu, m2 >> 16);
            if (in_a) ma = max(ma, m);
            else mb = max(mb, m);
            if (m > wmax) {
                bad = true;
                continue;
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const uint32_t w = (wd[e >> 1] >> ((e & 1) * 16)) & 0xFFFFu;
                if (w != 0u) atomicAdd(sh + w, 1u);
            }
        }
        ma = __reduce_max_sync(0xffffffffu, ma);
        mb = __reduce_max_sync(0xffffffffu, mb);
        if (lane == 0) {
            if (ma != 0u) atomicMax(v.rowmax + ra, static_cast<int>(ma));
            if (mb != 0u) atomicMax(v.rowmax + rb, static_cast<int>(mb));
        }
    }
    if (bad) atomicOr(&v.ctl->err, TR_ERR_BAD_WEIGHT);
    __syncthreads();
    for (int q = t; q <= n; q += 1024)
        if (sh[q]) atomicAdd(&v.hist[q], sh[q]);
}

__global__ void __launch_bounds__(1024) select_kernel(ManyViews vs)
{
    int lb;
    const ProbView v = vs.get(ST_SELECT, blockIdx.x, lb);   // launch descriptors: before the wait
    pdl_wait();
    pdl_release();
    __shared__ int sbuf[33];
    select_alpha(v, sbuf);
}

// Whether a chunk holds a weight of at least alpha (few do: the passes over the
// active rows visit the entries of those only; a learned weight never exceeds
// the plain one).
__device__ __forceinline__ bool chunk_reaches(uint4 q, int alpha)
{
    const uint32_t m = __vmaxu2(__vmaxu2(q.x, q.y), __vmaxu2(q.z, q.w));
    return static_cast<int>(m & 0xFFFFu) >= alpha || static_cast<int>(m >> 16) >= alpha;
}

// Adds a chunk's #{weight > alpha} and #{weight == alpha} to g and e.
__device__ __forceinline__ void count_chunk(const ProbView& v, int row, int c, uint4 q, int alpha, bool learned, int& g,
                                            int& e)
{
    if (!chunk_reaches(q, alpha)) return;
#pragma unroll
    for (int el = 0; el < 8; ++el) {
        const uint32_t word = el < 2 ? q.x : el < 4 ? q.y : el < 6 ? q.z : q.w;
        int pw = static_cast<int>((word >> ((el & 1) * 16)) & 0xFFFFu);
        if (learned) pw = pivot_weight(v, row, c * 8 + el, pw);
        g += pw > alpha;
        e += pw == alpha;
    }
}

// Per-row counts of the weight > alpha and weight == alpha edges.  A block
// owns a group of eight row pairs.  Rows whose largest weight (recorded by the
// SC^2 pass or the histogram) is below alpha hold no such edge and are skipped
// without reading W (the learned pivot weight floor(W p_i p_j) never exceeds
// W).  The chunks of the remaining rows are spread over all the block's
// threads, so a block with one or two such rows reads them in one round.
// Rows holding such edges are appended to the active list as (row, #gt, #eq),
// in any order.
// select_here (one problem whose histogram is complete): every block chooses
// the threshold itself from the histogram, staged in dynamic shared memory
// while its row maxima load, and block 0 records it for the later passes;
// otherwise it comes from the select launch.
template <class VS>
__global__ void __launch_bounds__(kCountThreads, 3) count_kernel(VS vs, int select_here)
{
    int lb;
    const ProbView v = vs.get(ST_COUNT, blockIdx.x, lb);   // launch descriptors: before the wait
    pdl_wait();
    pdl_release();
    extern __shared__ __align__(16) uint32_t shist_stage[];   // select_here: n + 4 words
    __shared__ RowGroup sg;
    __shared__ int sgt[16], seq[16];
    __shared__ int ssel[40];
    const int n = v.n;
    const int t = threadIdx.x;
    int row;
    bool act = group_row(lb, t, n, row);
    const int rmax = (act && v.rowmax != nullptr) ? __ldg(v.rowmax + row) : 0;
    int n_sel, alpha;
    if (select_here) {
        select_alpha(v, ssel, shist_stage, ssel + 33);
        __syncthreads();
        n_sel = ssel[34];
        alpha = ssel[35];
        if (lb == 0 && t == 0) {
            v.ctl->n_edges = ssel[33];
            v.ctl->n_sel = n_sel;
            v.ctl->alpha = alpha;
            v.ctl->c_gt = ssel[36];
            v.ctl->m_ties = ssel[37];
        }
    } else {
        n_sel = v.ctl->n_sel;
        alpha = v.ctl->alpha;
    }
    if (n_sel == 0) return;                   // uniform over the block
    const bool learned = v.prob != nullptr;
    if (t < 32) {
        if (act && v.rowmax != nullptr) act = rmax >= alpha;
        if (act && learned) act = learned_row_bound(v, row) >= static_cast<float>(alpha);
        group_offsets(sg, t, row, act, n);
        if (t < 16) sgt[t] = seq[t] = 0;
    }
    __syncthreads();
    if (sg.off[16] == 0) return;              // uniform over the block
    int kcur = -1, g = 0, e = 0;              // running counts of entry kcur
    auto flush = [&]() {
        if (g) atomicAdd(&sgt[kcur], g);
        if (e) atomicAdd(&seq[kcur], e);
    };
    for_group_chunks(v, sg, t, [&](int k, int row_k, int c, uint4 qm) {
        if (k != kcur) {
            if (kcur >= 0) flush();
            kcur = k;
            g = e = 0;
        }
        count_chunk(v, row_k, c, qm, alpha, learned, g, e);
    });
    if (kcur >= 0) flush();
    __syncthreads();
    if (t < 16 && (sgt[t] | seq[t]))
        v.active[atomicAdd(&v.ctl->n_active, 1u)] = make_int4(sg.row[t], sgt[t], seq[t], 0);
}

// The same counts in a batch of many problems: a warp per group, without block
// barriers; the threshold comes from the select launch.  With a block per group
// the pass over 256 problems took 364 us (blocks that start, find their problem
// and read nothing; with four groups per block it was bound by its barriers), so
// 125 (device times in a profiler's launch list, cold caches).
__global__ void __launch_bounds__(kCountThreads, 4) count_warp_kernel(ManyViews vs)
{
    int lb;
    const ProbView v = vs.get(ST_COUNT, blockIdx.x, lb);   // launch descriptors: before the wait
    pdl_wait();
    pdl_release();
    __shared__ RowGroup sgs[kCountThreads / 32];
    __shared__ int scnt[kCountThreads / 32][16];   // #gt | #eq << 16 (a row has fewer than 2^15 entries)
    const int n = v.n, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    RowGroup& sg = sgs[warp];
    int row;
    bool act = group_row(lb * (kCountThreads / 32) + warp, lane, n, row);
    const int rmax = act ? __ldg(v.rowmax + row) : 0;
    const int alpha = v.ctl->alpha;
    if (v.ctl->n_sel == 0) return;
    const bool learned = v.prob != nullptr;
    act = act && rmax >= alpha;
    if (act && learned) act = learned_row_bound(v, row) >= static_cast<float>(alpha);
    if (!__any_sync(0xffffffffu, act)) return;
    group_offsets(sg, lane, row, act, n);
    if (lane < 16) scnt[warp][lane] = 0;
    __syncwarp();
    for_group_chunks<32>(v, sg, lane, [&](int k, int row_k, int c, uint4 q) {
        int g = 0, e = 0;
        count_chunk(v, row_k, c, q, alpha, learned, g, e);
        if ((g | e) != 0) atomicAdd(&scnt[warp][k], g | (e << 16));
    });
    __syncwarp();
    static_assert(TURBOREG_MAX_N <= 32768, "a row's counts fit 16 bits each");
    if (lane < 16) {
        const uint32_t ge = static_cast<uint32_t>(scnt[warp][lane]);
        if (ge != 0u)
            v.active[atomicAdd(&v.ctl->n_active, 1u)] =
                make_int4(sg.row[lane], static_cast<int>(ge & 0xFFFFu), static_cast<int>(ge >> 16), 0);
    }
}

// A warp per active row (most batches; one problem of up to 1024 matches):
// lane l reads chunks 4l .. 4l + 3 of each 128-chunk sweep (lane order =
// column order), the next sweep in flight, and needs no block barrier.  A
// block's eight rows then run side by side: with a block per row and n/8
// blocks, a problem whose rows are all active took eight rows in turn (10.5 us
// at n = 67), and a batch's blocks mostly started for nothing (256 problems:
// 613 us, so 136, measured as the count pass above).  Same slots and tie ranks as the block form below.
template <class VS>
__global__ void __launch_bounds__(256) emit_warp_kernel(VS vs)
{
    int lb;
    const ProbView v = vs.get(ST_EMIT, blockIdx.x, lb);   // launch descriptors: before the wait
    pdl_wait();
    pdl_release();
    const int lane = threadIdx.x & 31;
    const int n = v.n, eb = emit_blocks(n, v.emit_few);
    const int a0 = (threadIdx.x >> 5) * eb + lb;          // this warp's first active row
    const int n_sel = v.ctl->n_sel;
    const int nact = static_cast<int>(v.ctl->n_active);
    const int m = v.ctl->m_ties, alpha = v.ctl->alpha, c_gt = v.ctl->c_gt;
    int4 ar = a0 < n ? v.active[a0] : make_int4(0, 0, 0, 0);   // speculative: a0 < n is inside the list's capacity
    if (n_sel == 0) return;
    const int c1 = (n - 1) >> 3;
    for (int a = a0; a < nact; a += 8 * eb) {
        if (a != a0) ar = v.active[a];
        const int i = ar.x, ng = ar.y, ne = ar.z;
        const uint16_t* wrow = v.w + (size_t)i * v.n_pad;
        const int cb0 = (i + 1) >> 3;
        uint4 q[4];
        auto load = [&](int cb) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int cc = cb + lane * 4 + k;
                q[k] = cc <= c1 ? *reinterpret_cast<const uint4*>(wrow + cc * 8) : make_uint4(0u, 0u, 0u, 0u);
            }
        };
        load(cb0);
        int base_g = 0;
        if (lane == 0 && ng > 0) base_g = static_cast<int>(atomicAdd(&v.ctl->gt_slot, static_cast<uint32_t>(ng)));
        int base_e = 0;   // ties in active rows above i
        if (ne > 0) {
            for (int b = lane; b < nact; b += 32) {
                const int4 o = v.active[b];
                base_e += o.x < i ? o.z : 0;
            }
            base_e = __reduce_add_sync(0xffffffffu, base_e);
        }
        int left_e = base_e < m ? min(ne, m - base_e) : 0, left_g = ng;   // edges of this row still to write
        base_g = __shfl_sync(0xffffffffu, base_g, 0);
        for (int cb = cb0; cb <= c1 && (left_g > 0 || left_e > 0); cb += 128) {
            uint32_t gm = 0u, em = 0u;   // bit 8 k + e: chunk k, element e
            const int cfirst = cb + lane * 4;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (!chunk_reaches(q[k], alpha)) continue;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const uint32_t word = e < 2 ? q[k].x : e < 4 ? q[k].y : e < 6 ? q[k].z : q[k].w;
                    const int j = (cfirst + k) * 8 + e;
                    const bool in = j > i && j < n;
                    const int w = in ? pivot_weight(v, i, j, (word >> ((e & 1) * 16)) & 0xFFFF) : 0;
                    gm |= static_cast<uint32_t>(in && w > alpha) << (8 * k + e);
                    em |= static_cast<uint32_t>(in && w == alpha) << (8 * k + e);
                }
            }
            if (cb + 128 <= c1) load(cb + 128);
            // inclusive prefix sums of both counts over the lanes (at most 32 x 32 each)
            const uint32_t own = static_cast<uint32_t>(__popc(gm)) | (static_cast<uint32_t>(__popc(em)) << 16);
            uint32_t incl = own;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += y;
            }
            const uint32_t tot = __shfl_sync(0xffffffffu, incl, 31), excl = incl - own;
            int rg = base_g + static_cast<int>(excl & 0xFFFFu), re = static_cast<int>(excl >> 16);
            for (; gm; gm &= gm - 1u) {
                const int b = __ffs(gm) - 1;
                const int j = (cfirst + (b >> 3)) * 8 + (b & 7);
                v.cand[rg++] = edge_key(pivot_weight(v, i, j, wrow[j]), i, j, n);
            }
            for (; em && re < left_e; em &= em - 1u, ++re) {
                const int b = __ffs(em) - 1;
                v.cand[c_gt + base_e + re] = edge_key(alpha, i, (cfirst + (b >> 3)) * 8 + (b & 7), n);
            }
            base_g += static_cast<int>(tot & 0xFFFFu);
            left_g -= static_cast<int>(tot & 0xFFFFu);
            base_e += static_cast<int>(tot >> 16);
            left_e -= static_cast<int>(tot >> 16);
        }
    }
}

// A block per active row (one or a few larger problems: a row is read in one or
// two rounds).  Blocks take the active rows in any order.  W > alpha edges take slots
// base + rank-in-row from one atomic per row (any slots in [0, c_gt) will
// do: the rank pass orders the keys).  Ties must be the m lowest (i, j):
// a row with ties sums the tie counts of the active rows above it (its tie
// prefix) and keeps tie ranks prefix + rank-in-row < m.  Thread t reads
// chunks 4t .. 4t+3 of each 1024-chunk sweep (thread order = column order).
// The block's first active row is read speculatively in the same round as
// the counters, and the row's first sweep, its tie prefix and its slot
// atomic go out together in the next.
template <class VS>
__global__ void __launch_bounds__(256) emit_kernel(VS vs)
{
    int lb;
    const ProbView v = vs.get(ST_EMIT, blockIdx.x, lb);   // launch descriptors: before the wait
    pdl_wait();
    pdl_release();
    __shared__ int sg[8], se[8];
    __shared__ int s_base;
    // the counters through L1: every warp of every block reads them
    const int n_sel = v.ctl->n_sel;
    const int nact = static_cast<int>(v.ctl->n_active);
    const int m = v.ctl->m_ties, alpha = v.ctl->alpha;
    const int4 ar0 = v.active[lb];                  // lb < n_pad: inside the list's capacity
    if (n_sel == 0) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c1 = (v.n - 1) >> 3;
    const int eb = emit_blocks(v.n, 0);
    for (int a = lb; a < nact; a += eb) {
        const int4 ar = a == lb ? ar0 : v.active[a];
        const int i = ar.x, ng = ar.y, ne = ar.z;
        const uint16_t* wrow = v.w + (size_t)i * v.n_pad;
        // first sweep of the row
        const int cb0 = (i + 1) >> 3;
        uint4 q[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int cc = cb0 + threadIdx.x * 4 + k;
            q[k] = cc <= c1 ? *reinterpret_cast<const uint4*>(wrow + cc * 8) : make_uint4(0u, 0u, 0u, 0u);
        }
        // slots of the W > alpha edges
        if (threadIdx.x == 0)
            s_base = ng > 0 ? static_cast<int>(atomicAdd(&v.ctl->gt_slot, static_cast<uint32_t>(ng))) : 0;
        // tie prefix: ties in active rows above i
        int pe = 0;
        if (ne > 0) {
            int part = 0;
            for (int b = threadIdx.x; b < nact; b += blockDim.x) {
                const int4 o = v.active[b];
                part += o.x < i ? o.z : 0;
            }
#pragma unroll
            for (int off = 16; off >= 1; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
            if (lane == 0) se[warp] = part;
            __syncthreads();
            for (int w8 = 0; w8 < 8; ++w8) pe += se[w8];
        }
        __syncthreads();
        const bool want_eq = ne > 0 && pe < m;
        if (ng == 0 && !want_eq) continue;   // uniform over the block
        const int pg = s_base;
        const int c_gt = v.ctl->c_gt;
        int base_g = pg, base_e = pe;
        for (int cb = cb0; cb <= c1; cb += blockDim.x * 4) {
            uint32_t gm = 0, em = 0;   // bit 8*k + e: chunk k, element e
            const int cfirst = cb + threadIdx.x * 4;
            if (cb != cb0) {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    q[k] = cfirst + k <= c1 ? *reinterpret_cast<const uint4*>(wrow + (cfirst + k) * 8)
                                            : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (!chunk_reaches(q[k], alpha)) continue;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const uint32_t word = e < 2 ? q[k].x : e < 4 ? q[k].y : e < 6 ? q[k].z : q[k].w;
                    const int j = (cfirst + k) * 8 + e;
                    const bool in = j > i && j < v.n;
                    const int w = in ? pivot_weight(v, i, j, (word >> ((e & 1) * 16)) & 0xFFFF) : 0;
                    gm |= static_cast<uint32_t>(in && w > alpha) << (8 * k + e);
                    em |= static_cast<uint32_t>(in && w == alpha) << (8 * k + e);
                }
            }
            // block exclusive scans of the two counts (thread order = column order)
            const int g = __popc(gm), eN = __popc(em);
            int gi = g, ei = eN;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int x = __shfl_up_sync(0xffffffffu, gi, off);
                const int y = __shfl_up_sync(0xffffffffu, ei, off);
                if (lane >= off) { gi += x; ei += y; }
            }
            if (lane == 31) { sg[warp] = gi; se[warp] = ei; }
            __syncthreads();
            int wg = 0, we = 0, tg = 0, te = 0;
            for (int w8 = 0; w8 < 8; ++w8) {
                if (w8 < warp) { wg += sg[w8]; we += se[w8]; }
                tg += sg[w8];
                te += se[w8];
            }
            __syncthreads();
            int rg = base_g + wg + gi - g, re = base_e + we + ei - eN;
            while (gm) {
                const int b = __ffs(gm) - 1;
                gm &= gm - 1;
                const int j = (cfirst + (b >> 3)) * 8 + (b & 7);
                v.cand[rg++] = edge_key(pivot_weight(v, i, j, wrow[j]), i, j, v.n);
            }
            while (em) {
                const int b = __ffs(em) - 1;
                em &= em - 1;
                if (re < m) v.cand[c_gt + re] = edge_key(alpha, i, (cfirst + (b >> 3)) * 8 + (b & 7), v.n);
                ++re;
            }
            base_g += tg;
            base_e += te;
            if (base_g - pg >= ng && (!want_eq || base_e >= m || base_e - pe >= ne)) break;
        }
    }
}

// Large batches: a problem's selected keys sorted in place, largest first (one
// block per problem, bitonic in shared memory), so that the clique search takes
// pivot c from key c.  Finding each key's rank there instead, one warp per key
// over all K1 keys, was 380 of the search's 2100 warp instructions per pivot;
// the sort takes 1/40 of that (but a launch more: pgs_dense has the line).  A
// pass of stride 32 or less stays inside the 64 keys of a warp.
__global__ void __launch_bounds__(1024) sort_kernel(ManyViews vs)
{
    const ProbView& v = vs.bt.views[blockIdx.x];   // launch descriptors: before the wait
    extern __shared__ uint64_t sk[];
    pdl_wait();
    pdl_release();
    const int cnt = v.ctl->n_sel;
    int P = 64;
    while (P < cnt) P <<= 1;
    for (int q = threadIdx.x; q < P; q += blockDim.x) sk[q] = q < cnt ? __ldcg(v.cand + q) : 0ull;
    __syncthreads();
    for (int k = 2; k <= P; k <<= 1) {
        for (int j = k >> 1; j >= 1; j >>= 1) {
            for (int q = threadIdx.x; q < P / 2; q += blockDim.x) {
                const int a = 2 * q - (q & (j - 1)), b = a + j;   // pair q of stride j
                const uint64_t x = sk[a], y = sk[b];
                if ((x < y) == ((a & k) == 0)) {
                    sk[a] = y;
                    sk[b] = x;
                }
            }
            if (j > 32 || (j == 1 && k >= 64)) __syncthreads();   // the next pass leaves the warp's 64 keys
            else __syncwarp();
        }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < cnt; q += blockDim.x) v.cand[q] = sk[q];
}

// 32 candidates per block (one per lane); the 8 warps split the comparison
// range; all n_sel keys of the problem are staged in shared memory.
__global__ void __launch_bounds__(256) rank_kernel(OneView vs, int32_t* n_out)
{
    int lb;
    const ProbView v = vs.get(ST_RANK, blockIdx.x, lb);
    pdl_wait();
    pdl_release();
    extern __shared__ uint64_t sk[];
    __shared__ int part[8][32];
    const int n_sel = v.ctl->n_sel;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lb == 0 && threadIdx.x == 0)
        *n_out = (v.ctl->err & TR_ERR_BAD_WEIGHT) != 0u ? -TURBOREG_ERR_INVALID_ARG : n_sel;
    if (lb * 32 >= n_sel) return;
    for (int q = threadIdx.x; q < n_sel; q += blockDim.x) sk[q] = v.cand[q];
    __syncthreads();
    const int e = lb * 32 + lane;
    const uint64_t key = (e < n_sel) ? sk[e] : ~0ull;
    const int chunk = (n_sel + 7) / 8;
    const int f0 = warp * chunk, f1 = min(n_sel, f0 + chunk);
    int cnt = 0;
#pragma unroll 8
    for (int f = f0; f < f1; ++f) cnt += sk[f] > key;
    part[warp][lane] = cnt;
    __syncthreads();
    if (warp == 0 && e < n_sel) {
        int rank = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) rank += part[w][lane];
        const uint32_t lin = 0xFFFFFFFFu - static_cast<uint32_t>(key & 0xFFFFFFFFull);
        const int i = static_cast<int>(lin / static_cast<uint32_t>(v.n));
        const int j = static_cast<int>(lin % static_cast<uint32_t>(v.n));
        v.piv[rank] = make_int4(i, j, static_cast<int>(key >> 32), 0);
    }
}

}  // namespace

cudaError_t topk_setup()
{
    cudaError_t e = cudaFuncSetAttribute(sort_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TURBOREG_K1_MAX * 8);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(rank_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TURBOREG_K1_MAX * 8);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(learned_hist_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                kHistSmemMaxBins * 4);
}

void launch_hist(const Batch& b, int total, int max_n, cudaStream_t s)
{
    if (max_n + 1 <= kHistSmemMaxBins)
        launch_pdl(learned_hist_kernel<true>, total, kCountThreads, (max_n + 1) * 4, s, ManyViews{b});
    else
        launch_pdl(learned_hist_kernel<false>, total, kCountThreads, 0, s, ManyViews{b});
}

void launch_select(const Batch& b, cudaStream_t s) { launch_pdl(select_kernel, b.num, 1024, 0, s, ManyViews{b}); }

void launch_count_emit(const Batch& b, const int32_t tot[kNumBatchStages], bool select_here, int max_n, int max_k1,
                       cudaStream_t s)
{
    const ManyViews vs{b};
    if (count_by_warp(b.num)) {
        launch_pdl(count_warp_kernel, tot[ST_COUNT], 256, 0, s, vs);
    } else {
        const size_t stage = select_here ? static_cast<size_t>((max_n + 4) / 4 * 4) * 4 : 0;
        launch_pdl(count_kernel<ManyViews>, tot[ST_COUNT], kCountThreads, stage, s, vs, select_here ? 1 : 0);
    }
    if (emit_by_warp(b.num, max_n)) launch_pdl(emit_warp_kernel<ManyViews>, tot[ST_EMIT], 256, 0, s, vs);
    else launch_pdl(emit_kernel<ManyViews>, tot[ST_EMIT], 256, 0, s, vs);
    if (pgs_dense(b.num, tot[ST_PGS], device_sms())) {
        int cap = 64;
        while (cap < max_k1) cap <<= 1;
        launch_pdl(sort_kernel, b.num, cap / 2 < 1024 ? cap / 2 : 1024, static_cast<size_t>(cap) * 8, s, vs);
    }
}

// One problem passed by value (no device-side problem table); the count blocks
// choose the threshold (n <= 8192: the histogram fits in 48 KB).
void launch_topk_single(const ProbView& v, int32_t* n_out, cudaStream_t s)
{
    const OneView vs{v};
    const int warps = (v.n + 1) / 2 * caller_windows(v.n), sms = device_sms();
    launch_pdl(caller_hist_kernel, (warps + 31) / 32 < sms ? (warps + 31) / 32 : sms, 1024, (v.n + 1) * 4, s, vs);
    launch_pdl(count_kernel<OneView>, count_groups(v.n), kCountThreads, static_cast<size_t>((v.n + 4) / 4 * 4) * 4, s,
               vs, 1);
    if (emit_by_warp(1, v.n)) launch_pdl(emit_warp_kernel<OneView>, emit_blocks(v.n, 0), 256, 0, s, vs);
    else launch_pdl(emit_kernel<OneView>, emit_blocks(v.n, 0), 256, 0, s, vs);
    launch_pdl(rank_kernel, (v.k1 + 31) / 32, 256, v.k1 * 8, s, vs, n_out);
}

}  // namespace tr
