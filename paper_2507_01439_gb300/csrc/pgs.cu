// Stage 4: Pivot-Guided Search (Eq. 5-7, Alg. 1) on the O2Graph or on the
// undirected SC^2 graph.
//
// O2Graph (Def. 2), pivot p = (i, j) (i < j):
//   N(i,j) = { z : G~_iz > 0 and G~_jz > 0 }            (Eq. 5)
// On the O2Graph G~_iz > 0 needs i < z, so z > j; and for a pivot edge,
// G~_iz > 0 <=> G_iz = 1 (j is then a common neighbour of i and z).  So
//   N(i,j) = { z > j : G_iz = G_jz = 1 } = bits of (row_i AND row_j) above j.
//   S(z)   = W_ij + W_iz + W_jz                          (Eq. 6)
// and the K2 largest S (ties: lower z) form the pivot's TurboCliques (Eq. 7),
// written in the Alg. 2 layout h = r * |P| + p.  Empty slots are invalid.
// Undirected SC^2 graph: the same with z over every common neighbour
// (z != i, j follows from the zero diagonal) and W read symmetrically,
// W_ab = W_min(a,b),max(a,b) (only the upper triangle is stored).
//
// One warp per selected edge (Eq. 4).  One problem or a small batch: in the order
// the selection wrote them; the warp first finds the edge's pivot index, its rank
// among the selected keys (staged once per block in shared memory).  A large batch: the keys
// are sorted, so edge c is pivot c.  All outputs go to the pivot index.
// Candidates: every lane loads its share of both rows' bitset words at once
// (eight words of each per lane in flight), and the warp compacts the set bits
// of their AND into a per-warp list in shared memory (popcount prefix sums).
// Scoring: lanes take list entries l, l + 32, ..., eight at a time so that
// their 16 weight loads are in flight together (sixteen at a time measured
// slower), and keep private top-K2 lists of 32-bit keys S << 15 | ~z (S is
// below 3 * 2^15, z below 2^15); the warp merges the 32 lists with K2 warp-wide
// maxima.  A list that would overflow is scored and emptied first, so any graph
// density works.
//
// Kabsch (Sec. 3.5): one lane per clique in FP32; for ill-conditioned cliques
// the warp computes the FP64 triangle normals with six lanes per clique
// (triangle x or y, component 0..2) and the clique's lane redoes the closed
// form with them.  One problem or a small batch: each warp solves its own pivot's
// cliques at once.  A large batch: a kernel of its own solves 32 cliques to a warp, and the search,
// bound by the latency of its gathers, keeps twice the warps per SM without
// the closed form's registers.
#include <type_traits>

#include "tr_common.cuh"
#include "tr_kabsch.cuh"
#include "tr_problem.h"

namespace tr {

namespace {

constexpr int kCand = 1024;   // per-warp candidate list (z indices, 16 bits)
constexpr int kListBytes = 8 * kCand * 2;   // the 8 warps' lists
constexpr int kWords = 8;     // bitset words per lane per load round
constexpr int kBatch = 8;     // list entries per lane per scoring round (16 weight loads in flight)

// Kabsch of the lanes' cliques: cl = (i, j, z, valid), h their hypothesis
// numbers, has: whether this lane has one (lanes below `lanes` at most).
__device__ __forceinline__ void solve_cliques(const ProbView& v, int4 cl, int h, bool has, int lanes)
{
    const int lane = threadIdx.x & 31;
    float P[3][3], Q[3][3];
    KabschOut o;
    o.ok = false;
    bool need = false;
    const bool present = has && cl.w != 0;
    if (present) {
        load_clique(v, cl, P, Q);
        kabsch3(P, Q, o);
        need = !(o.ok && o.kappa <= v.kappa_fp64);
    }
    const uint32_t needm = __ballot_sync(0xffffffffu, need);
    if (needm != 0u) {
        // FP64 normals, five cliques per round: lane L works for clique
        // base + L / 6, triangle (L / 3) & 1 (x, y), component L % 3
        float nx[3] = {0.f, 0.f, 0.f}, ny[3] = {0.f, 0.f, 0.f};
        for (int base = 0; base < lanes && (needm >> base) != 0u; base += 5) {
            if (((needm >> base) & 31u) == 0u) continue;
            const int r = base + lane / 6;
            const int src = r < 32 ? r : 31;
            const int idx[3] = {__shfl_sync(0xffffffffu, cl.x, src), __shfl_sync(0xffffffffu, cl.y, src),
                                __shfl_sync(0xffffffffu, cl.z, src)};
            const bool act = lane < 30 && r < lanes && ((needm >> src) & 1u);
            float val = 0.f;
            if (act) {
                const int tri = (lane / 3) & 1, comp = lane % 3;
                float T3[3][3];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const float* pt = v.pts8 + (size_t)idx[a] * 8 + 3 * tri;
                    T3[a][0] = pt[0]; T3[a][1] = pt[1]; T3[a][2] = pt[2];
                }
                val = exact_normal_comp(T3, comp);
            }
            // lane r of this round collects its six components from lanes 6 (r - base) ..
            const int mine0 = 6 * (lane - base);
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const int from = (lane >= base && lane < base + 5) ? mine0 + k : 0;
                const float g = __shfl_sync(0xffffffffu, val, from);
                if (lane >= base && lane < base + 5) {
                    if (k < 3) nx[k] = g;
                    else ny[k - 3] = g;
                }
            }
        }
        if (need) kabsch3<true>(P, Q, o, nx, ny);
    }
    if (has) store_hypothesis(v, h, present, o, need ? 2u : 0u);
}

// Kabsch of a large batch's cliques, a lane each.
__global__ void __launch_bounds__(128) solve_kernel(ManyViews vs)
{
    int lb;
    const ProbView v = vs.get(ST_KABSCH, blockIdx.x, lb);   // launch descriptors: before the wait
    pdl_wait();
    pdl_release();
    const int h = lb * 128 + static_cast<int>(threadIdx.x);
    const bool has = h < v.ctl->n_pivots * v.k2;
    if (!__any_sync(0xffffffffu, has)) return;
    solve_cliques(v, has ? v.cliques[h] : make_int4(0, 0, 0, 0), h, has, 32);
}

// kDense: a large batch (keys sorted, cliques solved by solve_kernel, registers
// bounded for four blocks per SM: many waves of blocks, latency hidden by
// occupancy); otherwise two blocks, with more registers per warp (one problem:
// a single wave)
template <int K2C, bool kDense>
__global__ void __launch_bounds__(256, kDense ? 4 : 2) pgs_kernel(ManyViews vs)
{
    // dynamic shared memory: per-warp candidate lists, then the selected edge keys (unless dense)
    extern __shared__ __align__(16) uint8_t pgs_smem[];
    uint16_t (*scand)[kCand] = reinterpret_cast<uint16_t (*)[kCand]>(pgs_smem);
    uint64_t* skey = reinterpret_cast<uint64_t*>(pgs_smem + kListBytes);
    int lb;
    const ProbView v = vs.get(ST_PGS, blockIdx.x, lb);   // launch descriptors: before the wait
    pdl_wait();
    pdl_release();   // the balanced verification tile caps itself at four blocks per SM, so
                     // blocks placed beside these still end up evenly spread
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the selected edges (Eq. 4); keys W << 32 | ~(i n + j) are unique, larger =
    // heavier, then lower (i, j), and a pivot's index is its rank, the number of
    // larger keys.  Unless dense, all K1 key slots are staged in the same round of
    // loads as the number of selected edges (the selection fills the first
    // n_sel; the rest are ignored).
    const int np = v.ctl->n_sel;   // through L1: every warp of every block reads it
    const int kcap = v.k1;
    // warp w of block b takes selected edge w * blocks + b; dense:
    // 8 b + w, so that a block's pivots share rows more often
    const int c = kDense ? lb * 8 + warp : warp * ((kcap + 7) / 8) + lb;
    const uint64_t mykey = c < kcap ? __ldcg(v.cand + c) : 0ull;
    for (int q0 = threadIdx.x; !kDense && q0 < kcap; q0 += 8 * static_cast<int>(blockDim.x)) {
        uint64_t kk[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int q = q0 + u * static_cast<int>(blockDim.x);
            kk[u] = q < kcap ? __ldcg(v.cand + q) : 0ull;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int q = q0 + u * static_cast<int>(blockDim.x);
            if (q < kcap) skey[q] = kk[u];
        }
    }
    if (lb == 0 && threadIdx.x == 0) v.ctl->n_pivots = np;
    const uint32_t lin = 0xFFFFFFFFu - static_cast<uint32_t>(mykey & 0xFFFFFFFFull);
    const int i = c < np ? static_cast<int>(lin / static_cast<uint32_t>(v.n)) : 0;
    const int j = c < np ? static_cast<int>(lin % static_cast<uint32_t>(v.n)) : 0;
    const int wij = static_cast<int>(mykey >> 32);
    const bool undirected = v.graph_mode == TURBOREG_GRAPH_SC2;
    const uint32_t* bi = v.bits + (size_t)i * v.ldb;
    const uint32_t* bj = v.bits + (size_t)j * v.ldb;
    // the first round of this pivot's bitset words, in flight across the
    // block barrier and the rank count
    const int zs = undirected ? 0 : j + 1;
    const int w0 = zs >> 5;
    uint32_t mw0[kWords];
#pragma unroll
    for (int t = 0; t < kWords; ++t) {
        const int wd = w0 + lane + 32 * t;
        mw0[t] = (c < np && wd < v.ldb) ? (__ldg(bi + wd) & __ldg(bj + wd)) : 0u;
    }
    const int k2 = K2C > 0 ? K2C : v.k2;
    int p = c;
    if constexpr (kDense) {
        if (c >= np) return;
    } else {
        __syncthreads();
        if (c >= np) return;
        p = 0;
        for (int q = lane; q < np; q += 32) p += skey[q] > mykey ? 1 : 0;
        p = __reduce_add_sync(0xffffffffu, p);
    }
    uint16_t* cand = scand[warp];
    const uint16_t* wi = v.w + (size_t)i * v.n_pad;
    const uint16_t* wj = v.w + (size_t)j * v.n_pad;

    constexpr int L = K2C > 0 ? K2C : TURBOREG_K2_MAX;
    static_assert(TURBOREG_MAX_N <= 32768, "S in 17 bits and z in 15");
    uint32_t top[L];
#pragma unroll
    for (int r = 0; r < L; ++r) top[r] = 0u;   // no key is 0: W_ij > 0

    auto insert = [&](int z, int wa, int wb) {   // into the descending list (keys are unique)
        uint32_t cur = (static_cast<uint32_t>(wij + wa + wb) << 15) | (32767u - static_cast<uint32_t>(z));
        if (L > 4 && cur <= top[L - 1]) return;
#pragma unroll
        for (int r = 0; r < L; ++r) {
            const uint32_t t = min(top[r], cur);
            top[r] = max(top[r], cur);
            cur = t;
        }
    };
    // score list entries [0, cnt): W_iz and W_jz of the z above j (rows i and j of W)
    // (apart from the column reads below: with both in one loop, whose selects and
    // addresses served either, the search took 650 us instead of 456 for 256
    // problems and 17.6 instead of 12 at N = 5000)
    auto score_rows = [&](int cnt) {
        for (int c0 = 0; c0 < cnt; c0 += 32 * kBatch) {
            int zq[kBatch], wa[kBatch], wb[kBatch];
#pragma unroll
            for (int b = 0; b < kBatch; ++b) {
                const int c = c0 + lane + 32 * b;
                zq[b] = c < cnt ? cand[c] : -1;
            }
#pragma unroll
            for (int b = 0; b < kBatch; ++b) {
                const int z = zq[b];
                wa[b] = z <= j ? 0 : static_cast<int>(wi[z]);
                wb[b] = z <= j ? 0 : static_cast<int>(wj[z]);
            }
#pragma unroll
            for (int b = 0; b < kBatch; ++b)
                if (zq[b] > j) insert(zq[b], wa[b], wb[b]);
        }
    };
    // The undirected search also meets z < j and reads W symmetrically, down a
    // column, a cache line per entry (41 us of clique search at N = 4333 and 13 %
    // density; 33 with the bound below).  Only entries that can still reach the
    // pivot's K2 best are read: W_iz and W_jz with z below are bounded by row
    // z's largest weight (and W_iz with z above i by row i's), and the K2-th of
    // the lanes' best keys so far bounds the K2-th best clique from below.  An
    // entry is left out only when its bound is strictly below, so ties stay.
    auto score_columns = [&](int cnt) {
        uint32_t thr = 0u, h = top[0];
        for (int r = 0; r < k2; ++r) {
            thr = __reduce_max_sync(0xffffffffu, h);
            if (h == thr) h = 0u;   // keys are unique: one lane (all of them at 0)
        }
        const int need = static_cast<int>(thr >> 15) - wij;
        const int rmi = v.rowmax[i];
        for (int c0 = 0; c0 < cnt; c0 += 32 * kBatch) {
            int zq[kBatch], wa[kBatch], wb[kBatch];
#pragma unroll
            for (int b = 0; b < kBatch; ++b) {
                const int c = c0 + lane + 32 * b;
                zq[b] = c < cnt ? cand[c] : -1;
                if (zq[b] > j) zq[b] = -1;
            }
#pragma unroll
            for (int b = 0; b < kBatch; ++b) wa[b] = zq[b] < 0 ? 0 : v.rowmax[zq[b]];
#pragma unroll
            for (int b = 0; b < kBatch; ++b)
                if ((zq[b] > i ? rmi : wa[b]) + wa[b] < need) zq[b] = -1;
#pragma unroll
            for (int b = 0; b < kBatch; ++b) {
                const int z = zq[b];
                wa[b] = z < 0 ? 0 : static_cast<int>(z > i ? wi[z] : v.w[(size_t)z * v.n_pad + i]);
                wb[b] = z < 0 ? 0 : static_cast<int>(v.w[(size_t)z * v.n_pad + j]);
            }
#pragma unroll
            for (int b = 0; b < kBatch; ++b)
                if (zq[b] >= 0) insert(zq[b], wa[b], wb[b]);
        }
    };
    auto score = [&](int cnt) {
        score_rows(cnt);
        if (undirected) score_columns(cnt);
    };

    // this pivot's cliques: lane r < k2 returns clique r
    auto search = [&]() {
        if (lane == 0) v.piv[p] = make_int4(i, j, wij, 0);
        int nlist = 0;
        for (int wb = w0; wb < v.ldb; wb += 32 * kWords) {
            uint32_t mw[kWords];
#pragma unroll
            for (int t = 0; t < kWords; ++t) {
                const int wd = wb + lane + 32 * t;
                mw[t] = wb == w0 ? mw0[t] : wd < v.ldb ? (__ldg(bi + wd) & __ldg(bj + wd)) : 0u;
                if (wd == w0) mw[t] &= ~0u << (zs & 31);
            }
            // one prefix sum per round: lane l writes its candidates (all its words)
            // after those of lanes < l; the list order does not matter
            int cnt = 0;
#pragma unroll
            for (int t = 0; t < kWords; ++t) cnt += __popc(mw[t]);
            int incl = cnt;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += y;
            }
            const int total = __shfl_sync(0xffffffffu, incl, 31);
            if (nlist + total <= kCand) {
                int pos = nlist + incl - cnt;
#pragma unroll
                for (int t = 0; t < kWords; ++t) {
                    const int zb = (wb + lane + 32 * t) * 32;
                    for (uint32_t m = mw[t]; m != 0u; m &= m - 1u) cand[pos++] = static_cast<uint16_t>(zb + __ffs(m) - 1);
                }
                nlist += total;
            } else {
                // dense rows: word by word, scoring the list whenever it would overflow
#pragma unroll 1
                for (int t = 0; t < kWords; ++t) {
                    const int c1 = __popc(mw[t]);
                    int in1 = c1;
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
                        const int y = __shfl_up_sync(0xffffffffu, in1, off);
                        if (lane >= off) in1 += y;
                    }
                    const int tot1 = __shfl_sync(0xffffffffu, in1, 31);
                    if (nlist + tot1 > kCand) {   // warp-uniform
                        __syncwarp();
                        score(nlist);
                        nlist = 0;
                        __syncwarp();
                    }
                    int pos = nlist + in1 - c1;
                    const int zb = (wb + lane + 32 * t) * 32;
                    for (uint32_t m = mw[t]; m != 0u; m &= m - 1u) cand[pos++] = static_cast<uint16_t>(zb + __ffs(m) - 1);
                    nlist += tot1;
                }
            }
        }
        __syncwarp();
        score(nlist);

        // warp merge: k2 rounds of argmax over the lanes' list heads; lane r keeps
        // round r's clique
        int head = 0;
        int4 mine_cl = make_int4(i, j, -1, 0);
        for (int r = 0; r < k2; ++r) {
            uint32_t mine = 0u;
#pragma unroll
            for (int q = 0; q < L; ++q)
                if (q == head) mine = top[q];
            const uint32_t best = __reduce_max_sync(0xffffffffu, mine);
            if (best == mine && mine != 0u) ++head;
            const int4 cl = best != 0u ? make_int4(i, j, 32767 - static_cast<int>(best & 32767u), 1) : make_int4(i, j, -1, 0);
            if (lane == 0) v.cliques[static_cast<size_t>(r) * np + p] = cl;
            if (lane == r) mine_cl = cl;
        }
        return mine_cl;
    };
    const int4 cl = search();
    if (!kDense) solve_cliques(v, cl, lane * np + p, lane < k2, k2);
}

}  // namespace

cudaError_t pgs_setup()
{
    cudaError_t e = cudaSuccess;
    const void* fns[] = {
        reinterpret_cast<const void*>(pgs_kernel<0, false>), reinterpret_cast<const void*>(pgs_kernel<1, false>),
        reinterpret_cast<const void*>(pgs_kernel<2, false>), reinterpret_cast<const void*>(pgs_kernel<3, false>),
        reinterpret_cast<const void*>(pgs_kernel<4, false>), reinterpret_cast<const void*>(pgs_kernel<0, true>),
        reinterpret_cast<const void*>(pgs_kernel<1, true>),  reinterpret_cast<const void*>(pgs_kernel<2, true>),
        reinterpret_cast<const void*>(pgs_kernel<3, true>),  reinterpret_cast<const void*>(pgs_kernel<4, true>)};
    for (const void* f : fns) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     kListBytes + TURBOREG_K1_MAX * static_cast<int>(sizeof(uint64_t)));
    }
    return e;
}

// k2 is the common K2 of the batch, or 0 when problems differ (generic list);
// max_k1 sizes the shared copy of the selected keys
void launch_pgs(const Batch& b, const int32_t tot[kNumBatchStages], int k2, int max_k1, cudaStream_t s)
{
    const int total = tot[ST_PGS];
    auto go = [&](auto dense) {
        constexpr bool kD = decltype(dense)::value;
        const ManyViews vs{b};
        const size_t smem = kListBytes + (kD ? 0 : static_cast<size_t>(max_k1) * sizeof(uint64_t));
        switch (k2) {
            case 1: launch_pdl(pgs_kernel<1, kD>, total, 256, smem, s, vs); break;
            case 2: launch_pdl(pgs_kernel<2, kD>, total, 256, smem, s, vs); break;
            case 3: launch_pdl(pgs_kernel<3, kD>, total, 256, smem, s, vs); break;
            case 4: launch_pdl(pgs_kernel<4, kD>, total, 256, smem, s, vs); break;
            default: launch_pdl(pgs_kernel<0, kD>, total, 256, smem, s, vs); break;
        }
    };
    if (pgs_dense(b.num, total, device_sms())) {
        go(std::true_type{});
        launch_pdl(solve_kernel, tot[ST_KABSCH], 128, 0, s, ManyViews{b});
    } else {
        go(std::false_type{});
    }
}

cudaError_t verify_setup();

cudaError_t verify_pgs_setup()
{
    const cudaError_t e = verify_setup();
    return e == cudaSuccess ? pgs_setup() : e;
}

}  // namespace tr
