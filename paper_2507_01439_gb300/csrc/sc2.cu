// Stage 2: SC^2 graph (Eq. 2) restricted to the O2Graph (Def. 2).
//
//   W_ij = G_ij * sum_k G_ik G_jk  for i < j,   i.e.  W = triu(G .* (G G), 1)
//
// Main path: a binary GEMM on the 5th-generation tensor cores.  G is stored
// as packed FP4 (E2M1) 0/1 values; since G is symmetric, G G = G G^T, so both
// MMA operands are K-major row blocks of the same matrix.  The MMAs are the
// block-scaled FP4 kind with every block scale 1.0; products of 0/1 are exact
// and the FP32 accumulator holds integers <= N-2 < 2^24 exactly, so the
// result is the integer SC^2 count.  FP4 operands carry twice the products
// per byte and per tensor-core cycle of FP8 ones, and the kernel is bound by
// exactly these two (at the full MMA rate the operands stream from L2 at
// ~17 TB/s with either type).  Only output blocks that contain some i < j are
// computed (the upper triangle, about half the square).  Measured against the
// FP8 kernel it replaced: 3640 -> 1388 us at N = 20000 (where the histogram
// also moved to shared memory and the block order keeps the operand in L2),
// 48 -> 35 us at N = 4333 (13 % density), 2838 -> 2137 us for 256 problems
// of N = 500 .. 5000.
//
// Work: 256 x 256 output blocks (bm <= bn), taken by 2-CTA clusters as pair
// MMAs (cta_group::2, each CTA's shared memory holding its halves of A and B)
// or, on request, as two 128 x 256 halves by independent CTAs.
//   warp 0 lane 0  TMA producer: 128-byte-swizzled K-major tiles, 256 columns
//                  of K per stage, into a ring of 2 to 5 stages (as many as fit
//                  beside the histogram)
//   warp 1 lane 0  MMA issuer: tcgen05.mma kind::mxf4, N=256 K=64, 4 per stage
//   warps 2..17    epilogue of the previous block while the next one runs
//   warp 18        scheduler: the next blocks' descriptors
//
// Tensor memory (512 columns): two 256-column accumulators and 16 columns of
// block scales do not fit side by side, so the accumulators overlap in 16
// columns: buffer 0 at columns 0..255, buffer 1 at 240..495, scales at
// 496..511.  The epilogue warps that own the shared columns read them first
// and report it (`tover`); the next block's MMAs wait for that, not for the
// whole epilogue.
//
// Alternative (sc2_bitset.cu): the same integers from the adjacency bitset
// with AND + popcount on CUDA cores, work only on the edges.
#include <atomic>

#include "tr_common.cuh"
#include "tr_problem.h"
#include "tr_select.cuh"

namespace tr {

namespace {

constexpr int kHalf = kSc2BM * kSc2BK;     // 16 KB: 128 rows x 128 bytes of one operand
constexpr int kEpiWarps = 16;              // 4 per TMEM lane quarter, each a quarter of the columns
constexpr int kEpiCols = 4 * kSc2BN / kEpiWarps;   // 64 columns per epilogue warp
constexpr int kSchedWarp = 2 + kEpiWarps;  // hands out the blocks
constexpr int kThreads = 32 * (kSchedWarp + 1);
constexpr int kMaxStages = 5;
constexpr int kRing = 4;                   // block descriptors in flight
constexpr int kBarBytes = 1024;            // mbarriers, TMEM slot, block descriptors
constexpr int kColBytes = kEpiWarps * kEpiCols * 4;   // column sums of an epilogue warp's block
constexpr int kStgBytes = kEpiWarps * 2048;   // W staging: 32 x 32 uint16 per epilogue warp
constexpr int kSmemMax = 232448;           // 227 KB opt-in limit per block
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kAcc1 = 240;            // first column of accumulator 1 (16 shared with accumulator 0)
constexpr uint32_t kScaleCol = 496;        // block scales: A from 496 (4 columns), B from 500 (8 columns)
constexpr int kPanel = 8;                  // column blocks per panel of the block order

template <bool kPair>
constexpr int stage_bytes() { return (kPair ? 2 : 3) * kHalf; }   // this CTA's part of A and B per stage

// Block u of a problem with nb = n_pad / 256 column blocks.  Blocks are
// ordered in panels of eight column blocks, row by row inside a panel, so
// that the blocks in flight at any time cover a compact patch of the output:
// at N = 20000 one wave of 76 blocks reads 17 of the 79 row blocks of G
// instead of all of them, and the 200 MB operand is served from L2.
__device__ __forceinline__ void block_of(int u, int nb, int& bm, int& bn)
{
    // panel P holds the columns 8P .. and starts at block 8P (8P + 1) / 2
    int P = static_cast<int>((sqrtf(8.0f * static_cast<float>(u) + 1.0f) - 1.0f) * 0.5f) / kPanel;
    while (kPanel * P * (kPanel * P + 1) / 2 > u) --P;
    while (kPanel * (P + 1) * (kPanel * (P + 1) + 1) / 2 <= u) ++P;
    const int c0 = kPanel * P;
    const int w = min(kPanel, nb - c0);
    int r = u - c0 * (c0 + 1) / 2;
    if (r < c0 * w) {
        bm = r / w;
        bn = c0 + r % w;
        return;
    }
    r -= c0 * w;
    int k = 0;
    while (r >= w - k) {
        r -= w - k;
        ++k;
    }
    bm = c0 + k;
    bn = c0 + k + r;
}

// Block k of this worker (cluster or CTA `c` of `C`): chunks of `L`
// consecutive blocks, strided over the workers (a batch takes several blocks
// of one problem in a row, so that its histogram is flushed less often).
__device__ __forceinline__ int block_index(int k, int c, int C, int L)
{
    return (c + k / L * C) * L + k % L;
}

// One block as the scheduler warp hands it to the others: its problem (-1: no
// more blocks), this CTA's part of it, and the problem's fields they need.
struct BlockInfo {
    int32_t p, nk, row0, colb;
    int32_t n, n_pad, ldb, flush;   // flush: the worker's next block belongs to another problem
    const uint32_t* bits;
    uint16_t* w;
    int32_t* rowscore;
    int32_t* rowmax;
    uint32_t* hist;
    const CUtensorMap* map;         // 128-row boxes; + 1: 256-row boxes
};
static_assert(sizeof(BlockInfo) == 80 && kRing * sizeof(BlockInfo) + 256 <= kBarBytes, "block ring fits");

// The bitset words of an epilogue warp's columns, fetched a block ahead, so
// that their latency overlaps the previous block's epilogue and the MMAs.
__device__ __forceinline__ uint2 epi_words(const BlockInfo& v, int row, int col)
{
    static_assert(kEpiCols == 64, "one 8-byte bitset load per warp row");
    return *reinterpret_cast<const uint2*>(v.bits + (size_t)(v.row0 + row) * v.ldb + ((v.colb + col) >> 5));
}

// The warp's 2 KB staging area holds its 32 x 32 block of W: row r as four
// 16-byte chunks, chunk q at slot q ^ ((r >> 1) & 3), so that row-wise and
// column-wise accesses are both free of bank conflicts.
__device__ __forceinline__ uint32_t stg_slot(int r, int q) { return static_cast<uint32_t>(r * 4 + (q ^ ((r >> 1) & 3))); }

// Bits of each 16-bit half unshuffled: even positions into its low byte, odd
// ones into its high byte (three butterfly steps).
__device__ __forceinline__ uint32_t unshuffle16(uint32_t x)
{
    uint32_t t = (x ^ (x >> 1)) & 0x22222222u;
    x ^= t ^ (t << 1);
    t = (x ^ (x >> 2)) & 0x0C0C0C0Cu;
    x ^= t ^ (t << 2);
    t = (x ^ (x >> 4)) & 0x00F000F0u;
    return x ^ t ^ (t << 4);
}

// Bytes of x picked by sel, a nibble with bit 3 set replicating the byte's
// sign bit (__byte_perm ignores that bit).
__device__ __forceinline__ uint32_t sign_bytes(uint32_t x, uint32_t sel)
{
    uint32_t r;
    asm("prmt.b32 %0, %1, 0, %2;" : "=r"(r) : "r"(x), "r"(sel));
    return r;
}

// Arrival on a barrier given by its address in the cluster's (pair) or this CTA's shared window.
template <bool kPair>
__device__ __forceinline__ void arrive_at(uint32_t bar)
{
    if (kPair) mbar_arrive_cluster(bar);
    else mbar_arrive_addr(bar);
}

// Where an edge weight is counted: this CTA's bins, the pair's bins (a weight's
// bin lies in the CTA of its parity, at half its index), or the global ones.
enum HistForm { kHistGlobal, kHistCta, kHistPair };

// Epilogue of one warp's 32 rows x 64 columns whose FP32 accumulator is at
// TMEM address tacc: masks with the adjacency words and i < j, stores uint16
// W, adds row and column sums to the SC^2 row scores, row maxima, and counts
// the edge weights.
//   integers   adding 2^23 leaves an accumulator's integer in its low 16 bits
//              (exact: it is an integer below 2^16); a byte permute packs two,
//              and one that replicates sign bits turns two adjacency bits into
//              their mask
//   W store    pass k writes rows 8k .. 8k + 7, lane l chunk l % 4 of row
//              8k + l / 4: each instruction covers 8 x 64 contiguous bytes
//   the rest   each lane visits only the set bits of its adjacency word, two
//              at a time: row sum and maximum in registers, column sum and bin
//              by shared-memory additions.  (Sums over all 32 x 32 entries in
//              packed halves took ~250 more instructions per chunk; the warps
//              are bound by their own instruction chains, four per scheduler.)
// first / over: the 32-column chunk to take first, and the barrier (or 0) to
// report to once its accumulator columns are in registers; drained: the
// barrier to report to once both chunks are.
// bins0 / bins1: the bins of even and odd weights (kHistPair: cluster addresses).
template <bool kPair, HistForm kHist>
__device__ __forceinline__ void sc2_epilogue(const BlockInfo& v, uint32_t tacc, int row_off, int col_off, int lane,
                                             uint2 words, uint32_t* shist, uint32_t bins0, uint32_t bins1, uint4* stg,
                                             int* csum, int first, uint32_t over, uint32_t drained)
{
    const int row0 = v.row0 + row_off, col_w = v.colb + col_off;
    const int row = row0 + lane, n_pad = v.n_pad;
    uint16_t* const w = v.w;
    uint32_t rsum = 0u, rmax = 0u;
    uint32_t acc[32];
    tmem_ld32(tacc + static_cast<uint32_t>(first * 32), acc);
    tmem_ld_wait32(acc);
    if (over != 0u) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) arrive_at<kPair>(over);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        static_assert(kEpiCols == 64, "two 32-column chunks");
        const int c = k ^ first;
        const int col0 = col_w + c * 32;
        uint32_t word = c == 0 ? words.x : words.y;
        if (col0 + 31 <= row) word = 0u;                       // keep only j > row
        else if (col0 <= row) word &= ~0u << (row - col0 + 1);
        const uint32_t ub = unshuffle16(word);
        const f2 magic = pk(8388608.f, 8388608.f);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t h[4];
#pragma unroll
            for (int e4 = 0; e4 < 4; ++e4) {
                const int e = 4 * q + e4;
                const f2 s = add2(pk(__uint_as_float(acc[2 * e]), __uint_as_float(acc[2 * e + 1])), magic);
                // columns 2e, 2e + 1: bit e % 8 of the two bytes of half e / 8, moved to the bytes' sign bits
                const uint32_t m = sign_bytes(ub << (7 - (e & 7)), e < 8 ? 0x9988u : 0xBBAAu);
                h[e4] = __byte_perm(static_cast<uint32_t>(s.v), static_cast<uint32_t>(s.v >> 32), 0x5410u) & m;
            }
            stg[stg_slot(lane, q)] = make_uint4(h[0], h[1], h[2], h[3]);
        }
        if (k == 0) tmem_ld32(tacc + static_cast<uint32_t>((first ^ 1) * 32), acc);   // in flight through chunk 0's stores
        __syncwarp();
        // W rows, as full 64-byte segments
#pragma unroll
        for (int k4 = 0; k4 < 4; ++k4) {
            const int r = 8 * k4 + (lane >> 2), q = lane & 3;
            *reinterpret_cast<uint4*>(w + (size_t)(row0 + r) * n_pad + col0 + q * 8) = stg[stg_slot(r, q)];
        }
        // this lane's edges
        int* const cs = csum + c * 32;
        auto edge_w = [&](int q) { return static_cast<uint32_t>(reinterpret_cast<const uint16_t*>(stg + stg_slot(lane, q >> 3))[q & 7]); };
        auto count = [&](int q, uint32_t x) {
            if (x == 0u) return;
            atomicAdd(cs + q, static_cast<int>(x));
            if (kHist == kHistCta) atomicAdd(&shist[x], 1u);
            else if (kHist == kHistPair) red_add_cluster(((x & 1u) ? bins1 : bins0) + ((x >> 1) << 2), 1u);
            else atomicAdd(&v.hist[x], 1u);
        };
        for (uint32_t bits = word; bits != 0u;) {
            const int q0 = __ffs(bits) - 1;
            bits &= bits - 1u;
            const int q1 = bits != 0u ? __ffs(bits) - 1 : q0;
            const uint32_t x0 = edge_w(q0), y = edge_w(q1);
            const uint32_t x1 = bits != 0u ? y : 0u;
            bits &= bits - 1u;
            rsum += x0 + x1;
            rmax = max(rmax, max(x0, x1));
            count(q0, x0);
            count(q1, x1);
        }
        if (k == 0) {
            // the accumulator is read: its next block's MMAs may begin
            tmem_ld_wait32(acc);
            tc_fence_before();
        }
        __syncwarp();   // the next chunk overwrites the staging area; the column sums are complete
        if (k == 0 && lane == 0) arrive_at<kPair>(drained);
    }
    if (rsum != 0u) atomicAdd(&v.rowscore[row], static_cast<int>(rsum));
    if (rmax != 0u && v.rowmax) atomicMax(&v.rowmax[row], static_cast<int>(rmax));
    static_assert(kEpiCols == 64, "two columns per lane");
    const int2 cc = reinterpret_cast<const int2*>(csum)[lane];
    if ((cc.x | cc.y) != 0) {
        reinterpret_cast<int2*>(csum)[lane] = make_int2(0, 0);
        if (cc.x) atomicAdd(&v.rowscore[col_w + 2 * lane], cc.x);
        if (cc.y) atomicAdd(&v.rowscore[col_w + 2 * lane + 1], cc.y);
    }
    __syncwarp();   // the sums are cleared before the next block adds to them
}

// kPair: 2-CTA clusters with pair MMAs (M = 256 over both CTAs); else CTAs of
// their own take 128-row halves of the blocks.  kHist: the edge-weight
// histogram is kept in shared memory, per CTA or (one problem) split over the
// pair, and added to the global one when the worker leaves a problem (the
// count pass or the select launch then chooses the pivot threshold from it);
// else every edge adds to the global bins.  In a batch each CTA adds its own
// bins; for one problem a cluster's are merged in its first CTA before.
// The scheduler warp finds each block's problem and descriptor fields up to
// four blocks ahead and hands them over through a ring in shared memory: read
// by every role for itself, they were a chain of up to eight dependent loads
// in front of each block's loads, MMAs and epilogue.
//   pair: both CTAs' producers load their 128 rows of A and of B, counted on
//         the leader's `full` barrier; the leader issues the MMAs, whose commits
//         release the stage in both CTAs (`empty`) and hand each CTA its
//         accumulator (`tfull`); the epilogue warps of both CTAs arrive on the
//         leader's `tempty` and `tover`
// Every wait is bounded; before exit each producer waits for the last stage
// releases and a cluster synchronises, so no arrival targets a finished CTA.
// auto_mode: one problem whose SC^2 path the CUDA-core kernel before this one
// chose; when it chose itself, every CTA returns at once (before any set-up).
template <bool kPair, HistForm kHist>
__global__ void __launch_bounds__(kThreads, 1) sc2_mma_kernel(Batch bt, int total, int hist_bins, int nst, int chunk,
                                                              int auto_mode)
{
    if (auto_mode) {
        const Ctl* ctl = bt.views[0].ctl;   // the descriptor before the wait, the flag after it
        pdl_wait();
        if (__ldcg(&ctl->sc2_path) != 2u) {
            pdl_release();
            return;
        }
    }
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    constexpr int kBPart = kPair ? kHalf : 2 * kHalf;    // this CTA's bytes of B per stage
    uint8_t* sA = smem;                                  // [stage] 128 rows x 128 B
    uint8_t* sB = smem + nst * kHalf;                    // [stage] 128 or 256 rows x 128 B
    uint8_t* tail = smem + nst * stage_bytes<kPair>();
    uint64_t* full = reinterpret_cast<uint64_t*>(tail);
    uint64_t* empty = full + kMaxStages;
    uint64_t* tfull = empty + kMaxStages;    // [2] accumulator ready
    uint64_t* tempty = tfull + 2;            // [2] accumulator drained
    uint64_t* tover = tempty + 2;            // the columns both accumulators share are read
    uint64_t* hsync = tover + 1;             // epilogue warps: a problem's bins complete / flushed
    uint64_t* sfull = hsync + 1;             // [kRing] block descriptor written / consumed
    uint64_t* sempty = sfull + kRing;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sempty + kRing);
    static_assert((2 * kMaxStages + 6 + 2 * kRing) * 8 + 4 <= 256, "barriers before the block ring");
    BlockInfo* ring = reinterpret_cast<BlockInfo*>(tail + 256);
    uint4* stg = reinterpret_cast<uint4*>(tail + kBarBytes);
    int* csums = reinterpret_cast<int*>(tail + kBarBytes + kStgBytes);
    uint32_t* shist = reinterpret_cast<uint32_t*>(tail + kBarBytes + kStgBytes + kColBytes);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nbins = kHist != kHistGlobal ? hist_bins : 0;   // words of this CTA's bins
    const uint32_t rank = kPair ? cluster_ctarank() : 0u;
    const bool leader = rank == 0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < nst; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], (kPair ? 2 : 1) * kEpiWarps);
        }
        mbar_init(tover, (kPair ? 2 : 1) * 4);
        mbar_init(hsync, kEpiWarps);
        for (int b = 0; b < kRing; ++b) {
            mbar_init(&sfull[b], 1);
            mbar_init(&sempty[b], kEpiWarps + 1 + (leader ? 1 : 0));   // epilogue warps, producer, the leader's issuer
        }
        fence_mbar_init();
    }
    for (int b = threadIdx.x; b < nbins; b += blockDim.x) shist[b] = 0u;
    for (int b = threadIdx.x; b < kEpiWarps * kEpiCols; b += blockDim.x) csums[b] = 0;
    if (warp == 0) {
        if (kPair) tmem_alloc_pair(tmem_slot, kTmemCols);
        else tmem_alloc(tmem_slot, kTmemCols);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    if (warp >= 4 && warp < 8) {   // warps 4..7: TMEM lane quarters 0..3; every block scale is 1.0 (E8M0 127)
        tmem_st16(tmem + kScaleCol + (static_cast<uint32_t>((warp & 3) * 32) << 16), 0x7F7F7F7Fu);
        tmem_st_wait();
    }
    tc_fence_before();
    __syncthreads();
    if (kPair) cluster_sync_all();   // both CTAs' barriers and tensor memory are ready
    tc_fence_after();
    bool ok = true;
    // worker (cluster or CTA) c of C; a pair takes whole blocks, a CTA halves of them
    const int c = static_cast<int>(kPair ? blockIdx.x >> 1 : blockIdx.x);
    const int C = static_cast<int>(kPair ? gridDim.x >> 1 : gridDim.x);
    const int nu = kPair ? total >> 1 : total;
    const uint32_t full_l = kPair ? mapa_shared(&full[0], 0) : 0u;      // leader's barriers, cluster addresses
    const uint32_t tempty_l = kPair ? mapa_shared(&tempty[0], 0) : smem_u32(&tempty[0]);
    const uint32_t tover_l = kPair ? mapa_shared(tover, 0) : smem_u32(tover);
    // the set-up above (barriers, tensor memory, shared histogram) overlaps the
    // previous stage; its outputs are read only from here on
    pdl_wait();
    pdl_release();

    if (warp == 0) {
        if (lane == 0) {
            // ---------------- TMA producer ----------------
            int s = 0;
            uint32_t ph = 0u;
            for (int k = 0; ok; ++k) {
                if (!mbar_wait(&sfull[k % kRing], (k / kRing) & 1)) { ok = false; break; }
                const BlockInfo& bi = ring[k % kRing];
                const int p = bi.p, nk = bi.nk, row0 = bi.row0, colb = bi.colb;
                const CUtensorMap* mA = bi.map;
                mbar_arrive(&sempty[k % kRing]);
                if (p < 0) break;
                for (int kb = 0; kb < nk; ++kb) {
                    if (!mbar_wait(&empty[s], ph ^ 1u)) { ok = false; break; }
                    if (kPair) {
                        if (leader) mbar_arrive_expect_tx(&full[s], 4 * kHalf);   // both CTAs' A and B halves
                        const uint32_t bar = full_l + static_cast<uint32_t>(s * sizeof(uint64_t));
                        tma_load_2d_pair(sA + s * kHalf, mA, kb * kSc2BK, row0, bar);
                        tma_load_2d_pair(sB + s * kHalf, mA, kb * kSc2BK, colb + static_cast<int>(rank) * kSc2BM, bar);
                    } else {
                        mbar_arrive_expect_tx(&full[s], 3 * kHalf);
                        tma_load_2d(sA + s * kHalf, mA, kb * kSc2BK, row0, &full[s]);
                        tma_load_2d(sB + s * kBPart, mA + 1, kb * kSc2BK, colb, &full[s]);
                    }
                    if (++s == nst) { s = 0; ph ^= 1u; }
                }
            }
            // tail: the last releases of every stage have arrived here
            for (int q = 0; kPair && q < nst; ++q) {
                if (!mbar_wait(&empty[s], ph ^ 1u)) { ok = false; break; }
                if (++s == nst) { s = 0; ph ^= 1u; }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0 && leader) {
            // ---------------- MMA issuer (a pair's leader) ----------------
            constexpr uint32_t kIdesc = idesc_mxf4(kPair ? 2 * kSc2BM : kSc2BM, kSc2BN);
            const uint32_t sfa = tmem + kScaleCol, sfb = tmem + kScaleCol + 4;
            int s = 0;
            uint32_t ph = 0u;
            for (int k = 0; ok; ++k) {
                if (!mbar_wait(&sfull[k % kRing], (k / kRing) & 1)) { ok = false; break; }
                const int p = ring[k % kRing].p, nk = ring[k % kRing].nk;
                mbar_arrive(&sempty[k % kRing]);
                if (p < 0) break;
                const int buf = k & 1;
                const uint32_t use = static_cast<uint32_t>(k >> 1);
                // this accumulator drained, and the previous one's shared columns read
                if (!mbar_wait(&tempty[buf], (use & 1u) ^ 1u) ||
                    (k > 0 && !mbar_wait(tover, static_cast<uint32_t>(k - 1) & 1u))) { ok = false; break; }
                tc_fence_after();
                const uint32_t d = tmem + (buf ? kAcc1 : 0u);
                for (int kb = 0; kb < nk; ++kb) {
                    if (!mbar_wait(&full[s], ph)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t a0 = smem_u32(sA + s * kHalf);
                    const uint32_t b0 = smem_u32(sB + s * kBPart);
#pragma unroll
                    for (int q = 0; q < kSc2BK / 32; ++q)   // K = 64 FP4 (32 bytes) per MMA
                        mma_mxf4<kPair>(d, sdesc_k_sw128(a0 + q * 32), sdesc_k_sw128(b0 + q * 32), kIdesc, sfa, sfb,
                                        (kb | q) != 0 ? 1u : 0u);
                    if (kPair) mma_commit_pair_mc(&empty[s], 0x3);
                    else mma_commit(&empty[s]);
                    if (++s == nst) { s = 0; ph ^= 1u; }
                }
                if (!ok) break;
                if (kPair) mma_commit_pair_mc(&tfull[buf], 0x3);
                else mma_commit(&tfull[buf]);
            }
        }
        __syncwarp();
    } else if (warp == kSchedWarp) {
        // ---------------- scheduler ----------------
        const int32_t* pr = bt.pre + ST_GEMM * (bt.num + 1);
        int p = 0;
        for (int k = 0;; ++k) {
            const int u = block_index(k, c, C, chunk);
            const int slot = k % kRing;
            // failure injection (tests only): the first worker's second block is never handed out
            if (k == 1 && c == 0 && (bt.views[0].dbg & TR_DBG_STALL_SC2) != 0u) {
                ok = false;
                break;
            }
            if (k >= kRing && !__all_sync(0xffffffffu, mbar_wait(&sempty[slot], (k / kRing - 1) & 1))) {
                ok = false;
                break;
            }
            if (u >= nu) {
                if (lane == 0) {
                    ring[slot].p = -1;
                    mbar_arrive(&sfull[slot]);
                }
                break;
            }
            // the last problem that begins at or before this block (blocks only move forward)
            const int t = kPair ? 2 * u : u;
            for (int step = 32; step == 32; p += step)
                step = __popc(__ballot_sync(0xffffffffu, p + 1 + lane < bt.num && __ldg(pr + min(p + 1 + lane, bt.num)) <= t));
            if (lane == 0) {
                const ProbView& v = bt.views[p];
                const int un = block_index(k + 1, c, C, chunk);
                const int lt = t - __ldg(pr + p), nb = v.n_pad / kSc2BN;
                int bm, bn;
                block_of(lt >> 1, nb, bm, bn);
                BlockInfo bi;
                bi.p = p;
                bi.nk = nb;   // K stages of 256 columns
                bi.row0 = bm * kSc2BN + (kPair ? static_cast<int>(rank) : lt & 1) * kSc2BM;
                bi.colb = bn * kSc2BN;
                bi.n = v.n;
                bi.n_pad = v.n_pad;
                bi.ldb = v.ldb;
                bi.flush = un < nu && (kPair ? 2 * un : un) >= __ldg(pr + p + 1) ? 1 : 0;
                bi.bits = v.bits;
                bi.w = v.w;
                bi.rowscore = v.rowscore;
                bi.rowmax = v.rowmax;
                bi.hist = v.hist;
                bi.map = bt.maps + 2 * p;
                ring[slot] = bi;
                mbar_arrive(&sfull[slot]);
            }
            __syncwarp();
        }
    } else {
        // ---------------- epilogue warps ----------------
        const int quarter = warp & 3;              // TMEM lanes this warp may access
        const int part = (warp - 2) >> 2;          // column part of the block
        const uint32_t lane_off = static_cast<uint32_t>(quarter * 32) << 16;
        const int ro = quarter * 32, co = part * kEpiCols;
        const uint32_t bins0 = kHist == kHistPair ? mapa_shared(shist, 0) : 0u;
        const uint32_t bins1 = kHist == kHistPair ? mapa_shared(shist, 1) : 0u;
        uint2 words = make_uint2(0u, 0u);
        ok = __all_sync(0xffffffffu, mbar_wait(&sfull[0], 0u));
        if (ok && ring[0].p >= 0) words = epi_words(ring[0], ro + lane, co);
        for (int k = 0; ok; ++k) {
            const BlockInfo& v = ring[k % kRing];
            if (v.p < 0) break;
            // the next block's descriptor and adjacency words
            const BlockInfo& vn = ring[(k + 1) % kRing];
            if (!__all_sync(0xffffffffu, mbar_wait(&sfull[(k + 1) % kRing], ((k + 1) / kRing) & 1))) { ok = false; break; }
            uint2 words_n = make_uint2(0u, 0u);
            if (vn.p >= 0) words_n = epi_words(vn, ro + lane, co);
            const int buf = k & 1;
            const bool got = mbar_wait(&tfull[buf], static_cast<uint32_t>(k >> 1) & 1u);
            if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
            tc_fence_after();
            // the shared columns: the last 16 of accumulator 0, the first 16 of accumulator 1
            const bool owner = buf == 0 ? part == 3 : part == 0;
            sc2_epilogue<kPair, kHist>(v, tmem + (buf ? kAcc1 : 0u) + static_cast<uint32_t>(co) + lane_off, ro, co, lane,
                                       words, shist, bins0, bins1, stg + (warp - 2) * 128, csums + (warp - 2) * kEpiCols,
                                       buf == 0 && part == 3 ? 1 : 0, owner ? tover_l : 0u,
                                       tempty_l + static_cast<uint32_t>(buf * sizeof(uint64_t)));
            const bool flush = kHist == kHistCta && v.flush != 0;
            const int nf = v.n;
            uint32_t* const ghist = v.hist;
            __syncwarp();   // every lane's reads of the descriptor are done
            if (lane == 0) mbar_arrive(&sempty[k % kRing]);
            words = words_n;
            if (flush) {
                // the epilogue warps add this problem's bins to its global
                // histogram and clear them (a rendezvous before and after)
                if (lane == 0) mbar_arrive(hsync);
                if (!__all_sync(0xffffffffu, mbar_wait(hsync, 0u))) { ok = false; break; }
                for (int b = (warp - 2) * 32 + lane + 1; b <= nf; b += 32 * kEpiWarps) {
                    const uint32_t h = shist[b];
                    if (h) {
                        atomicAdd(ghist + b, h);
                        shist[b] = 0u;
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(hsync);
                if (!__all_sync(0xffffffffu, mbar_wait(hsync, 1u))) { ok = false; break; }
            }
        }
    }
    if (!ok && lane == 0) mark_timeout(bt);
    tc_fence_before();
    __syncthreads();
    // the problem of this worker's last block (both CTAs of a cluster take the
    // same blocks): its bins are still in shared memory
    int p_last = -1;
    if (c * chunk < nu) {
        const int nc = (nu + chunk - 1) / chunk;
        const int lc = c + (nc - 1 - c) / C * C;
        const int ul = min(nu, (lc + 1) * chunk) - 1;
        int lt;
        p_last = locate(bt, ST_GEMM, kPair ? 2 * ul : ul, lt);
    }
    // One problem: the peer's histogram into the leader's (distributed shared
    // memory), so that one CTA per cluster adds to the global bins.  Not in a
    // batch: the leader may still be emptying its bins of an earlier problem
    // (nothing orders its flush against the peer's end), so each CTA adds its own.
    const bool merge = kPair && kHist == kHistCta && bt.num == 1;
    if (merge && !leader && p_last >= 0) {
        const uint32_t lead_hist = mapa_shared(shist, 0);
        for (int b = threadIdx.x + 1; b < nbins; b += blockDim.x) {
            const uint32_t h = shist[b];
            if (h) red_add_cluster(lead_hist + 4u * static_cast<uint32_t>(b), h);
        }
    }
    if (kPair) cluster_sync_all();   // neither CTA exits or frees tensor memory while the other may still use it;
                                     // orders the peer's additions before the leader's flush
    if (warp == 0) {
        tc_fence_after();
        if (kPair) tmem_dealloc_pair(tmem, kTmemCols);
        else tmem_dealloc(tmem, kTmemCols);
    }
    if (kHist == kHistGlobal || p_last < 0 || (merge && !leader)) return;
    // the worker's histogram into the global one, from which the count pass
    // (one problem) or the select launch (a batch) chooses the pivot threshold
    const ProbView vl = bt.views[p_last];
    if (kHist == kHistPair) {
        for (int b = threadIdx.x; b < nbins; b += blockDim.x)
            if (shist[b]) atomicAdd(&vl.hist[2 * b + static_cast<int>(rank)], shist[b]);
    } else {
        for (int b = threadIdx.x + 1; b <= vl.n; b += blockDim.x)
            if (shist[b]) atomicAdd(&vl.hist[b], shist[b]);
    }
}

std::atomic<int> g_sc2_sms{0};
int g_sc2_pair_clusters = 0;   // co-resident 2-CTA clusters of the pair kernels (0: use single CTAs)

template <bool kPair>
size_t smem_bytes(int nst, int bins)
{
    return static_cast<size_t>(nst) * stage_bytes<kPair>() + kBarBytes + kStgBytes + kColBytes + 1024 +
           static_cast<size_t>(bins) * 4;
}

// Ring stages beside `bins` histogram bins (at most kMaxStages; 0: fewer than two fit).
template <bool kPair>
int stages_for(int bins)
{
    int nst = kMaxStages;
    while (nst > 1 && smem_bytes<kPair>(nst, bins) > static_cast<size_t>(kSmemMax)) --nst;
    return nst > 1 ? nst : 0;
}

// Blocks a worker takes in a row: one for a single problem; in a batch up to
// four, while that leaves every worker at least 16 chunks.
int chunk_for(const Batch& b, int units, int workers)
{
    if (b.num == 1) return 1;
    const int l = units / (workers * 16);
    return l < 1 ? 1 : l > 4 ? 4 : l;
}

template <bool kPair, HistForm kHist>
cudaError_t launch_mma(const Batch& b, int total_tiles, int bins, cudaStream_t s, int auto_mode)
{
    const int nst = stages_for<kPair>(bins);
    const int units = kPair ? total_tiles / 2 : total_tiles;
    int workers = kPair ? g_sc2_pair_clusters : device_sms();
    const int chunk = chunk_for(b, units, workers);
    if (workers > units) workers = units;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(kPair ? 2 * workers : workers));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem_bytes<kPair>(nst, bins);
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 2;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = kPair ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, sc2_mma_kernel<kPair, kHist>, b, total_tiles, bins, nst, chunk, auto_mode);
}

template <bool kPair, HistForm kHist>
cudaError_t mma_attr()
{
    return cudaFuncSetAttribute(sc2_mma_kernel<kPair, kHist>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
}

}  // namespace

// Asked of the current device on first use: a trainer, the allocation-free
// selection and a context each may be the only part of the library in a process.
int device_sms()
{
    int n = g_sc2_sms.load(std::memory_order_relaxed), dev = 0;
    if (n > 0) return n;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)
        return 148;   // no device to ask
    g_sc2_sms.store(n, std::memory_order_relaxed);
    return n;
}

int sc2_pair_clusters() { return g_sc2_pair_clusters; }

cudaError_t sc2_tcgen05_setup()
{
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) g_sc2_sms.store(sms, std::memory_order_relaxed);
    if (e == cudaSuccess) e = mma_attr<true, kHistCta>();
    if (e == cudaSuccess) e = mma_attr<true, kHistPair>();
    if (e == cudaSuccess) e = mma_attr<true, kHistGlobal>();
    if (e == cudaSuccess) e = mma_attr<false, kHistCta>();
    if (e == cudaSuccess) e = mma_attr<false, kHistGlobal>();
    if (e == cudaSuccess) {
        // how many 2-CTA clusters fit at once with the largest shared-memory request
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(2 * 256);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = kSmemMax;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int nc = 0;
        if (cudaOccupancyMaxActiveClusters(&nc, sc2_mma_kernel<true, kHistCta>, &cfg) == cudaSuccess)
            g_sc2_pair_clusters = nc;
        else
            cudaGetLastError();   // no cluster support: the single-CTA kernel is used
    }
    return e;
}

// The pair form keeps a CTA's bins beside its ring.  One problem whose bins
// would cost the ring a stage splits them over the pair: at N = 20000 that
// leaves four stages beside 40 KB of bins instead of three beside 80 KB (and at
// N = 32768 three beside 64 KB, where 128 KB leave fewer than two).  A batch does not (its CTAs flush their bins by
// themselves between problems): above N = 31 999 its edges add to the global
// bins, as the single-CTA form's do above 23 807 (larger stages).
bool launch_sc2_tcgen05(const Batch& b, int total_tiles, int max_n, bool pair_mma, cudaStream_t s, bool auto_mode)
{
    const int bins = max_n + 1;
    if (pair_mma && g_sc2_pair_clusters > 0) {
        static_assert(2 * stage_bytes<true>() + kBarBytes + kStgBytes + kColBytes + 1024 +
                      (TURBOREG_MAX_N / 2 + 2) * 4 <= kSmemMax, "half of the largest histogram fits beside two stages");
        const int half = bins / 2 + 1;
        if (b.num == 1 && stages_for<true>(half) > stages_for<true>(bins)) {
            launch_mma<true, kHistPair>(b, total_tiles, half, s, auto_mode ? 1 : 0);
        } else if (stages_for<true>(bins) > 0) {
            launch_mma<true, kHistCta>(b, total_tiles, bins, s, auto_mode ? 1 : 0);
        } else {
            launch_mma<true, kHistGlobal>(b, total_tiles, 0, s, 0);
            return false;
        }
    } else if (stages_for<false>(bins) > 0) {
        launch_mma<false, kHistCta>(b, total_tiles, bins, s, 0);
    } else {
        launch_mma<false, kHistGlobal>(b, total_tiles, 0, s, 0);
        return false;
    }
    return b.num == 1;
}


}  // namespace tr
