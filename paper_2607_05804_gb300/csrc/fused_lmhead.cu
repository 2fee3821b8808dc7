// Fused LM heads + OPD loss (sm_103a): the student and teacher logits of the
// supervised tokens are produced tile by tile on the tensor cores and folded
// into the loss statistics in the epilogue; no whole logit matrix is stored.
//
//   forward   Z_t = H_t W_t^T (K = d_t), then Z_s = H_s W_s^T (K = d_s), per
//             256-row x 256-vocab tile, accumulated in tensor memory (512 fp32
//             columns per CTA: Z_t in [0,256), Z_s in [256,512)); the epilogue
//             folds each tile into per-row online statistics (max, sum exp,
//             sum exp (z_s - z_t)) for both models over a group of tiles;
//   merge     per row: LSE_s, LSE_t, KL = E_p[z_s - z_t] - (LSE_s - LSE_t);
//   backward  G = w p_s ((z_s - z_t) - E_p[z_s - z_t]) = dL/dz_s in bf16.  The
//             rows are taken in chunks of at most kChunkTiles row tiles: the
//             forward epilogue of a chunk also leaves z_s and z_s - z_t (fp32,
//             the very values it folded) in a chunk-sized scratch, and k_fused_g
//             turns them into G.  A workspace without that scratch recomputes
//             the tiles instead (k_fused_lm<kRecompute>).  Recomputing costs as much
//             tensor work as the whole forward pass, the scratch 18 bytes of HBM per
//             logit: 9,826 rows x 151,936, d 4096 / 5120, dH: 43.2 -> 27.1 ms; 308
//             rows with dW: 3.65 -> 2.65 ms;
//   dH_s      = G W_s by a second tensor-core GEMM over the vocabulary, W_s read
//             in place as an MN-major operand.
//
// GEMM structure: persistent 2-CTA clusters, one CTA per SM.  A tile is
// computed by the pair with cta_group::2 instructions (M = 256, N = 256): each
// CTA stages its own 128 rows of A and 128 rows of B per 64-deep k-block, so a
// pair reads 2/3 of the operand bytes two independent 128 x 256 tiles would.
// In each CTA warp 0 streams the operand tiles with TMA (128-byte swizzle)
// into a 5-stage ring, every copy counted on the even CTA's barrier; warp 1
// allocates tensor memory, and in the even CTA one thread issues tcgen05.mma
// and multicasts its commits to both CTAs; warps 2..17 read this CTA's 128
// accumulator rows back (tcgen05.ld) for the epilogue.  The two halves of the
// accumulator are released separately: the epilogue copies Z_t of tile j into
// registers while Z_s of tile j is computed, and reads Z_s of tile j while Z_t
// of tile j+1 is computed.  The backward epilogue stages each warp's 32 x 64
// block of G in shared memory (128-byte swizzle) and writes it with a TMA
// store, so G leaves the SM in whole 128-byte rows.  Every wait is bounded; on timeout the kernel
// records TURNOPD_ERR_TIMEOUT, keeps its hand-off sequence without waiting,
// drains its in-flight copies and tensor-core work with bounded waits, and
// releases its tensor memory before it exits.

#include <cudaTypedefs.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "ptx.cuh"

namespace turnopd {
namespace {

constexpr int BM = 128;             // accumulator rows per CTA
constexpr int BMP = 2 * BM;         // rows per pair tile
constexpr int BN = 256;             // columns per pair tile
constexpr int BNH = BN / 2;         // B rows staged per CTA
// Operand ring depth: 5 x 32 KB plus the 64 KB G staging buffer fills the
// 227 KB of shared memory a CTA may use (measured: 4 and 6 stages, the
// latter with direct G stores, are both slower).
#ifndef TURNOPD_FUSED_STAGES
#define TURNOPD_FUSED_STAGES 5
#endif
// L2 prefetch distance of the B operand in k-blocks (0: none).  Measured on
// GB300 it slows the GEMMs (the extra tensor requests compete with the ring's
// own copies), so it is off.
#ifndef TURNOPD_FUSED_PF
#define TURNOPD_FUSED_PF 0
#endif
constexpr int BK = 64, STAGES = TURNOPD_FUSED_STAGES;
constexpr int kPrefetch = TURNOPD_FUSED_PF;   // k-blocks of B brought into L2 ahead of the ring
constexpr int A_BYTES = BM * BK * 2, B_BYTES = BNH * BK * 2, STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int kEpiWarps = 16;                    // 4 per tensor-memory lane quarter
constexpr int kColQuarters = kEpiWarps / 4;      // column slices of a tile
constexpr int kEpiCols = BN / kColQuarters;      // 64 columns per epilogue thread
constexpr int kThreads = 32 * (2 + kEpiWarps);
constexpr uint32_t kLimit = 1u << 24;
constexpr int kTilesPerGroup = 10;  // vocabulary tiles one work unit folds into one partial, at most
constexpr int kMinTilesPerGroup = 4;
constexpr uint32_t kColT = 0, kColS = 256;  // tensor-memory columns of Z_t and Z_s
constexpr uint16_t kPairMask = 0x3;

struct FusedArgs {
    int64_t vocab;
    int64_t vpad;          // G row length (vocab rounded up to BK)
    int d_s, d_t;
    const int4 *rows;      // compacted supervised rows {token, row, y, w bits}
    const int32_t *nvalid;
    int pairs;             // 2-CTA pairs of the launch (pick_group)
    int chunk, chunk_tiles;  // this launch's row tiles: chunk_range(m_tiles, chunk_tiles, chunk)
    int min_group;         // least vocabulary tiles per group that `part` has room for
    float *part;           // [groups][kColQuarters][part_rows][8] partial statistics
    int64_t part_rows;     // rows of `part`: those of the chunk
    float4 *z;             // chunk scratch (kForwardStore), see z_index
    const float *rowc;     // [cap][4]: lse_s * log2e - log2 |w|, E_p[z_s - z_t], sign w, -
    __nv_bfloat16 *G;      // [cap][vpad] backward output
    int32_t *status;
};

// The phase test comes first: the issuing thread's critical path holds no
// other shared-memory access (a load of the timeout flag on every k-block
// costs the tensor pipe about a third of its throughput).
__device__ __forceinline__ bool wait_lim(uint64_t *bar, uint32_t parity, int32_t *status, int *dead,
                                         bool cluster_scope = false)
{
    if (cluster_scope ? mbar_try_wait_cluster(bar, parity) : mbar_try_wait(bar, parity))
        return true;
    if (*(volatile int *)dead)
        return false;
    for (uint32_t i = 0; i < kLimit; ++i)
        if (cluster_scope ? mbar_try_wait_cluster(bar, parity) : mbar_try_wait(bar, parity))
            return true;
    *(volatile int *)dead = 1;
    set_status(status, TURNOPD_ERR_TIMEOUT);
    return false;
}

// Bounded wait used while draining at exit (also after a timeout).
__device__ __forceinline__ void wait_drain(uint64_t *bar, uint32_t parity)
{
    for (uint32_t i = 0; i < kLimit; ++i)
        if (mbar_try_wait_cluster(bar, parity))
            return;
}

// Shared memory: ring of STAGES x (A tile | B half tile), then barriers.  The
// layout is identical in both CTAs of a pair (the tensor-core instructions
// address the peer's operands at the issuing CTA's offsets).
struct FusedSmem {
    uint8_t *a, *b;
    uint8_t *stg;               // backward: per-epilogue-warp 32 x 64 bf16 G staging (4 KB each)
    uint64_t *full, *empty;
    uint64_t *acc_t, *acc_s;    // tensor core -> epilogue: Z_t / Z_s of a tile complete
    uint64_t *free_t, *free_s;  // epilogue (both CTAs) -> tensor core: columns read
    uint64_t *drain;
    uint32_t *tslot;
};

__device__ __forceinline__ FusedSmem carve(uint8_t *raw, int b_region, int stg_bytes)
{
    FusedSmem s;
    uint8_t *base = raw + ((1024 - (smem_u32(raw) & 1023)) & 1023);
    s.a = base;
    s.b = base + STAGES * A_BYTES;
    s.stg = s.b + b_region;
    s.full = reinterpret_cast<uint64_t *>(s.stg + stg_bytes);
    s.empty = s.full + STAGES;
    s.acc_t = s.empty + STAGES;
    s.acc_s = s.acc_t + 1;
    s.free_t = s.acc_s + 1;
    s.free_s = s.free_t + 1;
    s.drain = s.free_s + 1;
    s.tslot = reinterpret_cast<uint32_t *>(s.drain + 1);
    return s;
}

constexpr int kLmBRegion = STAGES * B_BYTES;
constexpr int kStgWarpBytes = 32 * kEpiCols * 2;             // 32 rows x 128 B
static_assert(kStgWarpBytes == 32 * 32 * 4, "a 32 x 32 fp32 box of dW_s fits it");
constexpr int kStgBytes = kEpiWarps * kStgWarpBytes;          // 64 KB
// The dH kernel reads B as an MN-major operand; 16 KB of slack after the ring
// keeps every address its descriptors can form inside the allocation.
constexpr int kDhBRegion = STAGES * B_BYTES + 16384;
static_assert(kStgBytes >= 16384, "the staging buffers stand in for the slack in k_fused_dw");
constexpr size_t kFusedSmem = STAGES * A_BYTES + kLmBRegion + kStgBytes + 1024 + 256;
static_assert(kFusedSmem <= 232448, "shared memory per CTA");
constexpr size_t kDhSmem = STAGES * A_BYTES + kDhBRegion + 1024 + 256;
static_assert(kDhSmem <= 232448, "shared memory per CTA");

__device__ __forceinline__ void init_barriers(const FusedSmem &sm)
{
    for (int s = 0; s < STAGES; ++s) {
        mbar_init(&sm.full[s], 1);
        mbar_init(&sm.empty[s], 1);
    }
    mbar_init(sm.acc_t, 1);
    mbar_init(sm.acc_s, 1);
    mbar_init(sm.free_t, 2 * kEpiWarps);
    mbar_init(sm.free_s, 2 * kEpiWarps);
    mbar_init(sm.drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Common prologue: barriers, tensor memory for the pair, cluster-wide visibility.
__device__ __forceinline__ uint32_t pair_prologue(const FusedSmem &sm, int *s_dead, uint32_t ncols)
{
    const int warp = threadIdx.x / 32;
    if (threadIdx.x == 0) {
        *s_dead = 0;
        init_barriers(sm);
    }
    if (warp == 1) {
        tmem_alloc_pair(sm.tslot, ncols);
        tmem_relinquish_pair();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    tc_fence_after();
    return *sm.tslot;
}

// Producer exit (both CTAs): wait (bounded) until the tensor core has released
// the last copy of every stage, so no multicast commit is still on its way to
// this CTA's barriers; the even CTA also waits for its full barriers, which
// count the copies of both CTAs.
__device__ __forceinline__ void drain_producer(const FusedSmem &sm, uint32_t issued, uint32_t rank)
{
    const uint32_t first = issued > STAGES ? issued - STAGES : 0;
    for (uint32_t j = first; j < issued; ++j) {
        if (rank == 0)
            wait_drain(&sm.full[j % STAGES], (j / STAGES) & 1);
        wait_drain(&sm.empty[j % STAGES], (j / STAGES) & 1);
    }
}

// Epilogue -> tensor core: this warp has finished reading a half of the accumulator.
__device__ __forceinline__ void release_cols(uint32_t bar_leader, int lane)
{
    tc_fence_before();
    __syncwarp();
    if (lane == 0)
        mbar_arrive_cluster(bar_leader);
}

// Common epilogue of the kernels: every tcgen05 operation of the pair is
// complete (drain barrier in both CTAs) before tensor memory is released.
__device__ __forceinline__ void pair_epilogue(const FusedSmem &sm, uint32_t tmem, uint32_t ncols, uint32_t rank)
{
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    if (warp == 1 && lane == 0) {
        if (rank == 0)
            tc_commit_pair(sm.drain, kPairMask);
        wait_drain(sm.drain, 0);
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    tc_fence_after();
    if (warp == 1)
        tmem_dealloc_pair(tmem, ncols);
}

// Work unit u -> (pair M tile, vocabulary group).  The M tiles are cut into
// blocks of at most kMBlock; the units of a block are enumerated group-major,
// so the pairs running side by side share the H rows of one block and the W
// tiles of a few groups: a working set of about (kMBlock + pairs / kMBlock)
// 4.7 MB operand panels, which stays in L2.
constexpr int kMBlock = 16;
__device__ __forceinline__ void unit_coords(int u, int m_tiles, int n_groups, int *mt, int *g)
{
    const int nb = (m_tiles + kMBlock - 1) / kMBlock;
    const int mb = (m_tiles + nb - 1) / nb;          // block height (last block may be shorter)
    const int b = u / (mb * n_groups);
    const int rest = u - b * mb * n_groups;
    const int h = min(mb, m_tiles - b * mb);
    *g = rest / h;
    *mt = b * mb + rest % h;
}

// Vocabulary tiles per group: the largest of kTilesPerGroup .. min_group that gives the
// fewest tile steps to the pair with the most work.  A unit is indivisible, so a fixed
// group of 10 left the last wave of units nearly empty on few row tiles (2 row tiles of
// V = 151,936 on 76 pairs: 120 units, 20 tile steps for the busiest pair where 15.6
// would be even; groups of 8 take 16).
__device__ __forceinline__ int pick_group(int m_tiles, int n_tiles, int pairs, int min_group)
{
    int best = kTilesPerGroup, cost = INT32_MAX;
    for (int gs = kTilesPerGroup; gs >= min_group; --gs) {
        const int units = m_tiles * ((n_tiles + gs - 1) / gs);
        const int c = (units + pairs - 1) / pairs * gs;
        if (c < cost) {
            cost = c;
            best = gs;
        }
    }
    return best;
}

// Row tiles [*lo, *hi) of chunk c: the row tiles in the fewest chunks of at most
// chunk_tiles, as even as they come (empty past the last).
__device__ __forceinline__ void chunk_range(int m_tiles, int chunk_tiles, int c, int *lo, int *hi)
{
    const int n = (m_tiles + chunk_tiles - 1) / chunk_tiles;
    const int h = n > 0 ? (m_tiles + n - 1) / n : 0;
    *lo = min(m_tiles, c * h);
    *hi = min(m_tiles, *lo + h);
}

// The chunk scratch holds, for each block of 32 rows and each 4 columns, the 32 rows'
// z_s (16 bytes a row) and then their z_s - z_t: a warp of the epilogue, one row per
// lane, stores 512 contiguous bytes at a time, and k_fused_g reads them the same way.
__device__ __forceinline__ size_t z_index(int64_t vpad, int row_block, int64_t col4)
{
    return ((size_t)row_block * (size_t)(vpad / 4) + (size_t)col4) * 64;
}

// ----------------------------------------------------------------------------
// Forward statistics (kForward; kForwardStore also leaves the chunk's logits in the
// scratch) / backward logit gradient by recomputing the tiles (kRecompute).
// Work unit: one pair M tile x one vocabulary group of pick_group() 256-wide tiles,
// folded into one partial per row.
enum { kForward = 0, kRecompute = 1, kForwardStore = 2 };
template <int MODE>
__global__ void __launch_bounds__(kThreads, 1)
k_fused_lm(const __grid_constant__ CUtensorMap tHs, const __grid_constant__ CUtensorMap tWs,
           const __grid_constant__ CUtensorMap tHt, const __grid_constant__ CUtensorMap tWt,
           const __grid_constant__ CUtensorMap tGst, FusedArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ int s_dead;
    FusedSmem sm = carve(smem_raw, kLmBRegion, kStgBytes);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t rank = cluster_ctarank();
    const int pair = (int)cluster_id(), n_pairs = (int)cluster_count();
    const int nvalid = *a.nvalid;
    const int n_tiles = (int)((a.vocab + BN - 1) / BN);
    int mt_lo, mt_hi;
    chunk_range((nvalid + BMP - 1) / BMP, a.chunk_tiles, a.chunk, &mt_lo, &mt_hi);
    const int m_tiles = mt_hi - mt_lo;
    if (m_tiles == 0)  // the same for every CTA of the grid
        return;
    const int gsize = pick_group(m_tiles, n_tiles, a.pairs, a.min_group);
    const int n_groups = (n_tiles + gsize - 1) / gsize;
    const int units = m_tiles * n_groups;
    const int kb_s = a.d_s / BK, kb_t = a.d_t / BK;
    const uint32_t tmem = pair_prologue(sm, &s_dead, 512);

    if (warp == 0 && lane == 0) {
        // ---------------- producer: per tile the teacher k-blocks, then the student's
        tma_prefetch_desc(&tHs);
        tma_prefetch_desc(&tWs);
        tma_prefetch_desc(&tHt);
        tma_prefetch_desc(&tWt);
        const uint32_t full0 = mapa(smem_u32(sm.full), 0);
        const int kb_tile = kb_t + kb_s;
        uint32_t it = 0;
        for (int u = pair; u < units; u += n_pairs) {
            int mt, g;
            unit_coords(u, m_tiles, n_groups, &mt, &g);
            const int t0 = g * gsize, t1 = min(n_tiles, t0 + gsize);
            const int ya = (mt_lo + mt) * BMP + (int)rank * BM;
            const int n_pos = (t1 - t0) * kb_tile;   // (tile, k-block) positions of this unit
            // L2 prefetch of this CTA's B rows at unit position p
            auto prefetch_b = [&](int p) {
                if (kPrefetch == 0 || p >= n_pos)
                    return;
                const int nt2 = t0 + p / kb_tile, kb2 = p % kb_tile;
                const int yb2 = nt2 * BN + (int)rank * BNH;
                if (kb2 < kb_t)
                    tma_prefetch_l2_2d(&tWt, kb2 * BK, yb2);
                else
                    tma_prefetch_l2_2d(&tWs, (kb2 - kb_t) * BK, yb2);
            };
            for (int p = 0; p < kPrefetch; ++p)
                prefetch_b(p);
            for (int nt = t0; nt < t1; ++nt) {
                const int yb = nt * BN + (int)rank * BNH;
                for (int kb = 0; kb < kb_tile; ++kb, ++it) {
                    prefetch_b((nt - t0) * kb_tile + kb + kPrefetch);
                    const int s = it % STAGES;
                    if (it >= STAGES)
                        wait_lim(&sm.empty[s], ((it / STAGES) - 1) & 1, a.status, &s_dead);
                    if (rank == 0)
                        mbar_arrive_expect_tx(&sm.full[s], 2 * STAGE_BYTES);
                    const uint32_t fb = full0 + (uint32_t)s * 8u;
                    if (kb < kb_t) {
                        tma_load_2d_pair(sm.a + s * A_BYTES, &tHt, kb * BK, ya, fb);
                        tma_load_2d_pair(sm.b + s * B_BYTES, &tWt, kb * BK, yb, fb);
                    } else {
                        tma_load_2d_pair(sm.a + s * A_BYTES, &tHs, (kb - kb_t) * BK, ya, fb);
                        tma_load_2d_pair(sm.b + s * B_BYTES, &tWs, (kb - kb_t) * BK, yb, fb);
                    }
                }
            }
        }
        drain_producer(sm, it, rank);
    } else if (warp == 1 && lane == 0 && rank == 0) {
        // ---------------- MMA issuer (even CTA)
        constexpr uint32_t idesc = idesc_bf16_f32(BMP, BN);
        uint32_t it = 0, tile = 0;
        auto run_k = [&](uint32_t dcol, int nkb) {
            for (int kb = 0; kb < nkb; ++kb, ++it) {
                const int s = it % STAGES;
                // TMA -> tensor core hand-off: the mbarrier completion suffices
                wait_lim(&sm.full[s], (it / STAGES) & 1, a.status, &s_dead);
#pragma unroll
                for (int k = 0; k < BK / 16; ++k) {
                    const uint64_t ad = smem_desc_sw128(smem_u32(sm.a + s * A_BYTES) + k * 32);
                    const uint64_t bd = smem_desc_sw128(smem_u32(sm.b + s * B_BYTES) + k * 32);
                    tc_mma_pair(tmem + dcol, ad, bd, idesc, kb > 0 || k > 0);
                }
                tc_commit_pair(&sm.empty[s], kPairMask);
            }
        };
        for (int u = pair; u < units; u += n_pairs) {
            int mt, g;
            unit_coords(u, m_tiles, n_groups, &mt, &g);
            const int t0 = g * gsize, t1 = min(n_tiles, t0 + gsize);
            for (int nt = t0; nt < t1; ++nt, ++tile) {
                if (tile > 0)  // both epilogues hold Z_t of the previous tile in registers
                    wait_lim(sm.free_t, (tile - 1) & 1, a.status, &s_dead, true);
                tc_fence_after();
                run_k(kColT, kb_t);
                tc_commit_pair(sm.acc_t, kPairMask);
                if (tile > 0)  // both epilogues have read Z_s of the previous tile
                    wait_lim(sm.free_s, (tile - 1) & 1, a.status, &s_dead, true);
                tc_fence_after();
                run_k(kColS, kb_s);
                tc_commit_pair(sm.acc_s, kPairMask);
            }
        }
    } else if (warp >= 2) {
        // ---------------- epilogue: warp (q, cq) owns rows q*32.. and columns cq*64..
        const int ew = warp - 2;
        const int q = warp % 4;              // tensor-memory lane quarter this warp may read
        const int cq = ew / 4;               // column slice [cq*64, cq*64 + 64) of the tile
        const uint32_t lane_off = (uint32_t)(q * 32) << 16;
        const uint32_t col0 = (uint32_t)(cq * kEpiCols);
        const uint32_t free_t0 = mapa(smem_u32(sm.free_t), 0), free_s0 = mapa(smem_u32(sm.free_s), 0);
        uint8_t *stg = sm.stg + ew * kStgWarpBytes;
        uint32_t tile = 0;
        for (int u = pair; u < units; u += n_pairs) {
            int mt, g;
            unit_coords(u, m_tiles, n_groups, &mt, &g);
            const int t0 = g * gsize, t1 = min(n_tiles, t0 + gsize);
            const int lrow = mt * BMP + (int)rank * BM + q * 32 + lane;  // within the chunk
            const int row = mt_lo * BMP + lrow;
            const bool valid_row = row < nvalid;
            float ms = -INFINITY, ss = 0.f, sa = 0.f, mt_ = -INFINITY, st = 0.f;
            float nl = 0.f, cp = 0.f, sg = 1.f;
            if (MODE == kRecompute && valid_row) {
                const float4 c = reinterpret_cast<const float4 *>(a.rowc)[row];
                nl = c.x, cp = c.y, sg = c.z;
            }
            for (int nt = t0; nt < t1; ++nt, ++tile) {
                const int64_t vbase = (int64_t)nt * BN + col0;   // vocabulary id of column 0 here
                const int64_t left = a.vocab - vbase;
                const int nv = left <= 0 ? 0 : (left >= kEpiCols ? kEpiCols : (int)left);
                // Z_t: 64 columns into registers, then release them to the next tile
                float zt[kEpiCols];
                wait_lim(sm.acc_t, tile & 1, a.status, &s_dead);
                tc_fence_after();
                tmem_ld32(tmem + lane_off + kColT + col0, *reinterpret_cast<float(*)[32]>(&zt[0]));
                tmem_ld32(tmem + lane_off + kColT + col0 + 32, *reinterpret_cast<float(*)[32]>(&zt[32]));
                tmem_ld_wait();
                release_cols(free_t0, lane);
                if (MODE != kRecompute && nv > 0) {
                    float cmt = -INFINITY;
#pragma unroll
                    for (int j = 0; j < kEpiCols; ++j)
                        if (j < nv)
                            cmt = fmaxf(cmt, zt[j]);
                    if (cmt > mt_) {
                        st *= ex2((mt_ - cmt) * kLog2e);
                        mt_ = cmt;
                    }
                    const float ntt = -mt_ * kLog2e;
#pragma unroll
                    for (int j = 0; j < kEpiCols; ++j)
                        if (j < nv)
                            st += ex2(fmaf(zt[j], kLog2e, ntt));
                }
                // G columns [vbase, vbase + 64) lie wholly inside or outside [0, vpad)
                // (both multiples of 64); the staging buffer is free once the previous
                // tile's store has read it
                const bool in_g = MODE == kRecompute && vbase < a.vpad;
                if (in_g) {
                    if (lane == 0)
                        bulk_wait_read0();
                    __syncwarp();
                }
                // Z_s: 16 columns at a time
                wait_lim(sm.acc_s, tile & 1, a.status, &s_dead);
                tc_fence_after();
#pragma unroll
                for (int ch = 0; ch < kEpiCols / 16; ++ch) {
                    float zs[16];
                    tmem_ld16(tmem + lane_off + kColS + col0 + ch * 16, zs);
                    tmem_ld_wait();
                    const int c0 = ch * 16;
                    if (MODE == kForwardStore && vbase < a.vpad) {
                        float4 *zq = a.z + z_index(a.vpad, lrow / 32, (vbase + c0) / 4) + lane;
#pragma unroll
                        for (int j = 0; j < 16; j += 4) {
                            __stcs(zq + 16 * j, make_float4(zs[j], zs[j + 1], zs[j + 2], zs[j + 3]));
                            __stcs(zq + 16 * j + 32, make_float4(zs[j] - zt[c0 + j], zs[j + 1] - zt[c0 + j + 1],
                                                                  zs[j + 2] - zt[c0 + j + 2], zs[j + 3] - zt[c0 + j + 3]));
                        }
                    }
                    if (MODE != kRecompute) {
                        if (c0 < nv) {
                            float cmx = -INFINITY;
#pragma unroll
                            for (int j = 0; j < 16; ++j)
                                if (c0 + j < nv)
                                    cmx = fmaxf(cmx, zs[j]);
                            if (cmx > ms) {
                                const float f = ex2((ms - cmx) * kLog2e);
                                ss *= f;
                                sa *= f;
                                ms = cmx;
                            }
                            const float ns = -ms * kLog2e;
#pragma unroll
                            for (int j = 0; j < 16; ++j) {
                                if (c0 + j < nv) {
                                    const float e = ex2(fmaf(zs[j], kLog2e, ns));
                                    ss += e;
                                    sa = fmaf(e, zs[j] - zt[c0 + j], sa);
                                }
                            }
                        }
                    } else if (in_g) {
                        // G = w p ((z_s - z_t) - E_p[z_s - z_t]); zero beyond the vocabulary
                        // and on rows past the supervised ones.
                        uint32_t pk[8];
#pragma unroll
                        for (int j = 0; j < 16; j += 2) {
                            float g0 = 0.f, g1 = 0.f;
                            if (valid_row && c0 + j < nv)
                                g0 = sg * ex2(fmaf(zs[j], kLog2e, -nl)) * ((zs[j] - zt[c0 + j]) - cp);
                            if (valid_row && c0 + j + 1 < nv)
                                g1 = sg * ex2(fmaf(zs[j + 1], kLog2e, -nl)) *
                                     ((zs[j + 1] - zt[c0 + j + 1]) - cp);
                            pk[j / 2] = pack_bf16x2(g0, g1);
                        }
                        // this row's two 16-byte pieces 2ch, 2ch+1 of the 128-byte staging row,
                        // placed by the 128-byte swizzle (piece ^ row % 8)
                        uint8_t *srow = stg + lane * 128;
                        const int p0 = (2 * ch) ^ (lane & 7), p1 = (2 * ch + 1) ^ (lane & 7);
                        *reinterpret_cast<uint4 *>(srow + p0 * 16) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                        *reinterpret_cast<uint4 *>(srow + p1 * 16) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
                    }
                }
                release_cols(free_s0, lane);
                if (MODE == kRecompute && in_g) {
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) {
                        tma_store_2d(&tGst, (int)vbase, (mt_lo + mt) * BMP + (int)rank * BM + q * 32, stg);
                        bulk_commit();
                    }
                }
            }
            if (MODE != kRecompute && valid_row) {
                float *pp = a.part + (((size_t)g * kColQuarters + cq) * a.part_rows + lrow) * 8;
                reinterpret_cast<float4 *>(pp)[0] = make_float4(ms, ss, sa, mt_);
                reinterpret_cast<float4 *>(pp)[1] = make_float4(st, 0.f, 0.f, 0.f);
            }
        }
        if (MODE == kRecompute && lane == 0)
            bulk_wait0();
    }
    pair_epilogue(sm, tmem, 512, rank);
}

// ----------------------------------------------------------------------------
// dH = G W_s: A = G [rows, vpad] (K-major, K = vocabulary), B = W_s [V, d_s]
// read in place as an MN-major operand (per CTA two 64-column TMA boxes per
// stage).  Output pair tile 256 x 256 fp32 in tensor memory.  Work split, with
// P pairs: the first floor(tiles / P) * P tiles are whole tiles, one per pair
// per wave, written straight to their token rows; the remaining tiles'
// k-blocks are split evenly over all P pairs (each range covers at most two
// tiles) and written as partial tiles, which k_dh_fixup sums in pair order.
// The result is bitwise reproducible for a given number of pairs.
struct DhArgs {
    const int4 *rows;
    const int32_t *nvalid;
    int d_s;
    int kbs;         // vpad / BK
    float *dh;       // [T, d_s]
    float *partial;  // [P][2][BMP][BN]
    int32_t *status;
};

struct DhSeg {
    int tile, k0, k1, slot;  // slot -1: whole tile; 0/1: partial slot of this pair
};

template <class F>
__device__ __forceinline__ void dh_segments(int tiles, int kbs, int P, int c, F &&f)
{
    const int full = tiles / P * P;
    for (int t = c; t < full; t += P)
        f(DhSeg{t, 0, kbs, -1});
    const int rem = tiles - full;
    if (rem > 0) {
        const int64_t total = (int64_t)rem * kbs;
        const int64_t b = total * c / P, e = total * (c + 1) / P;
        int slot = 0;
        for (int64_t it = b; it < e;) {
            const int j = (int)(it / kbs), k0 = (int)(it % kbs);
            const int64_t k1l = k0 + (e - it);
            const int k1 = k1l < kbs ? (int)k1l : kbs;
            f(DhSeg{full + j, k0, k1, slot++});
            it += k1 - k0;
        }
    }
}

__global__ void __launch_bounds__(kThreads, 1)
k_fused_dh(const __grid_constant__ CUtensorMap tG, const __grid_constant__ CUtensorMap tW, DhArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ int s_dead;
    FusedSmem sm = carve(smem_raw, kDhBRegion, 0);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t rank = cluster_ctarank();
    const int pair = (int)cluster_id(), n_pairs = (int)cluster_count();
    const int nvalid = *a.nvalid;
    const int m_tiles = (nvalid + BMP - 1) / BMP;
    const int n_tiles = a.d_s / BN;
    const int tiles = m_tiles * n_tiles;
    const uint32_t tmem = pair_prologue(sm, &s_dead, 256);

    // whole tiles: N-tile fastest, so the pairs of one wave share the G rows (A)
    if (warp == 0 && lane == 0) {
        tma_prefetch_desc(&tG);
        tma_prefetch_desc(&tW);
        const uint32_t full0 = mapa(smem_u32(sm.full), 0);
        uint32_t it = 0;
        dh_segments(tiles, a.kbs, n_pairs, pair, [&](const DhSeg &sg) {
            const int mt = sg.tile / n_tiles, nt = sg.tile % n_tiles;
            const int ya = mt * BMP + (int)rank * BM;
            const int xb = nt * BN + (int)rank * BNH;
            auto prefetch = [&](int kb) {
                if (kPrefetch == 0 || kb >= sg.k1)
                    return;
                tma_prefetch_l2_2d(&tG, kb * BK, ya);
#pragma unroll
                for (int j = 0; j < BNH / 64; ++j)
                    tma_prefetch_l2_2d(&tW, xb + j * 64, kb * BK);
            };
            for (int p = 0; p < kPrefetch; ++p)
                prefetch(sg.k0 + p);
            for (int kb = sg.k0; kb < sg.k1; ++kb, ++it) {
                prefetch(kb + kPrefetch);
                const int s = it % STAGES;
                if (it >= STAGES)
                    wait_lim(&sm.empty[s], ((it / STAGES) - 1) & 1, a.status, &s_dead);
                if (rank == 0)
                    mbar_arrive_expect_tx(&sm.full[s], 2 * STAGE_BYTES);
                const uint32_t fb = full0 + (uint32_t)s * 8u;
                tma_load_2d_pair(sm.a + s * A_BYTES, &tG, kb * BK, ya, fb);
#pragma unroll
                for (int j = 0; j < BNH / 64; ++j)
                    tma_load_2d_pair(sm.b + s * B_BYTES + j * (64 * BK * 2), &tW, xb + j * 64, kb * BK, fb);
            }
        });
        drain_producer(sm, it, rank);
    } else if (warp == 1 && lane == 0 && rank == 0) {
        constexpr uint32_t idesc = idesc_bf16_f32(BMP, BN, true);
        uint32_t it = 0, tile = 0;
        dh_segments(tiles, a.kbs, n_pairs, pair, [&](const DhSeg &sg) {
            if (tile > 0)
                wait_lim(sm.free_s, (tile - 1) & 1, a.status, &s_dead, true);
            tc_fence_after();
            for (int kb = sg.k0; kb < sg.k1; ++kb, ++it) {
                const int s = it % STAGES;
                wait_lim(&sm.full[s], (it / STAGES) & 1, a.status, &s_dead);
#pragma unroll
                for (int k = 0; k < BK / 16; ++k) {
                    const uint64_t ad = smem_desc_sw128(smem_u32(sm.a + s * A_BYTES) + k * 32);
                    // 16 K-rows of 128 B per step; 64-wide N blocks 8 KB apart; 8-row atoms 1 KB apart
                    const uint64_t bd =
                        smem_desc_sw128_mn(smem_u32(sm.b + s * B_BYTES) + k * 2048, 64 * BK * 2, 1024);
                    tc_mma_pair(tmem, ad, bd, idesc, kb > sg.k0 || k > 0);
                }
                tc_commit_pair(&sm.empty[s], kPairMask);
            }
            tc_commit_pair(sm.acc_s, kPairMask);
            ++tile;
        });
    } else if (warp >= 2) {
        const int ew = warp - 2, q = warp % 4, cq = ew / 4;
        const uint32_t lane_off = (uint32_t)(q * 32) << 16;
        const int col0 = cq * kEpiCols;
        const int rloc = (int)rank * BM + q * 32 + lane;   // row within the pair tile
        const uint32_t free_s0 = mapa(smem_u32(sm.free_s), 0);
        uint32_t tile = 0;
        dh_segments(tiles, a.kbs, n_pairs, pair, [&](const DhSeg &sg) {
            const int mt = sg.tile / n_tiles, nt = sg.tile % n_tiles;
            const int row = mt * BMP + rloc;
            wait_lim(sm.acc_s, tile & 1, a.status, &s_dead);
            tc_fence_after();
            const bool valid = row < nvalid;
            float *dst = nullptr;
            if (valid) {
                if (sg.slot < 0)
                    dst = a.dh + (size_t)a.rows[row].x * a.d_s + nt * BN + col0;
                else
                    dst = a.partial + (((size_t)pair * 2 + sg.slot) * BMP + rloc) * BN + col0;
            }
#pragma unroll 1
            for (int ch = 0; ch < kEpiCols / 32; ++ch) {
                float v[32];
                tmem_ld32(tmem + lane_off + (uint32_t)(col0 + ch * 32), v);
                tmem_ld_wait();
                if (valid) {
                    float4 *d4 = reinterpret_cast<float4 *>(dst + ch * 32);
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        d4[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                }
            }
            release_cols(free_s0, lane);
            ++tile;
        });
    }
    pair_epilogue(sm, tmem, 256, rank);
}

// ----------------------------------------------------------------------------
// dW_s = G^T H_s: [V, d_s] fp32, K = the supervised tokens (padded to a k-block
// with zero rows of G and H_s).  A = G read as an MN-major operand (its
// columns are vocabulary ids), B = the gathered H_s read MN-major (columns are
// d_s); two 256-column accumulators in tensor memory, so the epilogue's stores
// of tile j overlap the MMAs of tile j+1.  Tiles: 256 vocabulary rows x 256
// columns of d_s, column tile fastest (pairs in flight share the G panel).
// With few tokens the kernel is bound by its 4 V d_s bytes of output: a warp copies
// its 32 x 64 block to registers, hands the accumulator back, and sends the block out
// through shared memory by TMA, whole 128-byte lines at a time (stores straight from
// the registers, one row a lane, touched 32 lines each, 16 bytes of every one: 1,122
// us for 308 tokens x 151,936 x 4,096; now 471, the output alone takes 366).
struct DwArgs {
    const int32_t *nvalid;
    int64_t vocab;
    int d_s;
    float *dw;       // [vocab, d_s]
    int32_t *status;
};

__global__ void __launch_bounds__(kThreads, 1)
k_fused_dw(const __grid_constant__ CUtensorMap tGmn, const __grid_constant__ CUtensorMap tHmn,
           const __grid_constant__ CUtensorMap tDw, DwArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ int s_dead;
    // the staging buffers after the ring are also its slack (kDhBRegion)
    FusedSmem sm = carve(smem_raw, kLmBRegion, kStgBytes);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t rank = cluster_ctarank();
    const int pair = (int)cluster_id(), n_pairs = (int)cluster_count();
    const int nvalid = *a.nvalid;
    const int kbs = (nvalid + BK - 1) / BK;
    const int v_tiles = (int)((a.vocab + BMP - 1) / BMP);
    const int d_tiles = a.d_s / BN;
    const int tiles = kbs > 0 ? v_tiles * d_tiles : 0;
    const uint32_t tmem = pair_prologue(sm, &s_dead, 512);
    uint64_t *accf[2] = {sm.acc_t, sm.acc_s};
    uint64_t *acce[2] = {sm.free_t, sm.free_s};

    if (warp == 0 && lane == 0) {
        tma_prefetch_desc(&tGmn);
        tma_prefetch_desc(&tHmn);
        const uint32_t full0 = mapa(smem_u32(sm.full), 0);
        uint32_t it = 0;
        for (int t = pair; t < tiles; t += n_pairs) {
            const int mv = t / d_tiles, nd = t % d_tiles;
            const int xa = mv * BMP + (int)rank * BM;   // this CTA's 128 vocabulary ids
            const int xb = nd * BN + (int)rank * BNH;   // this CTA's 128 columns of d_s
            for (int kb = 0; kb < kbs; ++kb, ++it) {
                const int s = it % STAGES;
                if (it >= STAGES)
                    wait_lim(&sm.empty[s], ((it / STAGES) - 1) & 1, a.status, &s_dead);
                if (rank == 0)
                    mbar_arrive_expect_tx(&sm.full[s], 2 * STAGE_BYTES);
                const uint32_t fb = full0 + (uint32_t)s * 8u;
#pragma unroll
                for (int j = 0; j < BM / 64; ++j)
                    tma_load_2d_pair(sm.a + s * A_BYTES + j * (64 * BK * 2), &tGmn, xa + j * 64, kb * BK, fb);
#pragma unroll
                for (int j = 0; j < BNH / 64; ++j)
                    tma_load_2d_pair(sm.b + s * B_BYTES + j * (64 * BK * 2), &tHmn, xb + j * 64, kb * BK, fb);
            }
        }
        drain_producer(sm, it, rank);
    } else if (warp == 1 && lane == 0 && rank == 0 && kbs > 0) {
        constexpr uint32_t idesc = idesc_bf16_f32(BMP, BN, true, true);
        uint32_t it = 0, tile = 0;
        for (int t = pair; t < tiles; t += n_pairs, ++tile) {
            const int buf = tile & 1;
            if (tile >= 2)  // both epilogues have read this buffer's previous tile
                wait_lim(acce[buf], ((tile >> 1) - 1) & 1, a.status, &s_dead, true);
            tc_fence_after();
            for (int kb = 0; kb < kbs; ++kb, ++it) {
                const int s = it % STAGES;
                wait_lim(&sm.full[s], (it / STAGES) & 1, a.status, &s_dead);
#pragma unroll
                for (int k = 0; k < BK / 16; ++k) {
                    // 16 K-rows (tokens) of 128 B per step; 64-wide M/N blocks 8 KB apart
                    const uint64_t ad = smem_desc_sw128_mn(smem_u32(sm.a + s * A_BYTES) + k * 2048, 64 * BK * 2, 1024);
                    const uint64_t bd = smem_desc_sw128_mn(smem_u32(sm.b + s * B_BYTES) + k * 2048, 64 * BK * 2, 1024);
                    tc_mma_pair(tmem + (uint32_t)buf * 256u, ad, bd, idesc, kb > 0 || k > 0);
                }
                tc_commit_pair(&sm.empty[s], kPairMask);
            }
            tc_commit_pair(accf[buf], kPairMask);
        }
    } else if (warp >= 2) {
        const int ew = warp - 2, q = warp % 4, cq = ew / 4;
        const uint32_t lane_off = (uint32_t)(q * 32) << 16;
        const int col0 = cq * kEpiCols;
        uint8_t *stg = sm.stg + ew * kStgWarpBytes;
        const uint32_t acce0[2] = {mapa(smem_u32(acce[0]), 0), mapa(smem_u32(acce[1]), 0)};
        uint32_t tile = 0;
        if (kbs == 0) {  // no supervised token: dW_s = 0
            for (int t = pair; t < v_tiles * d_tiles; t += n_pairs) {
                const int mv = t / d_tiles, nd = t % d_tiles;
                const int64_t v = (int64_t)mv * BMP + (int)rank * BM + q * 32 + lane;
                if (v < a.vocab) {
                    float4 *d4 = reinterpret_cast<float4 *>(a.dw + v * a.d_s + nd * BN + col0);
                    for (int jj = 0; jj < kEpiCols / 4; ++jj)
                        d4[jj] = make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
        }
        for (int t = pair; t < tiles; t += n_pairs, ++tile) {
            const int mv = t / d_tiles, nd = t % d_tiles, buf = tile & 1;
            const int v0 = mv * BMP + (int)rank * BM + q * 32;  // this warp's first vocabulary row
            wait_lim(accf[buf], (tile >> 1) & 1, a.status, &s_dead);
            tc_fence_after();
            float x[kEpiCols];
            tmem_ld32(tmem + lane_off + (uint32_t)buf * 256u + (uint32_t)col0, *reinterpret_cast<float(*)[32]>(&x[0]));
            tmem_ld32(tmem + lane_off + (uint32_t)buf * 256u + (uint32_t)col0 + 32,
                      *reinterpret_cast<float(*)[32]>(&x[32]));
            tmem_ld_wait();
            release_cols(acce0[buf], lane);
#pragma unroll
            for (int ch = 0; ch < kEpiCols / 32; ++ch) {
                if (lane == 0)
                    bulk_wait_read0();  // the staging buffer's previous box has left it
                __syncwarp();
#pragma unroll
                for (int jj = 0; jj < 8; ++jj)
                    *reinterpret_cast<float4 *>(stg + lane * 128 + (jj ^ (lane & 7)) * 16) =
                        make_float4(x[ch * 32 + 4 * jj], x[ch * 32 + 4 * jj + 1], x[ch * 32 + 4 * jj + 2],
                                    x[ch * 32 + 4 * jj + 3]);
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0 && v0 < a.vocab) {  // a box's rows past the vocabulary are clipped
                    tma_store_2d(&tDw, nd * BN + col0 + ch * 32, v0, stg);
                    bulk_commit();
                }
            }
        }
        if (lane == 0)
            bulk_wait0();
    }
    pair_epilogue(sm, tmem, 512, rank);
}

// Sum the partial tiles of the split part of dH in pair order (P = pairs of
// the dH launch, at most kMaxPairs) and write them to their token rows.  Job =
// (split tile, 8-row block).
constexpr int kMaxPairs = 256;
inline int max_pairs(int sms) { return std::max(1, std::min(kMaxPairs, sms / 2)); }
__global__ void __launch_bounds__(256)
k_dh_fixup(const float *__restrict__ partial, const int4 *__restrict__ rows, const int32_t *__restrict__ nvalid_p,
           int d_s, int kbs, int P, float *__restrict__ dh)
{
    __shared__ int s_src[kMaxPairs + 2];
    __shared__ int s_n;
    const int nvalid = *nvalid_p;
    const int n_tiles = d_s / BN;
    const int tiles = (nvalid + BMP - 1) / BMP * n_tiles;
    const int full = tiles / P * P;
    const int rem = tiles - full;
    const int64_t total = (int64_t)rem * kbs;
    constexpr int kRowsPerJob = 8;
    for (int job = blockIdx.x; job < rem * (BMP / kRowsPerJob); job += gridDim.x) {
        const int j = job / (BMP / kRowsPerJob), rb = job % (BMP / kRowsPerJob);
        __syncthreads();
        if (threadIdx.x == 0) {
            // pairs whose non-empty k-block range meets tile j's [lo, hi), in pair order
            const int64_t lo = (int64_t)j * kbs, hi = lo + kbs;
            int n = 0;
            // pair c's range starts at floor(total c / P): none before lo P / total - 1
            // reaches lo (walking all P pairs per job: 53 us for the 32 split tiles of 308
            // rows, now 18)
            for (int c = max(0, (int)(lo * P / total) - 1); c < P; ++c) {
                const int64_t b = total * c / P, en = total * (c + 1) / P;
                if (b >= hi)
                    break;
                if (b >= en || en <= lo)
                    continue;
                s_src[n++] = c * 2 + ((b / kbs == j) ? 0 : 1);
            }
            s_n = n;
        }
        __syncthreads();
        const int t = full + j, mt = t / n_tiles, nt = t % n_tiles;
        const int n = s_n;
        for (int e = threadIdx.x; e < kRowsPerJob * (BN / 4); e += blockDim.x) {
            const int r = rb * kRowsPerJob + e / (BN / 4), c4 = e % (BN / 4);
            const int row = mt * BMP + r;
            if (row >= nvalid)
                continue;
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int i = 0; i < n; ++i) {
                const float4 v = reinterpret_cast<const float4 *>(partial)[((size_t)s_src[i] * BMP + r) * (BN / 4) + c4];
                acc.x += v.x;
                acc.y += v.y;
                acc.z += v.z;
                acc.w += v.w;
            }
            reinterpret_cast<float4 *>(dh + (size_t)rows[row].x * d_s + nt * BN)[c4] = acc;
        }
    }
}

// ----------------------------------------------------------------------------
// Gather the supervised hidden rows: out[j] = h[token of row j] (16-byte copies).
// Rows from the supervised count up to the next pair-tile boundary are zeroed
// (the weight-gradient GEMM reads them as zero-weight tokens).
__global__ void k_gather_rows(const int4 *__restrict__ rows, const int32_t *__restrict__ nvalid,
                              const uint4 *__restrict__ h, int vec_per_row, uint4 *__restrict__ out)
{
    const int n = *nvalid;
    const int n_pad = (n + BMP - 1) / BMP * BMP;
    for (int j = blockIdx.x; j < n_pad; j += gridDim.x) {
        uint4 *dst = out + (int64_t)j * vec_per_row;
        if (j < n) {
            const uint4 *src = h + (int64_t)rows[j].x * vec_per_row;
            for (int c = threadIdx.x; c < vec_per_row; c += blockDim.x)
                dst[c] = src[c];
        } else {
            for (int c = threadIdx.x; c < vec_per_row; c += blockDim.x)
                dst[c] = make_uint4(0, 0, 0, 0);
        }
    }
}

// Per supervised row of the chunk: merge the vocabulary-group partials into LSE_s,
// LSE_t, KL; write l, w*l and the backward constants.  One warp per row, a record per
// lane and step, then a fixed tree over the lanes.  (One thread per row walked its 240
// records of V = 151,936 as one chain of loads and exponentials: 150 us whatever the
// number of rows; now 12 us for 308 rows, 13 for a chunk of 2,048.)
__global__ void __launch_bounds__(256)
k_fused_merge(const int4 *__restrict__ rows, FusedArgs a, float *__restrict__ token_loss,
              double *__restrict__ row_wl, float *__restrict__ rowc)
{
    const int n = *a.nvalid, lane = threadIdx.x & 31;
    const int n_tiles = (int)((a.vocab + BN - 1) / BN);
    int mt_lo, mt_hi;
    chunk_range((n + BMP - 1) / BMP, a.chunk_tiles, a.chunk, &mt_lo, &mt_hi);
    if (mt_lo == mt_hi)
        return;
    const int gsize = pick_group(mt_hi - mt_lo, n_tiles, a.pairs, a.min_group);
    const int recs = (n_tiles + gsize - 1) / gsize * kColQuarters;
    const int row0 = mt_lo * BMP, row1 = min(n, mt_hi * BMP);
    const int nwarp = gridDim.x * (blockDim.x / 32);
    for (int j = row0 + (int)(blockIdx.x * blockDim.x + threadIdx.x) / 32; j < row1; j += nwarp) {
        Student S = student_empty();
        Teacher T = teacher_empty();
        const float4 *pp = reinterpret_cast<const float4 *>(a.part) + (size_t)(j - row0) * 2;
#pragma unroll 4
        for (int gh = lane; gh < recs; gh += 32) {
            const float4 x = pp[(size_t)gh * a.part_rows * 2];
            const float4 y = pp[(size_t)gh * a.part_rows * 2 + 1];
            if (x.x != -INFINITY)
                S = student_merge(S, Student{x.x, x.y, x.z, 0.f});
            if (x.w != -INFINITY)
                T = teacher_merge(T, Teacher{x.w, y.x});
        }
        S = warp_merge(S);
        T = warp_merge(T);
        if (lane == 0) {
            const RowConst rc = row_const(S, T);
            const int4 m = rows[j];
            const float w = __int_as_float(m.w);
            const float ell = rc.kl;
            if (!isfinite(rc.lse_s) || !isfinite(rc.lse_t) || !isfinite(ell))
                set_status(a.status, TURNOPD_ERR_NONFINITE);
            token_loss[m.x] = ell;
            row_wl[j] = (double)w * (double)ell;
            // p |w| = 2^(z_s log2e - nl): nl = LSE_s log2e - log2 |w|
            reinterpret_cast<float4 *>(rowc)[j] =
                make_float4(rc.lse_s * kLog2e - log2f(fabsf(w)), rc.d + rc.cp, w < 0.f ? -1.f : 1.f, 0.f);
        }
    }
}

// G of one chunk from its stored logits: a stream of 8 bytes read and 2 written per
// logit, bound by HBM (2,048 rows x 151,936: 471 us, 6.6 TB/s).  A warp takes 32 rows x 64 columns at a time: 16 KB of scratch in
// whole 512-byte reads, one row per lane; the bf16 values cross the warp through shared
// memory (128-byte rows, 16-byte pieces swizzled by row % 8) and leave as whole 128-byte
// lines.  Columns past the vocabulary and rows past the supervised ones get zeros, as
// the GEMMs that read G want them.
constexpr int kGThreads = 256;
__global__ void __launch_bounds__(kGThreads)
k_fused_g(FusedArgs a)
{
    __shared__ __align__(128) uint8_t stage[kGThreads / 32][32 * 128];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n = *a.nvalid;
    int mt_lo, mt_hi;
    chunk_range((n + BMP - 1) / BMP, a.chunk_tiles, a.chunk, &mt_lo, &mt_hi);
    const int row_blocks = (mt_hi - mt_lo) * (BMP / 32);
    const int col_blocks = (int)(a.vpad / 64);
    const int64_t units = (int64_t)row_blocks * col_blocks;
    uint8_t *stg = stage[warp];
    const int64_t nw = (int64_t)gridDim.x * (kGThreads / 32);
    for (int64_t u = (int64_t)blockIdx.x * (kGThreads / 32) + warp; u < units; u += nw) {
        const int rb = (int)(u / col_blocks), cb = (int)(u % col_blocks);
        const int row = mt_lo * BMP + rb * 32 + lane;
        const bool valid = row < n;
        float nl = 0.f, cp = 0.f, sg = 1.f;
        if (valid) {
            const float4 c = reinterpret_cast<const float4 *>(a.rowc)[row];
            nl = c.x, cp = c.y, sg = c.z;
        }
        const int64_t left = a.vocab - (int64_t)cb * 64;
        const int nv = left >= 64 ? 64 : (int)left;
        const float4 *zq = a.z + z_index(a.vpad, rb, (int64_t)cb * 16) + lane;
        __syncwarp();  // the stage's previous block has been read
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            float4 zs[8], x[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                zs[j] = __ldcs(zq + (half * 8 + j) * 64);
                x[j] = __ldcs(zq + (half * 8 + j) * 64 + 32);
            }
#pragma unroll
            for (int j = 0; j < 8; j += 2) {
                uint32_t pk[4];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int c0 = half * 32 + (j + h) * 4;
                    const float zv[4] = {zs[j + h].x, zs[j + h].y, zs[j + h].z, zs[j + h].w};
                    const float xv[4] = {x[j + h].x, x[j + h].y, x[j + h].z, x[j + h].w};
                    float g[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        g[i] = valid && c0 + i < nv ? sg * ex2(fmaf(zv[i], kLog2e, -nl)) * (xv[i] - cp) : 0.f;
                    pk[2 * h] = pack_bf16x2(g[0], g[1]);
                    pk[2 * h + 1] = pack_bf16x2(g[2], g[3]);
                }
                const int piece = (half * 4 + j / 2) ^ (lane & 7);
                *reinterpret_cast<uint4 *>(stg + lane * 128 + piece * 16) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            }
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = i * 4 + lane / 8, c = lane % 8;
            const uint4 v = *reinterpret_cast<const uint4 *>(stg + r * 128 + (c ^ (r & 7)) * 16);
            *reinterpret_cast<uint4 *>(a.G + (size_t)(mt_lo * BMP + rb * 32 + r) * a.vpad + (size_t)cb * 64 + c * 8) = v;
        }
    }
}

// ---------------------------------------------------------------- host side

PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        cudaDriverEntryPointQueryResult q;
        void *p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return nullptr;
        fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

// 2-D bf16 (or fp32) tensor map over a row-major [rows, cols] matrix, 128-byte swizzle,
// box of box_cols (128 B) x box_rows; rows beyond the matrix read as zero.
bool make_map(CUtensorMap *m, const void *base, int64_t rows, int64_t cols, int box_rows, int box_cols,
              bool fp32 = false)
{
    auto fn = encode_fn();
    if (!fn)
        return false;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)cols * (fp32 ? 4 : 2)};
    cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
    cuuint32_t es[2] = {1, 1};
    return fn(m, fp32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
              const_cast<void *>(base), dims, strides, box, es,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct FusedLayout {
    int4 *rows;
    int32_t *blk_count, *nvalid;
    double *row_wl;
    __nv_bfloat16 *hs, *ht, *G;
    float *part, *rowc, *dh_partial;
    size_t base_bytes;   // without the chunk scratch: the least a call accepts
    float *chunk_part;   // [groups of kMinTilesPerGroup][kColQuarters][chunk rows][8]
    float4 *z;           // chunk logits
    size_t bytes;
};

// Row tiles of a chunk, and so the size of its scratch: 8 bytes per logit, 2.5 GB at
// V = 151,936.  A chunk is one launch, which reads both heads once.
#ifndef TURNOPD_FUSED_CHUNK
#define TURNOPD_FUSED_CHUNK 8
#endif
constexpr int kChunkTiles = TURNOPD_FUSED_CHUNK;

int groups_for(int64_t V, int tiles_per_group)
{
    return (int)(((V + BN - 1) / BN + tiles_per_group - 1) / tiles_per_group);
}

FusedLayout fused_layout(void *ws, int64_t T, int64_t V, int64_t d_s, int64_t d_t, int sms)
{
    const int n_groups = groups_for(V, kTilesPerGroup);
    const int64_t vpad = (V + BK - 1) / BK * BK;
    const int64_t cap = (T + BMP - 1) / BMP * BMP;
    const int64_t nblk = (T + kCompactBlock - 1) / kCompactBlock;
    char *p = static_cast<char *>(ws);
    size_t off = 0;
    auto take = [&](size_t n) {
        char *q = p ? p + off : nullptr;
        off += align256(n);
        return q;
    };
    FusedLayout L;
    L.rows = reinterpret_cast<int4 *>(take(sizeof(int4) * (size_t)T));
    L.blk_count = reinterpret_cast<int32_t *>(take(sizeof(int32_t) * (size_t)(nblk + 1)));
    L.nvalid = reinterpret_cast<int32_t *>(take(sizeof(int32_t)));
    L.row_wl = reinterpret_cast<double *>(take(sizeof(double) * (size_t)T));
    L.hs = reinterpret_cast<__nv_bfloat16 *>(take(2 * (size_t)cap * d_s));
    L.ht = reinterpret_cast<__nv_bfloat16 *>(take(2 * (size_t)cap * d_t));
    L.part = reinterpret_cast<float *>(take(sizeof(float) * 8 * kColQuarters * (size_t)n_groups * cap));
    L.rowc = reinterpret_cast<float *>(take(sizeof(float) * 4 * (size_t)cap));
    L.G = reinterpret_cast<__nv_bfloat16 *>(take(2 * (size_t)cap * vpad));
    L.dh_partial = reinterpret_cast<float *>(take(sizeof(float) * (size_t)max_pairs(sms) * 2 * BMP * BN));
    L.base_bytes = off + 256;
    const int64_t chunk = std::min<int64_t>(cap, (int64_t)kChunkTiles * BMP);
    L.chunk_part = reinterpret_cast<float *>(
        take(sizeof(float) * 8 * kColQuarters * (size_t)groups_for(V, kMinTilesPerGroup) * chunk));
    L.z = reinterpret_cast<float4 *>(take(8 * (size_t)chunk * vpad));
    L.bytes = off + 256;
    return L;
}

// Launch `kern` on `pairs` 2-CTA clusters.
template <class... KArgs, class... Args>
cudaError_t launch_pairs(void (*kern)(KArgs...), int pairs, size_t smem, cudaStream_t stream, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.gridDim = dim3(2 * pairs);
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// Co-resident 2-CTA clusters of `kern` (cached per device), at most max_pairs.
template <class... KArgs>
cudaError_t pairs_for(void (*kern)(KArgs...), size_t smem, int slot, int *pairs)
{
    static int cache[64][5] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return e;
    if (dev < 64 && cache[dev][slot] > 0) {
        *pairs = cache[dev][slot];
        return cudaSuccess;
    }
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess)
        return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.gridDim = dim3(2);
    int ncl = 0;
    e = cudaOccupancyMaxActiveClusters(&ncl, kern, &cfg);
    if (e != cudaSuccess)
        return e;
    if (ncl < 1)
        return cudaErrorInvalidConfiguration;
    ncl = std::min(ncl, max_pairs(device_sm_count()));
    if (dev < 64)
        cache[dev][slot] = ncl;
    *pairs = ncl;
    return cudaSuccess;
}

}  // namespace

size_t fused_workspace_bytes(int64_t T, int64_t V, int64_t d_s, int64_t d_t)
{
    return fused_layout(nullptr, T, V, d_s, d_t, device_sm_count()).bytes;
}

size_t fused_workspace_min_bytes(int64_t T, int64_t V, int64_t d_s, int64_t d_t)
{
    return fused_layout(nullptr, T, V, d_s, d_t, device_sm_count()).base_bytes;
}

cudaError_t launch_fused(const FusedCall &c, cudaStream_t stream)
{
    const int sms = device_sm_count();
    FusedLayout L = fused_layout(c.workspace, c.T, c.vocab, c.d_s, c.d_t, sms);
    const int64_t vpad = (c.vocab + BK - 1) / BK * BK;
    const int64_t cap = (c.T + BMP - 1) / BMP * BMP;

    // supervised rows (the compaction of the loss path), then the gathered hidden rows
    LossArgs la{};
    la.mask = c.mask;
    la.w = c.w;
    la.T = c.T;
    la.num_rows = c.T;
    la.vocab = c.vocab;
    la.mode = TURNOPD_FULL_VOCAB;
    la.token_loss = c.token_loss;
    la.status = c.status;
    cudaError_t e = launch_compaction(la, L.rows, L.blk_count, L.nvalid, stream);
    if (e != cudaSuccess)
        return e;
    k_gather_rows<<<sms * 4, 256, 0, stream>>>(L.rows, L.nvalid, static_cast<const uint4 *>(c.h_s), c.d_s / 8,
                                               reinterpret_cast<uint4 *>(L.hs));
    k_gather_rows<<<sms * 4, 256, 0, stream>>>(L.rows, L.nvalid, static_cast<const uint4 *>(c.h_t), c.d_t / 8,
                                               reinterpret_cast<uint4 *>(L.ht));
    e = cudaGetLastError();
    if (e != cudaSuccess)
        return e;

    alignas(64) CUtensorMap tHs, tWs, tHt, tWt, tG, tGst, tWmn, tGmn, tHmn, tDw;
    if (!make_map(&tHs, L.hs, cap, c.d_s, BM, BK) || !make_map(&tWs, c.W_s, c.vocab, c.d_s, BNH, BK) ||
        !make_map(&tHt, L.ht, cap, c.d_t, BM, BK) || !make_map(&tWt, c.W_t, c.vocab, c.d_t, BNH, BK) ||
        !make_map(&tG, L.G, cap, vpad, BM, BK) || !make_map(&tGst, L.G, cap, vpad, 32, kEpiCols) ||
        // W_s as the MN-major B of dH: boxes of 64 d-columns x BK vocabulary rows
        !make_map(&tWmn, c.W_s, c.vocab, c.d_s, BK, 64) ||
        // G and the gathered H_s as the MN-major operands of dW_s: 64 columns x BK token rows
        !make_map(&tGmn, L.G, cap, vpad, BK, 64) || !make_map(&tHmn, L.hs, cap, c.d_s, BK, 64) ||
        (c.dW_s && !make_map(&tDw, c.dW_s, c.vocab, c.d_s, 32, 32, true)))
        return cudaErrorInvalidValue;

    const bool backward = c.dh_s || c.dW_s;
    const bool store = backward && c.workspace_bytes >= L.bytes;
    int p_lm = 0, p_re = 0, p_dh = 0, p_dw = 0;
    if ((e = pairs_for(k_fused_dw, kFusedSmem, 3, &p_dw)) != cudaSuccess ||
        (e = store ? pairs_for(k_fused_lm<kForwardStore>, kFusedSmem, 4, &p_lm)
                   : pairs_for(k_fused_lm<kForward>, kFusedSmem, 0, &p_lm)) != cudaSuccess ||
        (e = pairs_for(k_fused_lm<kRecompute>, kFusedSmem, 1, &p_re)) != cudaSuccess ||
        (e = pairs_for(k_fused_dh, kDhSmem, 2, &p_dh)) != cudaSuccess)
        return e;

    FusedArgs fa;
    fa.vocab = c.vocab;
    fa.vpad = vpad;
    fa.d_s = (int)c.d_s;
    fa.d_t = (int)c.d_t;
    fa.rows = L.rows;
    fa.nvalid = L.nvalid;
    fa.pairs = p_lm;
    fa.chunk = 0;
    fa.chunk_tiles = store ? kChunkTiles : (int)(cap / BMP);
    fa.min_group = store ? kMinTilesPerGroup : kTilesPerGroup;
    fa.part = store ? L.chunk_part : L.part;
    fa.part_rows = store ? std::min<int64_t>(cap, (int64_t)kChunkTiles * BMP) : cap;
    fa.z = store ? L.z : nullptr;
    fa.rowc = L.rowc;
    fa.G = L.G;
    fa.status = c.status;

    // the number of supervised rows is known on the device alone: chunks past the last
    // supervised row are empty launches
    const int chunks = (int)((cap / BMP + fa.chunk_tiles - 1) / fa.chunk_tiles);
    const int merge_grid = (int)std::min<int64_t>((fa.part_rows + 7) / 8, (int64_t)sms * 8);
    for (fa.chunk = 0; fa.chunk < chunks; ++fa.chunk) {
        e = store ? launch_pairs(k_fused_lm<kForwardStore>, p_lm, kFusedSmem, stream, tHs, tWs, tHt, tWt, tGst, fa)
                  : launch_pairs(k_fused_lm<kForward>, p_lm, kFusedSmem, stream, tHs, tWs, tHt, tWt, tGst, fa);
        if (e != cudaSuccess)
            return e;
        k_fused_merge<<<merge_grid, 256, 0, stream>>>(L.rows, fa, c.token_loss, L.row_wl, L.rowc);
        if (store)
            k_fused_g<<<sms * 4, kGThreads, 0, stream>>>(fa);
        if ((e = cudaGetLastError()) != cudaSuccess)
            return e;
    }
    if (backward && !store) {
        fa.chunk = 0;
        fa.pairs = p_re;
        if ((e = launch_pairs(k_fused_lm<kRecompute>, p_re, kFusedSmem, stream, tHs, tWs, tHt, tWt, tGst, fa)) !=
            cudaSuccess)
            return e;
    }
    if (c.dW_s) {
        DwArgs wa;
        wa.nvalid = L.nvalid;
        wa.vocab = c.vocab;
        wa.d_s = (int)c.d_s;
        wa.dw = c.dW_s;
        wa.status = c.status;
        if ((e = launch_pairs(k_fused_dw, p_dw, kFusedSmem, stream, tGmn, tHmn, tDw, wa)) != cudaSuccess)
            return e;
    }
    if (c.dh_s) {
        launch_zero_masked_f32(c.mask, c.T, (int64_t)c.d_s, c.dh_s, stream);
        DhArgs da;
        da.rows = L.rows;
        da.nvalid = L.nvalid;
        da.d_s = (int)c.d_s;
        da.kbs = (int)(vpad / BK);
        da.dh = c.dh_s;
        da.partial = L.dh_partial;
        da.status = c.status;
        if ((e = launch_pairs(k_fused_dh, p_dh, kDhSmem, stream, tG, tWmn, da)) != cudaSuccess)
            return e;
        k_dh_fixup<<<2 * sms, 256, 0, stream>>>(L.dh_partial, L.rows, L.nvalid, (int)c.d_s, da.kbs, p_dh, c.dh_s);
    }
    launch_loss_sum(L.row_wl, L.nvalid, c.loss, c.status, stream);
    return cudaGetLastError();
}

}  // namespace turnopd
