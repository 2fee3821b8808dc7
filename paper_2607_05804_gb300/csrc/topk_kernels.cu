// Teacher top-K reverse KL: the paper's practical loss (loss_mode
// topk_reverse_kl, support size K_top = distill_topk; Algorithm 1, "top-K
// reverse-KL token losses").  For a supervised row, S = the K vocabulary ids
// of largest teacher logit (the lower id first among equal logits); both
// distributions are renormalised over S:
//   l   = sum_{v in S} ps_v (log ps_v - log pt_v)
//   g_v = w ps_v (log ps_v - log pt_v - l)  on S, 0 elsewhere (= w dl/dz_s).
//
// Short rows and rows of any other alignment: k_topk_short, one CTA a row.  Others:
// persistent CTAs, each with two rows in flight: streaming warps run pass A
// of a row while two or four selector warps run the later phases of the previous row
// (double-buffered buckets, named barriers).  Selection with 64-bit keys
// (order-preserving logit bits << 32 | ~id, so larger key = larger logit,
// then lower id):
//   pass A   one read of the teacher row, warp-uniform: for every group of 16
//            consecutive ids the largest logit is recorded in shared memory as
//            a 16-bit ordered bucket (the top 16 bits of the order-preserving
//            bits), and every thread keeps the largest logit it saw;
//   bound    (streaming warps) for K <= 96, tau = the K-th largest of the 8
//            largest lane maxima of every streaming warp: K-th largest of
//            distinct elements of the row, so a lower bound of the row's K-th
//            largest logit; above, the K-th largest thread maximum, or (K above
//            288, or rows of few groups) the K-th largest group bucket (K groups
//            each hold an element that large), by binary search on its value;
//            then the groups whose bucket reaches tau's are listed (and above K =
//            192, 160 for fp32, it is refined to the K-th largest bucket listed);
//   collect  (selector warps) only the listed groups are read again, in step
//            across the lanes (a few dozen per row at K = 50), and their
//            elements >= tau go to a shared-memory candidate buffer (1,024
//            entries, 2,048 above K = 512); when it overflows (rows of many
//            equal logits, sorted rows) a radix select over the row's keys >=
//            tau, one key byte per pass, raises tau until the keys above it fit
//            the buffer, then collects again (at most 6 passes for bf16 keys,
//            8 for fp32);
//   select   up to 256 candidates: the exact K-th largest by radix select (buffers
//            over 2 K), then each selected key's rank among the candidates is its
//            position;
//            more: a bitonic sort of the buffer.
// The KL over S is evaluated by one warp in fp32 with
// l = E_p[z_s - z_t] - (LSE_s - LSE_t) and g_v = w p_v ((z_s - z_t)_v - E_p[.]).

#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "kernels.h"

namespace turnopd {
namespace {

// streaming warps per CTA and CTAs per SM (measured, K = 50, full-size batches, fraction
// of the copy bandwidth packed / household / multihop: 8 x 3: 0.923 / 0.889 / 0.865;
// 12 x 2: 0.942 / 0.910 / 0.874; 10 x 2: 0.926 / 0.895 / 0.864; 14 x 2: 0.921 / 0.884 /
// 0.855; 8 x 2: 0.881 / 0.851 / 0.821; 24 x 1: 0.771 / 0.740 / 0.713)
#ifndef TURNOPD_TOPK_STREAM_WARPS
#define TURNOPD_TOPK_STREAM_WARPS 12
#endif
#ifndef TURNOPD_TOPK_MINB
#define TURNOPD_TOPK_MINB 2
#endif
constexpr int kTkStreamWarps = TURNOPD_TOPK_STREAM_WARPS;  // pass A, row after row
// Selector warps (the later phases, a row behind): SW is a template parameter of what they
// run, 2 up to K = 96 and 4 above, where they set the pace (their collect, sort and KL grow
// with K; sort_desc needs n >= 2 x 32 SW and n >= 256, so at most 4).  9,870 rows of V =
// 151,936, bf16: K = 256 sparse 863 us with 4, 1,115 with 2; K = 128 642, 641.
#ifndef TURNOPD_TOPK_SEL_LARGE
#define TURNOPD_TOPK_SEL_LARGE 4
#endif
constexpr int kTkSelSmall = 2, kTkSelLarge = TURNOPD_TOPK_SEL_LARGE;
constexpr int kTkStreamThreads = kTkStreamWarps * 32;
constexpr int kTkMinBlocks = TURNOPD_TOPK_MINB;  // CTAs (rows in flight) per SM
// named barriers: buffer b full (1 + b), buffer b free (3 + b), selectors only (5),
// streaming warps only (6)
constexpr int kBarFull = 1, kBarFree = 3, kBarSel = 5, kBarStream = 6;
constexpr int kTkGroupCap = 2048;  // candidate groups listed per row by the streaming warps
// candidate buffer (keys and student logits): 1,024 entries, 2,048 above K = 512
// (a power of two: the bitonic sort of a large buffer runs in place)
__host__ __device__ constexpr int topk_cap(int K) { return K <= 512 ? 1024 : 2048; }
// K up to which the streaming warps' lane maxima give the bound (the 8 largest
// of each warp's 32); the group buckets give it above
constexpr int kTkLaneTop = 8;
constexpr int kTkLaneBoundMaxK = kTkStreamWarps * kTkLaneTop;
// candidates above which the selection sorts the buffer instead of ranking
constexpr int kTkRankMax = 256;
constexpr uint32_t kTkQueue = 64;  // ring of group indices per selector warp (at most 63 held)
constexpr int kTkGroup = 16;      // ids per recorded bucket
constexpr int kRefine = 2;        // listed groups per streaming thread that the bound is refined on
// (K = 256 at V = 151,936: 863 us with it, 883 without; K = 128: 728 and 642; fp32, where the
// listed groups' second read weighs double, K = 192 at V = 98,304 207 and 235, K = 160 200 and 192)
constexpr int kRefineMinK = 192, kRefineMinKF32 = 160;
static_assert(kTkQueue >= 64 && (kTkQueue & (kTkQueue - 1)) == 0, "group ring");
static_assert(TURNOPD_TOPK_MAX_VOCAB / kTkGroup <= 65536, "group indices are 16-bit");
static_assert(TURNOPD_TOPK_MAX_VOCAB <= (1 << 20) && topk_cap(TURNOPD_TOPK_MAX) <= 2048,
              "a sorted key holds a 20-bit id and an 11-bit buffer position");

__device__ __forceinline__ uint32_t ord16(uint32_t u)
{
    u &= 0xFFFFu;
    if (u == 0x8000u)
        u = 0;  // -0 and +0 are the same logit
    return (u & 0x8000u) ? (~u & 0xFFFFu) : (u | 0x8000u);
}

__device__ __forceinline__ uint32_t ord32(uint32_t u)
{
    if (u == 0x80000000u)
        u = 0;
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ uint64_t mkkey(uint32_t ord, uint32_t id)
{
    return ((uint64_t)ord << 32) | (uint32_t)(~id);
}

__device__ __forceinline__ uint32_t key_id(uint64_t k) { return ~(uint32_t)k; }

template <bool BF16>
__device__ __forceinline__ float key_value(uint64_t k)
{
    const uint32_t o = (uint32_t)(k >> 32);
    if (BF16) {
        const uint32_t bits = (o & 0x8000u) ? (o & 0x7FFFu) : (~o & 0xFFFFu);
        return __uint_as_float(bits << 16);
    }
    const uint32_t bits = (o & 0x80000000u) ? (o & 0x7FFFFFFFu) : ~o;
    return __uint_as_float(bits);
}

__device__ __forceinline__ uint32_t bf16_max8_ord(const uint4 &v)
{
    const __nv_bfloat162 a = *reinterpret_cast<const __nv_bfloat162 *>(&v.x);
    const __nv_bfloat162 b = *reinterpret_cast<const __nv_bfloat162 *>(&v.y);
    const __nv_bfloat162 c = *reinterpret_cast<const __nv_bfloat162 *>(&v.z);
    const __nv_bfloat162 d = *reinterpret_cast<const __nv_bfloat162 *>(&v.w);
    const __nv_bfloat162 m = __hmax2(__hmax2(a, b), __hmax2(c, d));
    const __nv_bfloat16 mm = __hmax(m.x, m.y);
    return ord16(__bfloat16_as_ushort(mm));
}

// Ordered value of an element (16 significant bits for bf16, 32 for fp32).
template <bool BF16>
__device__ __forceinline__ uint32_t elem_ord(const void *row, int64_t e)
{
    return BF16 ? ord16(static_cast<const uint16_t *>(row)[e]) : ord32(static_cast<const uint32_t *>(row)[e]);
}

// 16-bit bucket of an ordered value: monotone in the value.
template <bool BF16>
__device__ __forceinline__ uint32_t bucket(uint32_t ord)
{
    return BF16 ? ord : ord >> 16;
}

// Largest ordered value of the elements e0 .. e0+15 of a row, clipped to V
// (element by element: the partial last group and misaligned rows).
template <bool BF16>
__device__ __forceinline__ uint32_t group_max_ord_scalar(const void *row, int64_t V, int64_t g)
{
    const int64_t e0 = g * kTkGroup;
    uint32_t m = 0;
    for (int64_t e = e0; e < e0 + kTkGroup && e < V; ++e)
        m = max(m, elem_ord<BF16>(row, e));
    return m;
}

// Ordered values of the 16 elements held in the 16-byte vectors v[0 .. VPG).
template <bool BF16>
__device__ __forceinline__ void unpack_ords(const uint4 *v, uint32_t (&o)[kTkGroup])
{
    if (BF16) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const uint32_t w4[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
#pragma unroll
            for (int e = 0; e < 8; ++e)
                o[q * 8 + e] = ord16(e & 1 ? w4[e >> 1] >> 16 : w4[e >> 1]);
        }
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            o[q * 4 + 0] = ord32(v[q].x);
            o[q * 4 + 1] = ord32(v[q].y);
            o[q * 4 + 2] = ord32(v[q].z);
            o[q * 4 + 3] = ord32(v[q].w);
        }
    }
}

__device__ __forceinline__ void named_sync(int id, int n)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void named_arrive(int id, int n)
{
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// Radix-select scratch of the selector warps: a 256-bin histogram of one key
// byte and the bin chosen from it.
struct SelScratch {
    uint32_t hist[256];
    int bin, need;
};

// The bin of the need-th largest key of a 256-bin histogram sc.hist (bin 255
// holds the largest keys): sc.bin = that bin, or -1 when the histogram holds
// fewer than need keys; sc.need = the count still needed inside the bin,
// negated when the bin holds exactly that many.  Run by one warp (lane 0..31).
__device__ __forceinline__ void pick_bin(SelScratch &sc, int need, int lane)
{
    int c[8], tot = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        c[e] = (int)sc.hist[255 - 8 * lane - e];
        tot += c[e];
    }
    int incl = tot;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off)
            incl += y;
    }
    const int excl = incl - tot;
    const unsigned hit = __ballot_sync(0xffffffffu, excl < need && incl >= need);
    if (hit == 0u) {
        if (lane == 0)
            sc.bin = -1;
    } else if (lane == __ffs(hit) - 1) {
        int cum = excl;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            if (cum + c[e] >= need) {
                sc.bin = 255 - 8 * lane - e;
                sc.need = (cum + c[e] == need) ? -(need - cum) : need - cum;
                break;
            }
            cum += c[e];
        }
    }
}

// Radix select over the selector warps: the K-th largest of the nonzero keys
// in keys[0, n) (keys are unique; 0 marks an empty slot), deciding bytes
// hi_byte..lo_byte.  Returns t such that {keys >= t} holds the K largest keys
// when lo_byte = 0 (exactly K), or, when lo_byte > 0, the K-th largest key
// with its lower bytes cleared (every key of equal upper bytes is >= t).
// Returns 0 when fewer than K keys are present.  Stops early once the chosen
// bin holds exactly the remaining count.  Every selector thread (stid =
// 0 .. kTkSelThreads-1) calls it; it synchronises them on kBarSel.
template <int SW>
__device__ uint64_t sel_kth_largest(const uint64_t *keys, int n, int K, int hi_byte, int lo_byte,
                                    SelScratch &sc, int stid)
{
    constexpr int kTkSelThreads = 32 * SW;
    uint64_t prefix = 0, mask = 0;
    int need = K;
    for (int byte = hi_byte; byte >= lo_byte; --byte) {
        for (int i = stid; i < 256; i += kTkSelThreads)
            sc.hist[i] = 0;
        named_sync(kBarSel, kTkSelThreads);
        const int sh = 8 * byte;
        for (int i = stid; i < n; i += kTkSelThreads) {
            const uint64_t k = keys[i];
            if (k != 0 && (k & mask) == prefix)
                atomicAdd(&sc.hist[(k >> sh) & 255u], 1u);
        }
        named_sync(kBarSel, kTkSelThreads);
        if (stid < 32)
            pick_bin(sc, need, stid);
        named_sync(kBarSel, kTkSelThreads);
        const int bin = sc.bin, nd = sc.need;
        named_sync(kBarSel, kTkSelThreads);
        if (bin < 0)
            return 0;
        prefix |= (uint64_t)bin << sh;
        mask |= (uint64_t)255u << sh;
        if (nd < 0)  // every key of this prefix is selected
            return prefix;
        need = nd;
    }
    return prefix;
}

// Buckets of the 16-bit pair x at or above m.
__device__ __forceinline__ int count_ge2(uint32_t x, uint32_t m)
{
    return (int)((x & 0xFFFFu) >= m) + (int)((x >> 16) >= m);
}

// Sorts keys[0, n) (n a power of two, distinct keys but for 0 padding) in
// descending order: bitonic network over NT threads, each thread loading U pairs
// before it compares and stores any, synchronised by sync() after every step.
template <int U, int NT, class Sync>
__device__ __forceinline__ void sort_desc(uint64_t *keys, int n, int tid, Sync &&sync)
{
    const int np = n / 2;  // pairs per step
    for (int k = 2; k <= n; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i0 = tid; i0 < np; i0 += U * NT) {
                uint64_t x[U], y[U];
                int l[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int i = i0 + u * NT;
                    l[u] = 2 * i - (i & (j - 1));
                    if (i < np) {
                        x[u] = keys[l[u]];
                        y[u] = keys[l[u] + j];
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    // blocks with (l & k) == 0 descending, the others ascending; the last merge
                    // (k = n) is descending throughout
                    if (i0 + u * NT < np && (x[u] < y[u]) == ((l[u] & k) == 0)) {
                        keys[l[u]] = y[u];
                        keys[l[u] + j] = x[u];
                    }
                }
            }
            sync();
        }
}

struct TopkArgs {
    const void *zs, *zt;
    int64_t ld, vocab;
    int32_t K;
    const int4 *rows;
    const int32_t *nvalid;
    int32_t *topk_ids;   // [T, K] or null
    float *topk_grad;    // [T, K] or null
    void *grad;          // [R, ld] or null
    int32_t grad_dtype;
    float *token_loss;
    double *row_wl;
    int32_t *status;
};

// Dynamic shared memory: candidate keys, the K selected keys, candidate student
// logits, the K selected student logits / gradients, then two buffers of one
// 16-bit bucket per group of 16 ids.
__host__ __device__ __forceinline__ size_t topk_fixed_bytes(int K)
{
    return align256((sizeof(uint64_t) + sizeof(float)) * ((size_t)topk_cap(K) + (size_t)K));
}

__host__ __device__ __forceinline__ int64_t topk_groups(int64_t V) { return (V + kTkGroup - 1) / kTkGroup; }

__host__ __device__ __forceinline__ size_t topk_bucket_bytes(int64_t V)
{
    return align256(sizeof(uint16_t) * (size_t)topk_groups(V));
}

size_t topk_smem_bytes(int64_t V, int K) { return topk_fixed_bytes(K) + 2 * topk_bucket_bytes(V); }

// Who writes a dense gradient row's zeros: the selector warps, but on fp32 rows of 14,336 to 65,536
// ids the streaming warps (us of a step of 2e8 logits, by the selectors and by the stream: bf16 V =
// 16,384, K = 30 244 and 255; 151,936, K = 256 206 and 214; fp32, K = 30, 8,192 470 and 491, 16,384
// 320 and 304, 32,768 285 and 272, 151,936 275 and 281; K = 320, 32,768 543 and 522, 98,304 340 and 354).
enum DenseRow { kNoDense = 0, kZerosBySelectors = 1, kZerosByStream = 2 };

// One CTA holds two rows at a time: its streaming warps run pass A and the
// bound of row i + 1 (into bucket buffer (i + 1) % 2) while its SW selector
// warps run collect, select and the KL of row i from buffer i % 2, so the SM's
// teacher stream does not pause for the latency-bound phases.
template <bool BF16, int SW, int DN>
__global__ void __launch_bounds__(kTkStreamThreads + 32 * SW, kTkMinBlocks) k_topk_rows(TopkArgs a)
{
    constexpr int kTkSelWarps = SW, kTkSelThreads = 32 * SW, kTkThreads = kTkStreamThreads + kTkSelThreads;
    // the loss sum after this grid may take the first SM it frees (it waits for the grid)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    extern __shared__ __align__(128) uint64_t tk_smem[];
    const int K = a.K;
    uint64_t *s_cand = tk_smem;
    const int cap = topk_cap(K);
    uint64_t *s_top = s_cand + cap;
    float *s_cz = reinterpret_cast<float *>(s_top + K);   // student logit of each candidate
    float *s_g = s_cz + cap;                               // selected: student logit, then g
    uint16_t *s_bucket0 = reinterpret_cast<uint16_t *>(reinterpret_cast<unsigned char *>(tk_smem) +
                                                       topk_fixed_bytes(K));
    __shared__ SelScratch s_sel;
    __shared__ int4 s_meta[2];      // per buffer: the row (token, row, -, weight bits)

    __shared__ int s_n, s_over;
    __shared__ __align__(16) uint32_t s_wtop[2][kTkLaneBoundMaxK];  // per buffer: each warp's 8 largest lane maxima
    __shared__ uint32_t s_tau[2];                     // per buffer: the bound (ordered logit)
    __shared__ int s_ng[2];                           // per buffer: candidate groups found
    __shared__ uint16_t s_glist[2][kTkGroupCap];      // per buffer: their indices
    __shared__ uint16_t s_wq[kTkSelWarps][kTkQueue];  // per selector warp: groups found, not yet read
    __shared__ int s_scnt[2][kTkStreamWarps];         // per streaming warp: a count of buckets
    __shared__ uint32_t s_smax[kTkStreamWarps];       // per streaming warp: its largest bucket

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_rows = *a.nvalid;
    const int n_it = n_rows > (int)blockIdx.x ? (n_rows - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
    const size_t esz = BF16 ? 2 : 4;
    const bool vec_ok =
        ((reinterpret_cast<uintptr_t>(a.zt) | reinterpret_cast<uintptr_t>(a.zs) | (uintptr_t)(a.ld * esz)) & 15u) == 0;
    const int64_t ng = topk_groups(a.vocab);
    const int ngv = vec_ok ? (int)(a.vocab / kTkGroup) : 0;  // whole groups read as vectors
    const size_t bucket_elems = topk_bucket_bytes(a.vocab) / sizeof(uint16_t);
    constexpr int VPG = BF16 ? 2 : 4;  // 16-byte vectors per group
    // lower bound of the K-th largest logit: up to K = 96 every streaming warp contributes
    // the 8 largest of its lanes' maxima, and the K-th largest of these distinct elements
    // cannot exceed the row's K-th largest; above, the streaming warps take the K-th
    // largest thread maximum or group bucket.  SW tells which at compile time, but for fp32 rows on
    // two selector warps, which launch_topk also gives some K above 96.  (Tested at run time, bf16
    // rows of few K took 3-7 % longer: V = 12,288, K = 20, dense row, 314 us, now 295.)
    constexpr bool kOneBound = SW != kTkSelSmall || BF16;
    const bool lane_bound = kOneBound ? SW == kTkSelSmall : K <= kTkLaneBoundMaxK;

    // the dense gradient row's zeros, by nt threads
    auto zero_row = [&](int row, int t0, int nt) {
        const size_t gesz = a.grad_dtype == TURNOPD_BF16 ? 2 : 4;
        char *grow = static_cast<char *>(a.grad) + (size_t)row * (size_t)a.ld * gesz;
        const int64_t bytes = a.vocab * (int64_t)gesz;
        // 16-byte stores between a head up to the first 16-byte boundary and a tail
        const int64_t head = min(bytes, (int64_t)((16u - (reinterpret_cast<uintptr_t>(grow) & 15u)) & 15u));
        const int64_t nv16 = (bytes - head) / 16;
        uint4 *body = reinterpret_cast<uint4 *>(grow + head);
        for (int64_t q = t0; q < nv16; q += nt)
            __stcs(body + q, make_uint4(0, 0, 0, 0));
        for (int64_t q = t0; q < head / 2; q += nt)
            reinterpret_cast<uint16_t *>(grow)[q] = 0;
        for (int64_t q = (head + nv16 * 16) / 2 + t0; q < bytes / 2; q += nt)
            reinterpret_cast<uint16_t *>(grow)[q] = 0;
    };

    if (warp < kTkStreamWarps) {
        // ---- streaming warps: pass A, one row after another
        constexpr int U = 8 / VPG;  // groups per batch
        // one batch of whole groups: 8 loads (128 B) in flight per thread
        uint4 v[U * VPG];
        auto load_batch = [&](const uint4 *rv, int g0) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int g = g0 + u * kTkStreamThreads;
#pragma unroll
                for (int q = 0; q < VPG; ++q)
                    if (g < ngv)
                        v[u * VPG + q] = __ldg(rv + (size_t)g * VPG + q);
            }
        };
        auto row_vectors = [&](const int4 &mr) {
            return reinterpret_cast<const uint4 *>(static_cast<const char *>(a.zt) + (size_t)mr.y * (size_t)a.ld * esz);
        };
        // The largest value x <= hi with at least K counted at or above it (0: none), by binary
        // search; warp_count(x) is a warp's count.  The first pass probes 255 below hi (where
        // the K-th largest bucket of a row with a few hundred large logits lies), and only when
        // fewer than K reach that does the search span the rest.  The warps' counts alternate
        // between two rows of s_scnt, so one barrier a pass suffices: a pass's reads finish
        // before any thread passes the next barrier.
        auto kth_bucket = [&](uint32_t hi, auto &&warp_count) {
            uint32_t lo = 0;  // count(>= lo) >= K or lo = 0; the answer is in [lo, hi]
            const uint32_t probe = hi > 255u ? hi - 255u : 0u;
            for (int par = 0, first = 1; lo < hi; par ^= 1, first = 0) {
                const uint32_t mid = first && probe > lo ? probe : (lo + hi + 1) >> 1;
                const int c = warp_count(mid);
                if (lane == 0)
                    s_scnt[par][warp] = c;
                named_sync(kBarStream, kTkStreamThreads);
                int tot = 0;
#pragma unroll
                for (int w = 0; w < kTkStreamWarps; ++w)
                    tot += s_scnt[par][w];
                if (tot >= K)
                    lo = mid;
                else
                    hi = mid - 1;
            }
            return lo;
        };
        int4 m_next = n_it > 0 ? a.rows[blockIdx.x] : make_int4(0, 0, -1, 0);
        if (n_it > 0)
            load_batch(row_vectors(m_next), tid);  // the first batch of each row is loaded a row ahead
        for (int it = 0; it < n_it; ++it) {
            const int b = it & 1;
            const int4 m = m_next;  // loaded one row ahead
            if (it + 1 < n_it)
                m_next = a.rows[blockIdx.x + (it + 1) * gridDim.x];
            if (it >= 2)
                named_sync(kBarFree + b, kTkThreads);  // the selectors are done with row it - 2
            if (tid == 0) {
                s_meta[b] = m;
                s_tau[b] = 0;
            }
            const char *zt_row = static_cast<const char *>(a.zt) + (size_t)m.y * (size_t)a.ld * esz;
            uint16_t *s_bucket = s_bucket0 + b * bucket_elems;
            bool refine = false;  // the bound came from the thread maxima (below)
            // group buckets and the thread's largest logit; whole groups of a 16-byte
            // aligned row are read as vectors, a batch at a time
            uint32_t tmax = 0;
            const uint4 *rv = reinterpret_cast<const uint4 *>(zt_row);
            for (int g0 = tid; g0 < ngv; g0 += U * kTkStreamThreads) {
                if (g0 != tid)
                    load_batch(rv, g0);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int g = g0 + u * kTkStreamThreads;
                    if (g >= ngv)
                        break;
                    uint32_t o;
                    if (BF16) {
                        const uint32_t o0 = bf16_max8_ord(v[u * 2]), o1 = bf16_max8_ord(v[u * 2 + 1]);
                        o = max(o0, o1);
                    } else {
                        float mx = -INFINITY;
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            mx = fmaxf(mx, fmaxf(fmaxf(__uint_as_float(v[u * 4 + q].x), __uint_as_float(v[u * 4 + q].y)),
                                                 fmaxf(__uint_as_float(v[u * 4 + q].z), __uint_as_float(v[u * 4 + q].w))));
                        o = ord32(__float_as_uint(mx));
                    }
                    s_bucket[g] = (uint16_t)bucket<BF16>(o);
                    tmax = max(tmax, o);
                }
            }
            // the selectors write the K values over the zeros once this row's buffer is full
            if (DN == kZerosByStream)
                zero_row(m.y, tid, kTkStreamThreads);
            // groups left: the partial last group, or every group of a misaligned row
            for (int g = ngv + tid; g < (int)ng; g += kTkStreamThreads) {
                const uint32_t o = group_max_ord_scalar<BF16>(zt_row, a.vocab, g);
                s_bucket[g] = (uint16_t)bucket<BF16>(o);
                tmax = max(tmax, o);
            }
            if (it + 1 < n_it)
                load_batch(row_vectors(m_next), tid);  // in flight while the row is settled below
            if (lane_bound) {
                // the warp's 8 largest lane maxima: a bitonic sort of the 32 in registers,
                // descending, leaves them in lanes 0..7
                uint32_t x = tmax;
#pragma unroll
                for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
                    for (int j = k >> 1; j > 0; j >>= 1) {
                        const uint32_t y = __shfl_xor_sync(0xffffffffu, x, j);
                        x = (((lane & j) == 0) == ((lane & k) == 0)) ? max(x, y) : min(x, y);
                    }
                if (lane < kTkLaneTop)
                    s_wtop[b][warp * kTkLaneTop + lane] = x;
            }
            if (tid == 0)
                s_ng[b] = 0;
            named_sync(kBarStream, kTkStreamThreads);
            if (lane_bound) {
                constexpr int nw = kTkStreamWarps * kTkLaneTop;
                const uint4 *w4 = reinterpret_cast<const uint4 *>(s_wtop[b]);
                for (int u0 = tid; u0 < nw; u0 += kTkStreamThreads) {
                    const uint32_t v = s_wtop[b][u0];
                    int gt = 0, ge = 0;
#pragma unroll
                    for (int q = 0; q < nw / 4; ++q) {
                        const uint4 x = w4[q];
                        gt += (x.x > v) + (x.y > v) + (x.z > v) + (x.w > v);
                        ge += (x.x >= v) + (x.y >= v) + (x.z >= v) + (x.w >= v);
                    }
                    if (v != 0 && gt < K && ge >= K)
                        s_tau[b] = v;  // every such thread writes the same value
                }
            } else if (!(kOneBound && SW == kTkSelSmall) && a.vocab > cap) {
                // the K-th largest group bucket, by binary search on its value with counts of
                // the buckets at or above it: K groups each hold an element that large (no
                // bound, tau = 0, when the row has fewer than K groups)
                const uint4 *b4 = reinterpret_cast<const uint4 *>(s_bucket);
                const int n4 = (int)ng / 8;
                const uint32_t wmax = __reduce_max_sync(0xffffffffu, bucket<BF16>(tmax));
                if (lane == 0)
                    s_smax[warp] = wmax;
                named_sync(kBarStream, kTkStreamThreads);
                uint32_t hi = 0;
#pragma unroll
                for (int w = 0; w < kTkStreamWarps; ++w)
                    hi = max(hi, s_smax[w]);
                // Up to three quarters of the threads the K-th largest thread maximum stands in for
                // the K-th largest bucket: also K distinct elements, at most n ln 4 = 1.4 n elements
                // of a row reach it (n threads), and its passes count registers where the others
                // walk the row's buckets.
                const int n_thr = min((int)ng, kTkStreamThreads);
                const bool by_thread = K <= n_thr / 4 * 3;
                refine = by_thread && K > (BF16 ? kRefineMinK : kRefineMinKF32);
                const uint32_t tb = bucket<BF16>(tmax);
                uint32_t lo;
                if (by_thread)
                    lo = kth_bucket(hi, [&](uint32_t mid) { return __popc(__ballot_sync(0xffffffffu, tb >= mid)); });
                else
                    lo = kth_bucket(hi, [&](uint32_t mid) {
                        int c = 0;
                        for (int i = tid; i < n4; i += kTkStreamThreads) {
                            const uint4 q = b4[i];
                            c += count_ge2(q.x, mid) + count_ge2(q.y, mid) + count_ge2(q.z, mid) + count_ge2(q.w, mid);
                        }
                        for (int g = n4 * 8 + tid; g < (int)ng; g += kTkStreamThreads)
                            c += (uint32_t)s_bucket[g] >= mid;
                        return (int)__reduce_add_sync(0xffffffffu, c);
                    });
                if (tid == 0)
                    s_tau[b] = BF16 ? lo : lo << 16;
            }
            named_sync(kBarStream, kTkStreamThreads);
            // the whole groups that can hold an element >= tau: their bucket reaches tau's
            // (eight buckets a load; the list's order does not matter)
            const uint32_t taub = bucket<BF16>(s_tau[b]);
            auto list = [&](int g) {
                const int p = atomicAdd(&s_ng[b], 1);
                if (p < kTkGroupCap)
                    s_glist[b][p] = (uint16_t)g;
            };
            const uint4 *b8 = reinterpret_cast<const uint4 *>(s_bucket);
            const int n8 = ngv / 8;
            for (int i = tid; i < n8; i += kTkStreamThreads) {
                const uint4 q = b8[i];
                const uint32_t w4[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if (((w4[e >> 1] >> (16 * (e & 1))) & 0xFFFFu) >= taub)
                        list(i * 8 + e);
            }
            for (int g = n8 * 8 + tid; g < ngv; g += kTkStreamThreads)
                if (s_bucket[g] >= taub)
                    list(g);
            if (!(kOneBound && SW == kTkSelSmall) && refine) {
                // The list (about 1.6 K groups) holds every group whose bucket reaches the bound,
                // so the K-th largest bucket among the listed is the row's: K groups are at or
                // above it, and the list shrinks to those and its ties.
                named_sync(kBarStream, kTkStreamThreads);
                const int nl = s_ng[b];
                if (nl > K && nl <= kRefine * kTkStreamThreads && nl <= kTkGroupCap) {
                    uint16_t lg[kRefine];
                    uint32_t lb[kRefine];
                    uint32_t mx = 0;
#pragma unroll
                    for (int e = 0; e < kRefine; ++e) {
                        const int i = tid + e * kTkStreamThreads;
                        lg[e] = i < nl ? s_glist[b][i] : 0;
                        lb[e] = i < nl ? s_bucket[lg[e]] : 0u;
                        mx = max(mx, lb[e]);
                    }
                    mx = __reduce_max_sync(0xffffffffu, mx);
                    if (lane == 0)
                        s_smax[warp] = mx;
                    named_sync(kBarStream, kTkStreamThreads);
                    uint32_t hi = 0;
#pragma unroll
                    for (int w = 0; w < kTkStreamWarps; ++w)
                        hi = max(hi, s_smax[w]);
                    const uint32_t kth = kth_bucket(hi, [&](uint32_t mid) {
                        int c = 0;
#pragma unroll
                        for (int e = 0; e < kRefine; ++e)
                            c += __popc(__ballot_sync(0xffffffffu, lb[e] >= mid));
                        return c;
                    });
                    if (tid == 0) {
                        s_tau[b] = max(s_tau[b], BF16 ? kth : kth << 16);
                        s_ng[b] = 0;
                    }
                    named_sync(kBarStream, kTkStreamThreads);
#pragma unroll
                    for (int e = 0; e < kRefine; ++e)
                        if (tid + e * kTkStreamThreads < nl && lb[e] >= kth)
                            list(lg[e]);
                }
            }
            named_arrive(kBarFull + b, kTkThreads);  // row it is in buffer b
        }
        return;
    }

    // ---- selector warps: the phases after pass A, one row behind the stream
    const int stid = tid - kTkStreamThreads, swarp = stid >> 5;
    const int hi_val = BF16 ? 5 : 7;  // top byte of the ordered logit inside a key
    for (int it = 0; it < n_it; ++it) {
        const int b = it & 1;
        const int j = blockIdx.x + it * gridDim.x;
        named_sync(kBarFull + b, kTkThreads);
        const int4 m = s_meta[b];
        const int tok = m.x;
        const float w = __int_as_float(m.w);
        const char *zt_row = static_cast<const char *>(a.zt) + (size_t)m.y * (size_t)a.ld * esz;
        const char *zs_row = static_cast<const char *>(a.zs) + (size_t)m.y * (size_t)a.ld * esz;
        const uint16_t *s_bucket = s_bucket0 + b * bucket_elems;
        if (stid == 0) {
            s_n = 0;
            s_over = 0;
        }
        named_sync(kBarSel, kTkSelThreads);
        uint64_t tau = (uint64_t)s_tau[b] << 32;  // admits every id of logit >= tau's
        const int n_listed = s_ng[b];

        auto append = [&](uint64_t k, float zsv) {
            const int p = atomicAdd(&s_n, 1);
            if (p < cap) {
                s_cand[p] = k;
                s_cz[p] = zsv;
            } else {
                s_over = 1;
            }
        };
        const uint4 *rv = reinterpret_cast<const uint4 *>(zt_row);
        const uint4 *sv = reinterpret_cast<const uint4 *>(zs_row);
        // the candidate elements of one whole group: teacher vectors vt, student vectors vs
        auto scan_group = [&](const uint4 *vt, const uint4 *vs, int g) {
            uint32_t o[kTkGroup];
            unpack_ords<BF16>(vt, o);
            const uint32_t e0 = (uint32_t)g * kTkGroup;
#pragma unroll
            for (int e = 0; e < kTkGroup; ++e) {
                const uint64_t k = mkkey(o[e], e0 + e);
                if (k >= tau) {
                    const uint4 &x = vs[e / (16 / (int)esz)];
                    const int wi = (e % (16 / (int)esz)) * (int)esz / 4;
                    const uint32_t word = wi == 0 ? x.x : wi == 1 ? x.y : wi == 2 ? x.z : x.w;
                    const float zsv = BF16 ? __uint_as_float(((e & 1) ? word >> 16 : word & 0xFFFFu) << 16)
                                           : __uint_as_float(word);
                    append(k, zsv);
                }
            }
        };
        // visit(g, ok) for the whole groups (g < ngv) whose bucket reaches tb, one per lane
        // and call, the lanes converged.  Each warp walks its share of the buckets in step,
        // queues the groups that pass (ballot) in its ring in shared memory, and visits 32 at a
        // time, so the lanes' loads are in flight together (a lane that visited its groups
        // alone would hold the warp for one memory round trip per group).
        auto walk_groups = [&](uint32_t tb, auto &&visit) {
            uint16_t *q = s_wq[swarp];
            uint32_t head = 0, tail = 0;  // warp-uniform
            for (int g0 = swarp * 32; g0 < ngv; g0 += kTkSelThreads) {
                const int g = g0 + lane;
                const bool pass = g < ngv && s_bucket[g] >= tb;
                const unsigned hit = __ballot_sync(0xffffffffu, pass);
                if (pass)
                    q[(tail + __popc(hit & ((1u << lane) - 1u))) & (kTkQueue - 1)] = (uint16_t)g;
                tail += __popc(hit);
                __syncwarp();
                if (tail - head >= 32) {
                    const int gq = q[(head + lane) & (kTkQueue - 1)];
                    __syncwarp();
                    head += 32;
                    visit(gq, true);
                }
            }
            if (head != tail) {  // fewer than 32 left
                const bool ok = lane < (int)(tail - head);
                const int gq = ok ? q[(head + lane) & (kTkQueue - 1)] : 0;
                __syncwarp();
                visit(gq, ok);
            }
        };
        // the candidate elements of group g (ok): teacher and student vectors loaded together
        auto take_one = [&](int g, bool ok) {
            if (!ok)
                return;
            uint4 vt[VPG], vs[VPG];
#pragma unroll
            for (int q = 0; q < VPG; ++q) {
                vt[q] = __ldg(rv + (size_t)g * VPG + q);
                vs[q] = __ldg(sv + (size_t)g * VPG + q);
            }
            scan_group(vt, vs, g);
        };
        // elements >= tau live in groups whose bucket reaches tau's: the groups the
        // streaming warps listed, or (list overflow, raised tau) a walk over the buckets
        auto collect = [&](bool listed) {
            const uint32_t tb = bucket<BF16>((uint32_t)(tau >> 32));
            if (listed) {
                for (int i = stid; i < n_listed; i += kTkSelThreads)
                    take_one((int)s_glist[b][i], true);
            } else {
                walk_groups(tb, take_one);
            }
            // the partial last group and misaligned rows, element by element
            for (int g = ngv + stid; g < (int)ng; g += kTkSelThreads) {
                if (s_bucket[g] < tb)
                    continue;
                const int64_t e0 = (int64_t)g * kTkGroup;
                for (int64_t e = e0; e < e0 + kTkGroup && e < a.vocab; ++e) {
                    const uint64_t k = mkkey(elem_ord<BF16>(zt_row, e), (uint32_t)e);
                    if (k >= tau)
                        append(k, BF16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(zs_row)[e])
                                       : reinterpret_cast<const float *>(zs_row)[e]);
                }
            }
        };
        // f(k) for every key >= lo of the row: the whole groups whose bucket reaches
        // lo's are read again (teacher only, a group per lane in step), the partial
        // last group and misaligned rows element by element
        auto each_key = [&](uint64_t lo, auto &&f) {
            const uint32_t tb = bucket<BF16>((uint32_t)(lo >> 32));
            walk_groups(tb, [&](int g, bool ok) {
                if (!ok)
                    return;
                uint4 vt[VPG];
#pragma unroll
                for (int q = 0; q < VPG; ++q)
                    vt[q] = __ldg(rv + (size_t)g * VPG + q);
                uint32_t o[kTkGroup];
                unpack_ords<BF16>(vt, o);
                const uint32_t e0 = (uint32_t)g * kTkGroup;
#pragma unroll
                for (int e = 0; e < kTkGroup; ++e) {
                    const uint64_t k = mkkey(o[e], e0 + e);
                    if (k >= lo)
                        f(k);
                }
            });
            for (int g = ngv + stid; g < (int)ng; g += kTkSelThreads) {
                if (s_bucket[g] < tb)
                    continue;
                const int64_t e0 = (int64_t)g * kTkGroup;
                for (int64_t e = e0; e < e0 + kTkGroup && e < a.vocab; ++e) {
                    const uint64_t k = mkkey(elem_ord<BF16>(zt_row, e), (uint32_t)e);
                    if (k >= lo)
                        f(k);
                }
            }
        };
        collect(n_listed <= kTkGroupCap);
        named_sync(kBarSel, kTkSelThreads);
        if (s_over) {
            // ---- overflow: radix select over the row's keys >= tau, one key byte per
            // pass from the top, until the keys >= the chosen prefix fit the buffer.
            // Keys above the prefix number K - need; those with the prefix, cnt.
            uint64_t prefix = 0, pmask = 0;
            int need = K;
            for (int byte = hi_val; byte >= 0; --byte) {
                const int sh = 8 * byte;
                for (int i = stid; i < 256; i += kTkSelThreads)
                    s_sel.hist[i] = 0;
                named_sync(kBarSel, kTkSelThreads);
                each_key(max(tau, prefix), [&](uint64_t k) {
                    if ((k & pmask) == prefix)
                        atomicAdd(&s_sel.hist[(k >> sh) & 255u], 1u);
                });
                named_sync(kBarSel, kTkSelThreads);
                if (stid < 32)
                    pick_bin(s_sel, need, stid);
                named_sync(kBarSel, kTkSelThreads);
                const int bin = s_sel.bin, nd = s_sel.need;
                const int cnt = bin >= 0 ? (int)s_sel.hist[bin] : 0;
                named_sync(kBarSel, kTkSelThreads);
                if (bin < 0)
                    break;  // fewer than K keys >= tau: not reached, tau is a lower bound
                prefix |= (uint64_t)bin << sh;
                pmask |= (uint64_t)255u << sh;
                if (nd < 0 || K - nd + cnt <= cap)
                    break;
                need = nd;
            }
            tau = max(tau, prefix);
            if (stid == 0) {
                s_n = 0;
                s_over = 0;
            }
            named_sync(kBarSel, kTkSelThreads);
            collect(false);
            named_sync(kBarSel, kTkSelThreads);
        }
        const bool failed = s_over != 0;
        const int nc = min(s_n, cap);
        named_sync(kBarSel, kTkSelThreads);
        if (failed) {
            if (stid == 0) {
                set_status(a.status, TURNOPD_ERR_UNSUPPORTED);
                a.token_loss[tok] = 0.f;
                a.row_wl[j] = 0.0;
            }
        } else {
            if (nc > kTkRankMax) {
                // ---- the K largest of a large buffer: sort it (padded with 0 keys to a power
                // of two, at most the buffer's size) and take the first K
                // Each key carries its buffer position in its low 11 bits, below the id's 20:
                // ids are below 2^20, so ~id's upper 12 bits are ones and the order is kept.
                int n2 = 512;
                while (n2 < nc)
                    n2 <<= 1;
                for (int i = stid; i < n2; i += kTkSelThreads) {
                    const uint64_t k = s_cand[i];
                    s_cand[i] = i < nc ? (k & 0xFFFFFFFF00000000ull) | ((k & 0xFFFFFull) << 11) | (uint64_t)i : 0ull;
                }
                named_sync(kBarSel, kTkSelThreads);
                sort_desc<BF16 ? 4 : 2, kTkSelThreads>(s_cand, n2, stid, [&]() { named_sync(kBarSel, kTkSelThreads); });
                for (int r = stid; r < K; r += kTkSelThreads) {
                    const uint64_t p = s_cand[r];
                    s_top[r] = (p & 0xFFFFFFFF00000000ull) | 0xFFF00000ull | ((p >> 11) & 0xFFFFFull);
                    s_g[r] = s_cz[p & 0x7FFu];
                }
            } else {
                // ---- the K largest: each candidate's rank among the candidates is its position
                // (keys are unique).  A buffer of more than twice K is first cut to the K largest by
                // radix select; below that its passes cost more than the ranks they save.  Two keys
                // of the buffer are read a load, but for two warps and K > 16 (us of a step of 2e8
                // bf16 logits, pairs and singles: V = 8,192, K = 8 327 and 344, 30 383 and 378;
                // 151,936, K = 96 161 and 140).
                const uint64_t kth = nc <= max(2 * K, kTkSelThreads) ? 0 : sel_kth_largest<SW>(s_cand, nc, K, hi_val, 0, s_sel, stid);
                const bool singles = SW == kTkSelSmall && K > 16;
                if (!singles) {
                    if (stid == 0 && (nc & 1))
                        s_cand[nc] = 0;  // the last pair's second key
                    named_sync(kBarSel, kTkSelThreads);
                }
                const ulonglong2 *pairs = reinterpret_cast<const ulonglong2 *>(s_cand);
                for (int i = stid; i < nc; i += kTkSelThreads) {
                    const uint64_t k = s_cand[i];
                    if (k < kth)
                        continue;
                    int rank = 0;
                    if (singles) {
                        int q = 0;
                        for (; q + 4 <= nc; q += 4)
                            rank += (s_cand[q] > k) + (s_cand[q + 1] > k) + (s_cand[q + 2] > k) + (s_cand[q + 3] > k);
                        for (; q < nc; ++q)
                            rank += s_cand[q] > k;
                    } else {
#pragma unroll 2
                        for (int q = 0; q < (nc + 1) / 2; ++q) {
                            const ulonglong2 x = pairs[q];
                            rank += (int)(x.x > k) + (int)(x.y > k);
                        }
                    }
                    if (rank < K) {
                        s_top[rank] = k;
                        s_g[rank] = s_cz[i];
                    }
                }
            }
            named_sync(kBarSel, kTkSelThreads);

            // ---- KL over S (one warp, fp32)
            if (swarp == 0) {
                float m_s = -INFINITY, m_t = -INFINITY;
                for (int r = lane; r < K; r += 32) {
                    const float zt_v = key_value<BF16>(s_top[r]);
                    const float zs_v = s_g[r];  // student logit, carried with the candidate
                    m_s = fmaxf(m_s, zs_v);
                    m_t = fmaxf(m_t, zt_v);
                }
                m_s = warp_max_f(m_s);
                m_t = warp_max_f(m_t);
                float s_s = 0.f, s_t = 0.f, a_sd = 0.f;
                for (int r = lane; r < K; r += 32) {
                    const float zs_v = s_g[r], zt_v = key_value<BF16>(s_top[r]);
                    const float es = expf(zs_v - m_s);
                    s_s += es;
                    s_t += expf(zt_v - m_t);
                    a_sd = fmaf(es, zs_v - zt_v, a_sd);
                }
                s_s = warp_sum_f(s_s);
                s_t = warp_sum_f(s_t);
                a_sd = warp_sum_f(a_sd);
                const float ep = a_sd / s_s;                              // E_p[z_s - z_t]
                const float c = (m_s - m_t) + logf(s_s / s_t);            // LSE_s - LSE_t
                const float ell = ep - c;
                for (int r = lane; r < K; r += 32) {
                    const float zs_v = s_g[r], zt_v = key_value<BF16>(s_top[r]);
                    const float p = expf(zs_v - m_s) / s_s;
                    const float g = w * p * ((zs_v - zt_v) - ep);
                    s_g[r] = g;
                    if (a.topk_ids)
                        a.topk_ids[(size_t)tok * K + r] = (int32_t)key_id(s_top[r]);
                    if (a.topk_grad)
                        a.topk_grad[(size_t)tok * K + r] = g;
                }
                if (lane == 0) {
                    if (!isfinite(ell))
                        set_status(a.status, TURNOPD_ERR_NONFINITE);
                    a.token_loss[tok] = ell;
                    a.row_wl[j] = (double)w * (double)ell;
                }
            }
            // ---- dense gradient row: zeros, then the K entries
            if (DN) {
                const size_t gesz = a.grad_dtype == TURNOPD_BF16 ? 2 : 4;
                char *grow = static_cast<char *>(a.grad) + (size_t)m.y * (size_t)a.ld * gesz;
                if (DN == kZerosBySelectors)
                    zero_row(m.y, stid, kTkSelThreads);
                named_sync(kBarSel, kTkSelThreads);  // zeros and every entry of s_g are written
                for (int r = stid; r < K; r += kTkSelThreads) {
                    const uint32_t id = key_id(s_top[r]);
                    if (a.grad_dtype == TURNOPD_BF16)
                        reinterpret_cast<__nv_bfloat16 *>(grow)[id] = __float2bfloat16_rn(s_g[r]);
                    else
                        reinterpret_cast<float *>(grow)[id] = s_g[r];
                }
            }
        }
        named_sync(kBarSel, kTkSelThreads);  // buffer b and the candidate arrays are free
        if (it + 2 < n_it)
            named_arrive(kBarFree + b, kTkThreads);
    }
}

// ---------------------------------------------------------------- short rows

// The loss of a row from its K selected: l, ids and sparse gradient out, s_g (the student
// logits) replaced by the gradient.  One warp, fp32.
template <bool BF16>
__device__ __forceinline__ void short_kl(const TopkArgs &a, const int4 &m, int j, const uint64_t *s_top, float *s_g,
                                         int lane)
{
    const int K = a.K, tok = m.x;
    const float w = __int_as_float(m.w);
    float m_s = -INFINITY, m_t = -INFINITY;
    for (int r = lane; r < K; r += 32) {
        m_s = fmaxf(m_s, s_g[r]);
        m_t = fmaxf(m_t, key_value<BF16>(s_top[r]));
    }
    m_s = warp_max_f(m_s);
    m_t = warp_max_f(m_t);
    float s_s = 0.f, s_t = 0.f, a_sd = 0.f;
    for (int r = lane; r < K; r += 32) {
        const float zs_v = s_g[r], zt_v = key_value<BF16>(s_top[r]);
        const float es = expf(zs_v - m_s);
        s_s += es;
        s_t += expf(zt_v - m_t);
        a_sd = fmaf(es, zs_v - zt_v, a_sd);
    }
    s_s = warp_sum_f(s_s);
    s_t = warp_sum_f(s_t);
    a_sd = warp_sum_f(a_sd);
    const float ep = a_sd / s_s;                    // E_p[z_s - z_t]
    const float c = (m_s - m_t) + logf(s_s / s_t);  // LSE_s - LSE_t
    const float ell = ep - c;
    for (int r = lane; r < K; r += 32) {
        const float zs_v = s_g[r], zt_v = key_value<BF16>(s_top[r]);
        const float g = w * (expf(zs_v - m_s) / s_s) * ((zs_v - zt_v) - ep);
        s_g[r] = g;
        if (a.topk_ids)
            a.topk_ids[(size_t)tok * K + r] = (int32_t)key_id(s_top[r]);
        if (a.topk_grad)
            a.topk_grad[(size_t)tok * K + r] = g;
    }
    if (lane == 0) {
        if (!isfinite(ell))
            set_status(a.status, TURNOPD_ERR_NONFINITE);
        a.token_loss[tok] = ell;
        a.row_wl[j] = (double)w * (double)ell;
    }
}

// Candidates a short row's CTA holds: the K selected and the ties of the last bucket.
__host__ __device__ constexpr int short_cap(int K) { return K <= 128 ? 256 : K <= 256 ? 512 : K <= 512 ? 1024 : 2048; }
// Ids it lists: where the last bucket holds more than the candidates, the K-th key is found among
// these.  (One-warp CTAs, 32 on an SM, keep the shared memory for the cache.)
__host__ __device__ constexpr int short_list(int K, int nt) { return nt == 32 || K > 512 ? short_cap(K) : 1024; }
__host__ __device__ __forceinline__ size_t short_smem(int K, int nt)
{
    return (sizeof(uint64_t) + sizeof(float)) * (size_t)(short_cap(K) + K) + sizeof(int32_t) * (size_t)short_list(K, nt) + 16;
}
constexpr int kShortPerThread = 64;  // elements of a row per thread
// Aligned rows up to here take the kernel below: what 128 threads hold, 256 from K = 64.
// k_topk_rows reads the other rows faster.  us of a step of 2e8 bf16 logits, here and there: V =
// 8,184, K = 8 275 and 386, 50 316 and 501, 96 356 and 1,890; V = 8,192 (256 threads), K = 64 551
// and 676; 12,288, K = 32 370 and 290, 50 392 and 322, 64 394 and 453; 16,376, K = 64 322 and 376,
// 256 516 and 879; 24,576 (512 threads), K = 80 434 and 284, 256 576 and 540, 288 606 and 576.
// fp32 rows cross at the same places.  Rows that are not 16-byte aligned, which k_topk_rows reads
// element by element, take it at every length it holds (32,700, K = 50: 1,248 GB/s and 448).
int short_max_vocab(int K) { return kShortPerThread * (K < 64 ? 128 : 256) - 7; }

template <bool BF16>
__device__ __forceinline__ uint64_t row_key(const char *zt_row, int id)
{
    return mkkey(elem_ord<BF16>(zt_row, id), (uint32_t)id);
}

// The K elements of largest key among `total` ids (listed in ids, or all of a row's), in any order,
// into key and cz: radix select of the K-th key, a byte a pass (ids are below 65,536, so ~id's upper
// bytes are all ones), then every key at or above it.  Lanes of equal digit add up before the
// histogram, which a row of equal logits would serialise.  For rows with more ties than a short row's
// CTA holds, fewer than K finite logits, or a NaN.  (Bit by bit over the whole row, 48 or 64
// passes, before.  us of a step of 1e8 logits, K = 50: fp32 V = 4,096 with 1,000 added to every logit
// 3,604 and 418, with multiples of 3 3,395 and 464; bf16 8,176, multiples of 3, 1,809 and 247.)
template <bool BF16, int NT>
__device__ __forceinline__ void short_ties(const char *zt_row, const char *zs_row, const int32_t *ids, int total, int K,
                                           uint64_t *key, float *cz, int *n)
{
    static_assert(sizeof(SelScratch) <= 256 * sizeof(uint64_t), "key is free until the keys are collected");
    SelScratch &sc = *reinterpret_cast<SelScratch *>(key);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    auto sync = [&]() {
        if (NT == 32)
            __syncwarp();
        else
            __syncthreads();
    };
    uint64_t prefix = 0xFFFF0000ull, mask = 0xFFFF0000ull;
    int need = K;
    for (int byte = BF16 ? 5 : 7; byte >= 0; byte -= byte == 4 ? 3 : 1) {
        for (int i = tid; i < 256; i += NT)
            sc.hist[i] = 0;
        sync();
        for (int i0 = warp * 32; i0 < total; i0 += NT) {
            const int i = i0 + lane;
            uint32_t digit = 256;
            if (i < total) {
                const uint64_t k = row_key<BF16>(zt_row, ids ? ids[i] : i);
                if ((k & mask) == (prefix & mask))
                    digit = (uint32_t)(k >> (8 * byte)) & 255u;
            }
            const unsigned same = __match_any_sync(0xffffffffu, digit);
            if (digit < 256 && lane == __ffs(same) - 1)
                atomicAdd(&sc.hist[digit], (uint32_t)__popc(same));
        }
        sync();
        if (warp == 0)
            pick_bin(sc, need, lane);
        sync();
        const int bin = sc.bin, nd = sc.need;
        sync();
        prefix |= (uint64_t)bin << (8 * byte);
        mask |= 255ull << (8 * byte);
        if (nd < 0)  // every key of this prefix is among the K
            break;
        need = nd;
    }
    if (tid == 0)
        *n = 0;
    sync();
    for (int i = tid; i < total; i += NT) {
        const int id = ids ? ids[i] : i;
        const uint64_t k = row_key<BF16>(zt_row, id);
        if (k >= prefix) {
            const int p = atomicAdd(n, 1);
            key[p] = k;
            cz[p] = BF16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(zs_row)[id])
                         : reinterpret_cast<const float *>(zs_row)[id];
        }
    }
}

// The same as a call, for the one-warp CTA, whose registers are all in use (inlined there it cost the
// ordinary rows 2-6 %, as a call in the larger CTAs 8-12 %).
template <bool BF16>
__device__ __noinline__ void short_ties_call(const char *zt_row, const char *zs_row, const int32_t *ids, int total,
                                             int K, uint64_t *key, float *cz, int *n)
{
    short_ties<BF16, 32>(zt_row, zs_row, ids, total, K, key, cz, n);
}

// The K largest of n candidates (a power of two above n fits the buffer) in order: a bitonic sort, as in
// k_topk_rows, each key carrying its buffer position below the id's 20 bits.
template <int NT>
__device__ __forceinline__ void short_sort(uint64_t *key, const float *cz, int n, int K, uint64_t *top, float *g)
{
    const int tid = threadIdx.x;
    auto sync = [&]() {
        if (NT == 32)
            __syncwarp();
        else
            __syncthreads();
    };
    int n2 = 512;
    while (n2 < n)
        n2 <<= 1;
    for (int i = tid; i < n2; i += NT) {
        const uint64_t k = key[i];
        key[i] = i < n ? (k & 0xFFFFFFFF00000000ull) | ((k & 0xFFFFFull) << 11) | (uint64_t)i : 0ull;
    }
    sync();
    sort_desc<2, NT>(key, n2, tid, sync);
    for (int r = tid; r < K; r += NT) {
        const uint64_t p = key[r];
        top[r] = (p & 0xFFFFFFFF00000000ull) | 0xFFF00000ull | ((p >> 11) & 0xFFFFFull);
        g[r] = cz[p & 0x7FFu];
    }
}
// Rows of up to 64 NT elements, one CTA of NT threads a row, any alignment: the row's
// 16-bit buckets (the logit itself for bf16) stay in registers, 2 to a word, from the only
// read of the teacher.  The K-th largest bucket comes from a binary search on its value, a
// compare and an add per pair and pass (bf16x2); the elements at or above it, K and the
// ties of the last bucket, are ranked by their full keys.  k_topk_rows spends 10 us and
// more a row on its two roles' hand-over and selection, whatever the row's length, with 608
// rows in flight, and its bound fails where a row has fewer groups than K; here a short row
// holds one to sixteen warps, up to 4,864 are in flight.  Bound by issue (3,200 warp
// instructions a row of 2,034 at K = 50, IPC 1.9).  GB/s of the step at 4e8 logits, bf16, in
// k_topk_rows and here: K = 50, V = 1,024 47 and 653, 2,034 47 and 988, 4,096 437 and 788;
// K = 256 82 and 265, 65 and 368, 101 and 463.
// SORT: the candidates are sorted, for K from 320 (kShortSortK), where ranks, whose cost grows with the
// square, take longer (us of a step of 1e8 bf16 logits, ranks and sort: V = 1,040, K = 320 2,950 and
// 2,154, 1,024 34,733 and 7,752; 4,096, K = 512 1,381 and 986, 1,024 4,790 and 2,149; 12,288, K = 256 319
// and 361, 288 346 and 369, 320 367 and 371).  Kernels of their own: in one, the sort's registers cost
// the other rows 4-8 %.
constexpr int kShortSortK = 320;
template <bool BF16, int NT, bool SORT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_topk_short(TopkArgs a)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    constexpr int NW = NT / 32;
    constexpr int ESZ = BF16 ? 2 : 4;
    extern __shared__ __align__(128) uint64_t tk_smem[];
    const int K = a.K, cap = short_cap(K), listed = short_list(K, NT);
    uint64_t *s_key = tk_smem;                                 // [cap] candidates
    uint64_t *s_top = s_key + cap;                             // [K] selected
    float *s_cz = reinterpret_cast<float *>(s_top + K);        // [cap] their student logits
    float *s_g = s_cz + cap;                                   // [K]
    int32_t *s_id = reinterpret_cast<int32_t *>(s_g + K);      // [listed]
    __shared__ int s_cnt[2][NW];
    __shared__ float s_max[NW];
    __shared__ int s_n;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int V = (int)a.vocab;
    const int n_rows = *a.nvalid;
    auto sync = [&]() {
        if (NT == 32)
            __syncwarp();
        else
            __syncthreads();
    };
    int par = 0;  // the warps' counts alternate between two rows of s_cnt: one barrier a count
    auto block_count = [&](int c) {  // c: this thread's
        c = __reduce_add_sync(0xffffffffu, c);
        if (NT == 32)
            return c;
        if (lane == 0)
            s_cnt[par][warp] = c;
        __syncthreads();
        int tot = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w)
            tot += s_cnt[par][w];
        par ^= 1;
        return tot;
    };
    auto bits_of = [](uint32_t o) { return (o & 0x8000u) ? o & 0x7FFFu : ~o & 0xFFFFu; };
    auto splat2 = [](uint32_t bits) {
        const uint32_t w = bits | bits << 16;
        return *reinterpret_cast<const __nv_bfloat162 *>(&w);
    };

    for (int j = blockIdx.x; j < n_rows; j += gridDim.x) {
        const int4 m = a.rows[j];
        const char *zt_row = static_cast<const char *>(a.zt) + (size_t)m.y * (size_t)a.ld * ESZ;
        const char *zs_row = static_cast<const char *>(a.zs) + (size_t)m.y * (size_t)a.ld * ESZ;
        // the row starts `head` elements into a 16-byte vector; octet q holds ids 8 q - head ..
        const int head = (int)(reinterpret_cast<uintptr_t>(zt_row) & 15u) / ESZ;
        const int octets = (head + V + 7) / 8;
        __nv_bfloat162 bk[kShortPerThread / 2];
        const char *vec = zt_row - head * ESZ;
#pragma unroll
        for (int u = 0; u < kShortPerThread / 8; ++u) {
            const int q = tid + u * NT, i0 = q * 8 - head;
            uint32_t w[4] = {0xff80ff80u, 0xff80ff80u, 0xff80ff80u, 0xff80ff80u};  // -inf: no element
            if (q < octets) {
                if (i0 >= 0 && i0 + 8 <= V) {
                    const uint4 x = __ldg(reinterpret_cast<const uint4 *>(vec) + q * (ESZ / 2));
                    if (BF16) {
                        w[0] = x.x, w[1] = x.y, w[2] = x.z, w[3] = x.w;
                    } else {
                        const uint4 y = __ldg(reinterpret_cast<const uint4 *>(vec) + q * 2 + 1);
                        w[0] = __byte_perm(x.x, x.y, 0x7632), w[1] = __byte_perm(x.z, x.w, 0x7632);
                        w[2] = __byte_perm(y.x, y.y, 0x7632), w[3] = __byte_perm(y.z, y.w, 0x7632);
                    }
                } else {  // the first or the last octet: element by element
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        if (i0 + e >= 0 && i0 + e < V) {
                            const uint32_t b = BF16 ? reinterpret_cast<const uint16_t *>(zt_row)[i0 + e]
                                                    : reinterpret_cast<const uint32_t *>(zt_row)[i0 + e] >> 16;
                            w[e / 2] = e & 1 ? (w[e / 2] & 0xFFFFu) | b << 16 : (w[e / 2] & 0xFFFF0000u) | b;
                        }
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)  // + 0: -0 and +0 are the same logit
                bk[u * 4 + k] = __hadd2(*reinterpret_cast<const __nv_bfloat162 *>(&w[k]), splat2(0));
        }
        if (a.grad) {  // the dense gradient row's zeros
            const size_t gesz = a.grad_dtype == TURNOPD_BF16 ? 2 : 4;
            char *grow = static_cast<char *>(a.grad) + (size_t)m.y * (size_t)a.ld * gesz;
            const int64_t bytes = (int64_t)V * (int64_t)gesz;
            const int64_t gh = min(bytes, (int64_t)((16u - (reinterpret_cast<uintptr_t>(grow) & 15u)) & 15u));
            const int64_t nv16 = (bytes - gh) / 16;
            uint4 *body = reinterpret_cast<uint4 *>(grow + gh);
            for (int64_t q = tid; q < nv16; q += NT)
                __stcs(body + q, make_uint4(0, 0, 0, 0));
            for (int64_t q = tid; q < gh / 2; q += NT)
                reinterpret_cast<uint16_t *>(grow)[q] = 0;
            for (int64_t q = (gh + nv16 * 16) / 2 + tid; q < bytes / 2; q += NT)
                reinterpret_cast<uint16_t *>(grow)[q] = 0;
        }
        // the row's largest bucket, NaN if one is
        __nv_bfloat162 mx = bk[0];
#pragma unroll
        for (int k = 1; k < kShortPerThread / 2; ++k)
            mx = __hmax2_nan(mx, bk[k]);
        auto max_nan = [](float x, float y) { return x != x || y != y ? NAN : fmaxf(x, y); };
        float top = max_nan(__bfloat162float(mx.x), __bfloat162float(mx.y));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            top = max_nan(top, __shfl_xor_sync(0xffffffffu, top, o));
        if (NT > 32) {
            if (lane == 0)
                s_max[warp] = top;
            __syncthreads();
#pragma unroll
            for (int w = 0; w < NW; ++w)
                top = max_nan(top, s_max[w]);
        }
        auto count = [&](const __nv_bfloat162 &x) {  // this thread's elements >= x (at most 32 in a half: exact)
            __nv_bfloat162 c = splat2(0);
#pragma unroll
            for (int k = 0; k < kShortPerThread / 2; ++k)
                c = __hadd2(c, __hge2(bk[k], x));
            return (int)(__bfloat162float(c.x) + __bfloat162float(c.y));
        };
        // the K-th largest bucket: the largest x with at least K elements >= x.  The first probe
        // is 255 below the maximum (where the K-th largest of a row of a few thousand lies)
        uint32_t hi = ord16(__float_as_uint(top) >> 16), lo = 0x0080u;  // the lowest finite value: V >= K elements
        const uint32_t probe = hi > 255u + lo ? hi - 255u : lo;
        for (bool first = true; lo < hi; first = false) {
            const uint32_t mid = first && probe > lo ? probe : (lo + hi + 1) >> 1;
            if (block_count(count(splat2(bits_of(mid)))) >= K)
                lo = mid;
            else
                hi = mid - 1;
        }
        // the elements at or above it, in a fixed order
        const __nv_bfloat162 T = splat2(bits_of(lo));
        const int mine = __reduce_add_sync(0xffffffffu, count(T));
        int base = 0, n = mine;
        if (NT > 32) {
            if (lane == 0)
                s_cnt[par][warp] = mine;
            __syncthreads();
            n = 0;
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                base += w < warp ? s_cnt[par][w] : 0;
                n += s_cnt[par][w];
            }
            par ^= 1;
        }
        if (n <= listed && n >= K && top == top) {
            const uint32_t below = (1u << lane) - 1u;
#pragma unroll
            for (int k = 0; k < kShortPerThread / 2; ++k) {
                const unsigned hit = __hge2_mask(bk[k], T);
                if (!__any_sync(0xffffffffu, hit))
                    continue;
                const int id = (tid + k / 4 * NT) * 8 - head + k % 4 * 2;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const bool in = h ? hit >> 16 : hit & 0xFFFFu;
                    const unsigned who = __ballot_sync(0xffffffffu, in);
                    if (in)
                        s_id[base + __popc(who & below)] = id + h;
                    base += __popc(who);
                }
            }
            sync();
            if (n <= cap)
                for (int i = tid; i < n; i += NT) {
                    const int id = s_id[i];
                    s_key[i] = row_key<BF16>(zt_row, id);
                    s_cz[i] = BF16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(zs_row)[id])
                                   : reinterpret_cast<const float *>(zs_row)[id];
                }
        }
        if (n > cap || n < K || top != top) {
            const bool from_list = n <= listed && n >= K && top == top;
            const int32_t *ids = from_list ? s_id : nullptr;
            if (NT == 32)
                short_ties_call<BF16>(zt_row, zs_row, ids, from_list ? n : V, K, s_key, s_cz, &s_n);
            else
                short_ties<BF16, NT>(zt_row, zs_row, ids, from_list ? n : V, K, s_key, s_cz, &s_n);
            n = K;
        }
        if (SORT) {
            sync();
            short_sort<NT>(s_key, s_cz, n, K, s_top, s_g);
        } else {
            if (tid == 0 && (n & 1))
                s_key[n] = 0;  // the last pair's second key
            sync();
            // each candidate's rank among the candidates is its position
            const ulonglong2 *pairs = reinterpret_cast<const ulonglong2 *>(s_key);
            for (int i = tid; i < n; i += NT) {
                const uint64_t k = s_key[i];
                int rank = 0;
#pragma unroll 4
                for (int q = 0; q < (n + 1) / 2; ++q) {
                    const ulonglong2 x = pairs[q];
                    rank += (int)(x.x > k) + (int)(x.y > k);
                }
                if (rank < K) {
                    s_top[rank] = k;
                    s_g[rank] = s_cz[i];
                }
            }
        }
        sync();
        if (warp == 0)
            short_kl<BF16>(a, m, j, s_top, s_g, lane);
        if (a.grad) {
            sync();
            const size_t gesz = a.grad_dtype == TURNOPD_BF16 ? 2 : 4;
            char *grow = static_cast<char *>(a.grad) + (size_t)m.y * (size_t)a.ld * gesz;
            for (int r = tid; r < K; r += NT) {
                const uint32_t id = key_id(s_top[r]);
                if (a.grad_dtype == TURNOPD_BF16)
                    reinterpret_cast<__nv_bfloat16 *>(grow)[id] = __float2bfloat16_rn(s_g[r]);
                else
                    reinterpret_cast<float *>(grow)[id] = s_g[r];
            }
        }
        sync();  // the shared arrays are free
    }
}

// Masked tokens' sparse rows: ids -1, gradients 0.
__global__ void k_topk_zero_masked(const uint8_t *mask, int64_t T, int32_t K, int32_t *ids, float *g)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < T * K; i += (int64_t)gridDim.x * blockDim.x) {
        if (mask[i / K])
            continue;
        if (ids)
            ids[i] = -1;
        if (g)
            g[i] = 0.f;
    }
}

}  // namespace

cudaError_t launch_topk(const TopkCall &c, cudaStream_t stream)
{
    LossWorkspace ws = loss_workspace_layout(c.workspace, c.T);
    LossArgs la{};
    la.mask = c.mask;
    la.row_of_token = c.row_of_token;
    la.w = c.w;
    la.T = c.T;
    la.num_rows = c.num_rows;
    la.vocab = c.vocab;
    la.mode = TURNOPD_FULL_VOCAB;
    la.token_loss = c.token_loss;
    la.status = c.status;
    cudaError_t e = launch_compaction(la, ws.rows, ws.blk_count, ws.nvalid, stream);
    if (e != cudaSuccess)
        return e;
    const int sms = device_sm_count();
    if ((c.topk_ids || c.topk_grad) && (c.flags & TURNOPD_ZERO_MASKED_GRAD)) {
        const int grid = (int)std::min<int64_t>((c.T * c.K + 255) / 256, (int64_t)sms * 8);
        k_topk_zero_masked<<<std::max(grid, 1), 256, 0, stream>>>(c.mask, c.T, c.K, c.topk_ids, c.topk_grad);
    }
    if (c.grad && (c.flags & TURNOPD_ZERO_MASKED_GRAD))
        launch_zero_masked_grad(c.mask, c.row_of_token, c.T, c.num_rows, c.ld, c.vocab, c.grad, c.grad_dtype,
                                stream);
    TopkArgs a{c.zs, c.zt, c.ld, c.vocab, c.K, ws.rows, ws.nvalid, c.topk_ids, c.topk_grad, c.grad,
               c.grad_dtype, c.token_loss, ws.row_wl, c.status};
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess)
        return e;
    using Kern = void (*)(TopkArgs);
    static size_t attr_smem[64][28] = {};
    const int di = dev < 64 ? dev : 0;
    auto launch = [&](Kern kern, int slot, int threads, size_t smem) {
        cudaError_t e = cudaSuccess;
        if (attr_smem[di][slot] < smem) {
            if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
                return e;
            attr_smem[di][slot] = smem;
        }
        int nb = 0;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, threads, smem)) != cudaSuccess)
            return e;
        if (nb < 1)
            return cudaErrorInvalidConfiguration;
        kern<<<sms * nb, threads, smem, stream>>>(a);
        return cudaGetLastError();
    };
    const bool bf16 = c.in_dtype == TURNOPD_BF16;
    // rows that a CTA holds in registers, with up to 7 elements before the first
    const int64_t span = c.vocab + 7;
    const size_t esz = bf16 ? 2 : 4;
    const bool aligned = ((reinterpret_cast<uintptr_t>(c.zt) | reinterpret_cast<uintptr_t>(c.zs) | (uintptr_t)(c.ld * esz)) & 15u) == 0;
    if (span <= (int64_t)kShortPerThread * 512 && (!aligned || c.vocab <= short_max_vocab(c.K))) {
        // one warp a row where many rows hide its latency; a few rows of K above 128 finish sooner on four
        // (up to 200 rows of 1,024 ids, K = 256, bf16: 37 us, 27 streamed, now 27)
        const bool one_warp = span <= kShortPerThread * 32 && (c.K <= 128 || c.T > (int64_t)sms * 8);
        const int s4 = one_warp ? 0 : span <= kShortPerThread * 128 ? 1 : span <= kShortPerThread * 256 ? 2 : 3;
        static const Kern shorts[2][2][4] = {
            {{k_topk_short<false, 32, false>, k_topk_short<false, 128, false>, k_topk_short<false, 256, false>,
              k_topk_short<false, 512, false>},
             {k_topk_short<true, 32, false>, k_topk_short<true, 128, false>, k_topk_short<true, 256, false>,
              k_topk_short<true, 512, false>}},
            {{k_topk_short<false, 32, true>, k_topk_short<false, 128, true>, k_topk_short<false, 256, true>,
              k_topk_short<false, 512, true>},
             {k_topk_short<true, 32, true>, k_topk_short<true, 128, true>, k_topk_short<true, 256, true>,
              k_topk_short<true, 512, true>}}};
        const int sort = c.K >= kShortSortK;
        static const int threads[4] = {32, 128, 256, 512};
        if ((e = launch(shorts[sort][bf16][s4], 12 + sort * 8 + bf16 * 4 + s4, threads[s4], short_smem(c.K, threads[s4]))) != cudaSuccess)
            return e;
        launch_loss_sum(ws.row_wl, ws.nvalid, c.loss, c.status, stream);
        return cudaGetLastError();
    }
    // four selector warps above K = 96.  fp32 rows above 131,072 ids without a dense row keep two for
    // K = 289-448: their bound walks the row's buckets, which the streaming warps do faster with 72
    // registers than with 64 (us of a step of 2e8 logits, two and four: V = 151,936, K = 290 222 and
    // 238, 320 224 and 238, 384 233 and 247, 448 247 and 251; 128,256, K = 320 238 and 238).
    const bool walk = !bf16 && !c.grad && c.K > 288 && c.K <= 448 && c.vocab > 131072;
    const bool large = c.K > kTkLaneBoundMaxK && !walk;
    const DenseRow dn = !c.grad ? kNoDense
                        : !bf16 && c.vocab > 14336 && c.vocab <= 65536 ? kZerosByStream : kZerosBySelectors;
    const int ti = (bf16 ? 0 : 1) + (large ? 2 : 0);
    static const Kern kerns[4][3] = {
        {k_topk_rows<true, kTkSelSmall, kNoDense>, k_topk_rows<true, kTkSelSmall, kZerosBySelectors>, nullptr},
        {k_topk_rows<false, kTkSelSmall, kNoDense>, k_topk_rows<false, kTkSelSmall, kZerosBySelectors>,
         k_topk_rows<false, kTkSelSmall, kZerosByStream>},
        {k_topk_rows<true, kTkSelLarge, kNoDense>, k_topk_rows<true, kTkSelLarge, kZerosBySelectors>, nullptr},
        {k_topk_rows<false, kTkSelLarge, kNoDense>, k_topk_rows<false, kTkSelLarge, kZerosBySelectors>,
         k_topk_rows<false, kTkSelLarge, kZerosByStream>}};
    if ((e = launch(kerns[ti][dn], ti * 3 + dn, kTkStreamThreads + 32 * (large ? kTkSelLarge : kTkSelSmall),
                    topk_smem_bytes(c.vocab, c.K))) != cudaSuccess)
        return e;
    launch_loss_sum(ws.row_wl, ws.nvalid, c.loss, c.status, stream);
    return cudaGetLastError();
}

}  // namespace turnopd
