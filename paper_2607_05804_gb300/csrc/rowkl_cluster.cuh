// Held-row kernels for the per-token OPD loss (sm_103a): bf16 and fp32 logits, any
// vocabulary and row stride.
//
// The gradient needs both rows of a token twice (statistics, then p_s and z_s - z_t).  A
// CTA, or a cluster of CTAs where the rows are longer than one's shared memory holds (V =
// 151,936 bf16: 607 KB for the two, 8 CTAs; fp32: 16), therefore owns one row at a time:
// CTA c of CS holds vector slice c of both in shared memory, so HBM is read exactly once per
// row and the gradient written once (911,616 algorithmic bytes per row in bf16).
//
// Per CTA (persistent, one per SM, rows cid, cid + nclusters, ...):
//   * slices stream into a ring of ST stages with bulk asynchronous copies
//     (cp.async.bulk, completion on a "full" mbarrier, L2 evict-first); a stage is refilled
//     once every warp of the group that used it has arrived on its "empty" mbarrier;
//   * G groups of threads take the rows in turn: while one waits for its row's data or
//     records, the others compute;
//   * stats(k): per thread a max pass (packed bf16x2 max) and a sum pass
//     (packed f32x2 arithmetic): S = sum exp(z - m) for both models and
//     A = sum exp(z_s - m_s)((z_s - z_t) - d), d taken at the student's max.
//     The CTA's partial is pushed to every CTA of the cluster with st.async
//     into a record ring; completion lands on the receiver's mbarrier
//     (32 bytes per sender), so no cluster-wide barrier runs per row;
//   * the group's first warp merges the CS records by the same fixed lane tree, so all
//     CTAs use bit-identical LSE and KL (deterministic);
//   * grad(k) from the resident slice.
// Each thread reads its vectors of a row from shared memory three times: for the maxima,
// for the sums and for the gradient (3 exponentials per element in all).
// Clusters of 8 fill 120 of the 152 SMs; a helper grid of one 512-thread CTA per
// free SM takes the last share of the rows, each row read from HBM once (staged
// through a cp.async ring) and again from L2 (k_row_helper below).
// Waits are bounded: on timeout the kernel records TURNOPD_ERR_TIMEOUT, stops
// computing and runs its remaining barriers without waiting, so it terminates.

#pragma once

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"
#include "packed.cuh"
#include "ptx.cuh"
#include "row_math.cuh"

namespace turnopd {
namespace {

constexpr uint32_t kCopyChunk = 65536;       // bytes per bulk copy instruction
constexpr uint32_t kWaitLimit = 1u << 22;    // mbarrier polls before giving up

// Per-row constants the gradient pass needs (computed once per row): p |w| (full) or p |w l|
// (sampled) is 2^(z_s log2e + nlw) |sg| (|sgl|).
struct GradConst {
    float lse_s, lse_t, kl;
    float nlw;        // -LSE_s log2e + log2 |w| or log2 |w l|; row_scale's hi where it is used
    float sg;         // sign of w; row_scale's c
    float nd, ncp;    // -sg d, -sg cp; with row_scale -d, -c cp
    float nc;         // -sg (d + cp)
    float sgl;        // sign of -w l (sampled); row_scale's c
    float gy;         // sampled: g_y = w l (1 - p_y)
};

// t 2^((z - m) log2e) as 2^(z log2e + hi) c, |c| <= 1 with the sign of t.  hi is -m log2e rounded
// up, plus the power of two taken out of a t above 1; c holds t and what the rounding added.  A
// constant -LSE log2e + log2 |w| rounded to one float instead is off by up to half an ulp of a
// number as large as the logits, in every element of the row at once (2-norm error of the fp32
// gradient, packed 4 x 4096, V = 151,936: 0.9-1.1e-6, with the two parts 1.4-1.9e-7; 2,803 and
// 2,817 us).  |c| <= 1 keeps c ((z_s - z_t) - d) finite where the student alone is masked with the
// type's lowest value.
struct Scale {
    float hi, c;
};
__device__ __forceinline__ Scale row_scale(float m, float t)
{
    const float M = fmaxf(m, kLowestRef);
    int k = 0;
    const float f = fabsf(t) > 1.f ? frexpf(t, &k) : t;
    const float h0 = __fmul_rn(-M, kLog2e), kf = (float)k;
    float h = __fadd_rn(h0, kf);
    const float kb = __fsub_rn(h, h0);  // h + lo = -M log2e + k, exactly
    float lo = __fadd_rn(__fmaf_rn(-M, kLog2e, -h0), __fadd_rn(__fsub_rn(h0, __fsub_rn(h, kb)), __fsub_rn(kf, kb)));
    if (lo > 0.f) {
        const float up = __int_as_float(__float_as_int(h) + (h < 0.f ? -1 : 1));  // the next float
        lo -= __fsub_rn(up, h);
        h = up;
    }
    return Scale{h, f * (lo > -0x1p-12f ? fmaf(lo, kLn2, 1.f) : exp2f(lo))};
}

// What a lane that does not count reads as: bf16's lowest finite value.  It adds 0 to every
// sum, also where a thread or a vector holds nothing else (scale_of).
constexpr uint32_t kFillHi = 0xff7fu;            // the upper 16 bits; as bf16 and, shifted, as fp32

// One 16-byte vector of logits: N elements, NP pairs of them, and the running maximum of
// vectors (packed for bf16).
template <typename T> struct Elem;
template <> struct Elem<__nv_bfloat16> {
    static constexpr int N = 8, NP = 4, LOG = 3;
    static constexpr uint32_t kFillWord = kFillHi | kFillHi << 16;
    using Max = uint32_t;  // two candidates
    __device__ static Max max_empty() { return 0xff80ff80u; }  // (-inf, -inf)
    __device__ static Max max_of(const uint4 &v) { return hmax4(v); }
    __device__ static Max max2(Max a, Max b) { return hmax2u(a, b); }
    __device__ static float value(Max m) { return fmaxf(bf16lo(m), bf16hi(m)); }
    __device__ static bool has(Max m, float x) { return bf16lo(m) == x || bf16hi(m) == x; }
    __device__ static float2 pair(const uint4 &v, int j) { return unpack2(word(v, j)); }
    // v with lane i replaced by the fill
    __device__ static uint4 fill_lane(uint4 v, int i)
    {
        const uint32_t keep = (i & 1) ? 0x0000ffffu : 0xffff0000u;
        const uint32_t fill = kFillWord & ~keep;
        const int w = i >> 1;
        v.x = w == 0 ? (v.x & keep) | fill : v.x;
        v.y = w == 1 ? (v.y & keep) | fill : v.y;
        v.z = w == 2 ? (v.z & keep) | fill : v.z;
        v.w = w == 3 ? (v.w & keep) | fill : v.w;
        return v;
    }
    // v with its lanes outside [lo, hi) replaced by the fill (the lanes of a row's first
    // and last vectors that belong to other rows or to padding)
    __device__ static uint4 keep_lanes(uint4 v, int lo, int hi)
    {
        uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const bool in0 = 2 * j >= lo && 2 * j < hi, in1 = 2 * j + 1 >= lo && 2 * j + 1 < hi;
            w[j] = (in0 ? w[j] & 0x0000ffffu : kFillHi) | (in1 ? w[j] & 0xffff0000u : kFillHi << 16);
        }
        return make_uint4(w[0], w[1], w[2], w[3]);
    }
    // lanes [lo, hi) of the vector at p read one element at a time, the others the fill: the
    // vector that would pass the end of the logits
    __device__ static uint4 load_lanes(const __nv_bfloat16 *p, int lo, int hi)
    {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t e0 = 2 * j >= lo && 2 * j < hi ? __bfloat16_as_ushort(p[2 * j]) : kFillHi;
            const uint32_t e1 = 2 * j + 1 >= lo && 2 * j + 1 < hi ? __bfloat16_as_ushort(p[2 * j + 1]) : kFillHi;
            w[j] = e0 | (e1 << 16);
        }
        return make_uint4(w[0], w[1], w[2], w[3]);
    }
    // the element at shared address `a` replaced by the fill; returns it
    __device__ static float swap_shared(uint32_t a)
    {
        uint32_t old;
        asm volatile("ld.shared.u16 %0, [%1];\n\tst.shared.u16 [%1], %2;\n\t" : "=r"(old) : "r"(a), "r"(kFillHi) : "memory");
        return __uint_as_float(old << 16);
    }
};
template <> struct Elem<float> {
    static constexpr int N = 4, NP = 2, LOG = 2;
    static constexpr uint32_t kFillWord = kFillHi << 16;
    using Max = float;
    __device__ static Max max_empty() { return -INFINITY; }
    __device__ static Max max_of(const uint4 &v)
    {
        return fmaxf(fmaxf(__uint_as_float(v.x), __uint_as_float(v.y)), fmaxf(__uint_as_float(v.z), __uint_as_float(v.w)));
    }
    __device__ static Max max2(Max a, Max b) { return fmaxf(a, b); }
    __device__ static float value(Max m) { return m; }
    __device__ static bool has(Max m, float x) { return m == x; }
    __device__ static float2 pair(const uint4 &v, int j)
    {
        return j == 0 ? make_float2(__uint_as_float(v.x), __uint_as_float(v.y))
                      : make_float2(__uint_as_float(v.z), __uint_as_float(v.w));
    }
    __device__ static uint4 fill_lane(uint4 v, int i)
    {
        v.x = i == 0 ? kFillWord : v.x;
        v.y = i == 1 ? kFillWord : v.y;
        v.z = i == 2 ? kFillWord : v.z;
        v.w = i == 3 ? kFillWord : v.w;
        return v;
    }
    __device__ static uint4 keep_lanes(uint4 v, int lo, int hi)
    {
        v.x = lo <= 0 && hi > 0 ? v.x : kFillWord;
        v.y = lo <= 1 && hi > 1 ? v.y : kFillWord;
        v.z = lo <= 2 && hi > 2 ? v.z : kFillWord;
        v.w = lo <= 3 && hi > 3 ? v.w : kFillWord;
        return v;
    }
    __device__ static uint4 load_lanes(const float *p, int lo, int hi)
    {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            w[j] = j >= lo && j < hi ? __float_as_uint(p[j]) : kFillWord;
        return make_uint4(w[0], w[1], w[2], w[3]);
    }
    __device__ static float swap_shared(uint32_t a)
    {
        uint32_t old;
        asm volatile("ld.shared.u32 %0, [%1];\n\tst.shared.u32 [%1], %2;\n\t" : "=r"(old) : "r"(a), "r"(kFillWord) : "memory");
        return __uint_as_float(old);
    }
};

// Full-vocabulary gradient of a pair from p |w| (pw) and x = z_s - z_t: w p (x - d - cp), d and cp
// subtracted one after the other (D) or as one constant; SC: the constants are row_scale's.
template <bool D, bool SC>
__device__ __forceinline__ float2 full_grad(float2 pw, float2 x, float2 SG, float2 ND, float2 NCP, float2 NC)
{
    if (SC)
        return fmul2(pw, ffma2(fadd2(x, ND), SG, NCP));
    return D ? fmul2(pw, fadd2(ffma2(x, SG, ND), NCP)) : fmul2(pw, ffma2(x, SG, NC));
}

// One vector of the gradient, g[NP] pairs, stored whole: vector q of the row at `off`.
template <typename T, bool G32>
__device__ __forceinline__ void store_grad(void *grad, size_t off, int q, const float2 *g)
{
    constexpr int N = Elem<T>::N, NP = Elem<T>::NP;
    if (G32) {
        float4 *dst = reinterpret_cast<float4 *>(static_cast<float *>(grad) + off + (size_t)q * N);
        __stcs(dst, make_float4(g[0].x, g[0].y, g[1].x, g[1].y));
        if (NP == 4)
            __stcs(dst + 1, make_float4(g[NP - 2].x, g[NP - 2].y, g[NP - 1].x, g[NP - 1].y));
    } else if (NP == 4) {
        uint4 o;
        o.x = pack_bf16x2(g[0].x, g[0].y);
        o.y = pack_bf16x2(g[1].x, g[1].y);
        o.z = pack_bf16x2(g[NP - 2].x, g[NP - 2].y);
        o.w = pack_bf16x2(g[NP - 1].x, g[NP - 1].y);
        __stcs(reinterpret_cast<uint4 *>(static_cast<__nv_bfloat16 *>(grad) + off + (size_t)q * N), o);
    } else {
        uint2 o;
        o.x = pack_bf16x2(g[0].x, g[0].y);
        o.y = pack_bf16x2(g[1].x, g[1].y);
        __stcs(reinterpret_cast<uint2 *>(static_cast<__nv_bfloat16 *>(grad) + off + (size_t)q * N), o);
    }
}

// Columns [lo, hi) of one vector of the gradient, one at a time.
template <typename T, bool G32>
__device__ __forceinline__ void store_grad_lanes(void *grad, size_t e, const float2 *g, int lo, int hi)
{
#pragma unroll
    for (int i = 0; i < Elem<T>::N; ++i)
        if (i >= lo && i < hi) {
            const float x = i & 1 ? g[i / 2].y : g[i / 2].x;
            if (G32)
                static_cast<float *>(grad)[e + i] = x;
            else
                static_cast<__nv_bfloat16 *>(grad)[e + i] = __float2bfloat16_rn(x);
        }
}

// How rows lie in the 16-byte grid: whole vectors, a partial last vector alone (the stride is
// a multiple of a vector's N elements, the vocabulary is not), or any stride.
enum RowForm { kWhole = 0, kTail = 1, kAny = 2 };

// Rows that are not whole (TL > kWhole): a row starts `head` elements into a 16-byte vector
// and ends `tail` elements into one (tail 0: at its end; head 0 in kTail).  Its vectors are
// those of the 16-byte grid that hold any of its columns; the first and the last may be
// partial.  (Rows of a stride that is no multiple of 8 took the portable kernel's 2-byte loads
// before: dense 4 x 1024 tokens, V = 50,001, bf16, step 1,075 us, now 230; 133 is its traffic
// at the copy bandwidth.  kTail apart from kAny: V = 33,001 of stride 33,008 641 -> 606 us.)
struct Ragged {
    int head, nvec, tail;
};
template <typename T, int TL> __device__ __forceinline__ Ragged ragged(int row, int64_t ld, int64_t vocab)
{
    constexpr int N = Elem<T>::N;
    Ragged g;
    g.head = TL == kAny ? ((row & (N - 1)) * (int)(ld & (N - 1))) & (N - 1) : 0;
    g.nvec = (int)((g.head + vocab + N - 1) / N);
    g.tail = (int)((g.head + vocab) & (N - 1));
    return g;
}

// The clusters' share of nvalid rows: the host's ratio, with a helper grid of few rows a
// CTA rounded down to whole turns (a helper CTA takes as long for a row as a cluster for
// eight, so a last turn of a few CTAs holds up a small batch).
__device__ __forceinline__ int split_rows(const RowIn &p, int nvalid)
{
    if (!p.split_den)
        return nvalid;
    const int h = nvalid - (int)((int64_t)nvalid * p.split_num / p.split_den);
    return nvalid - (h >= p.split_ctas && h < 8 * p.split_ctas ? h - h % p.split_ctas : h);
}

// G groups of NT threads per CTA take the rows of the cluster in turn (row k to group
// k % G), each thread VPT vectors of each model, from a ring of ST stages.  Record slots:
// 2G, so a slot is reused by the same group two rows later, after that group has read it
// (a peer can run at most G rows ahead of the slowest CTA in sending records).  SM: a
// sampled-token call, where every listed row carries its y in [0, V); otherwise the full
// vocabulary (y = -1).  TL: a RowForm.
template <typename T, int CS, int NT, int VPT, int G, int ST, bool G32, bool SM, int TL>
__global__ void __launch_bounds__(G * NT, 1) k_row_cluster(RowIn p, int slice_vec, int nvec)
{
    using E = Elem<T>;
    constexpr int N = E::N, NP = E::NP;
    constexpr int kStages = ST;
    constexpr int kSlots = 2 * G;
    static_assert(G <= 15 || NT == 32, "one named barrier per group");
    // Reference difference d (A = sum e ((z_s - z_t) - d), d at the student's
    // max): it keeps gradients at a dominant token accurate to fp32 relative
    // precision.  bf16 rows of an aligned stride with a bf16 gradient leave it out: the error of
    // E_p[z_s - z_t] is then ~1e-6 absolute, under a bf16 ulp of nearly all of those
    // gradients.  Rows of any other stride keep it whatever the types, as do fp32 logits.
    // (Relative error of g at a token 10, 12, 14 and 16 above the rest of its row, V = 50,001,
    // bf16: without it 0.3, 2, 12 and 18 %, with it the rounding's 0.4 % at each.)
    constexpr bool kUseD = G32 || N == 4 || (TL == kAny && !SM);
    constexpr bool kGradD = G32 || TL == kAny;  // the gradient subtracts d and cp one after the other
    constexpr bool kScale = kGradD && N == 4;    // the row's constant in two parts (row_scale)
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int s_dead;
    constexpr int NWG = NT / 32;  // warps per group
    const int tid = threadIdx.x, lane = tid & 31;
    const int group = tid / NT, gtid = tid % NT, gwarp = gtid >> 5;
    const uint32_t rank = cluster_ctarank();
    const int cid = (int)cluster_id(), ncl = (int)cluster_count();
    const uint32_t slice_bytes = (uint32_t)slice_vec * 16u;
    const uint32_t stage_bytes = 2u * slice_bytes;
    const int v0 = (int)rank * slice_vec;  // first vector of my slice
    const int my_vec = max(0, min(slice_vec, nvec - v0));
    // TL: in kAny the slice's vectors and the partial ones among them vary from row to row.
    // A partial vector's other lanes read as the fill in the
    // statistics (set in shared memory by the thread that reads the vector) and are
    // never written: the gradient loop stores whole vectors, that thread the partial
    // one's columns.  Without TL all of this compiles away.
    struct Slice {
        int my_vec, head0, g0, gvec, tailq, tail;  // head0: of the row (every slice)
        bool head;                                  // vector 0 is partial
    };
    auto slice_of = [&](int row) {
        Slice g{my_vec, 0, 0, my_vec, -1, 0, false};
        if (TL == kTail) {
            g.tail = (int)(p.vocab & (N - 1));
            g.tailq = my_vec > 0 && v0 + my_vec == nvec ? my_vec - 1 : -1;
            g.gvec = g.tailq >= 0 ? my_vec - 1 : my_vec;
        } else if (TL == kAny) {
            const Ragged r = ragged<T, TL>(row, p.ld, p.vocab);
            g.my_vec = max(0, min(slice_vec, r.nvec - v0));
            g.head0 = r.head;
            g.head = v0 == 0 && r.head > 0;
            g.tail = r.tail;
            g.tailq = r.tail && g.my_vec > 0 && v0 + g.my_vec == r.nvec ? g.my_vec - 1 : -1;
            g.g0 = g.head ? 1 : 0;
            g.gvec = g.tailq >= 0 ? g.my_vec - 1 : g.my_vec;
        }
        return g;
    };
    // the slice's last vector passes the end of the logits (kTail: only the last row's can)
    const int last_row = TL == kTail ? (int)((p.elems - p.vocab) / p.ld) : 0;
    auto cut = [&](const Slice &g, int row) {
        if (TL == kTail)
            return g.tailq >= 0 && row == last_row;
        return TL && g.tailq >= 0 && (int64_t)row * p.ld - g.head0 + (int64_t)(v0 + g.my_vec) * N > p.elems;
    };

    unsigned char *stage = smem;
    float *rec = reinterpret_cast<float *>(smem + kStages * stage_bytes);  // [kSlots][CS][8]
    int4 *meta = reinterpret_cast<int4 *>(rec + kSlots * CS * 8);          // [kStages]
    uint64_t *full = reinterpret_cast<uint64_t *>(meta + kStages);         // [kStages]
    uint64_t *empty = full + kStages;                                      // [kStages]
    uint64_t *recv = empty + kStages;                                      // [kSlots]
    float *red = reinterpret_cast<float *>(recv + kSlots);                 // [G][NWG][8]
    int *srow = reinterpret_cast<int *>(red + G * NWG * 8);            // [kStages] row in stage
    int *yown = srow + (kStages + 3) / 4 * 4;                                            // [kStages] thread reading y, or -1
    float *rcs = reinterpret_cast<float *>(yown + (kStages + 3) / 4 * 4);                 // [G][16] row constants; [15]: z_s[y]

    if (tid == 0) {
        s_dead = 0;
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], NWG);
            srow[s] = -1;
        }
        if (CS > 1)
            for (int s = 0; s < kSlots; ++s)
                mbar_init(&recv[s], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (CS > 1)
            for (int s = 0; s < kSlots; ++s)
                mbar_arrive_expect_tx(&recv[s], CS * 32u);  // first record of each slot
    }
    __syncthreads();
    if (CS > 1)
        cluster_sync();  // peers' barriers are initialised before any record is sent
    // Every CTA of this grid is resident: a helper grid launched after this one may
    // start now, on the SMs the clusters left free.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    const int nv_all = *p.nvalid;
    const int nvalid = split_rows(p, nv_all);
    const int n = nvalid > cid ? (nvalid - cid + ncl - 1) / ncl : 0;  // same for the whole cluster
    if (n == 0)
        return;

    const T *zs = static_cast<const T *>(p.zs);
    const T *zt = static_cast<const T *>(p.zt);

    auto dead = [&]() { return *(volatile int *)&s_dead != 0; };
    auto wait_bar = [&](uint64_t *bar, uint32_t parity, bool cluster_scope) {
        if (dead())
            return;
        for (uint32_t it = 0; it < kWaitLimit; ++it)
            if (cluster_scope ? mbar_try_wait_cluster(bar, parity) : mbar_try_wait(bar, parity))
                return;
        s_dead = 1;
        set_status(p.status, TURNOPD_ERR_TIMEOUT);
    };
    auto group_sync = [&]() {
        if (NT == 32)
            __syncwarp();
        else
            asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "r"(NT) : "memory");
    };

    // Data of row k: wait until the stage has been armed for row k, then for
    // its phase.  (A parity wait alone would also accept the phase of the
    // stage's previous row, k - kStages, when a group reaches row k early.)
    auto wait_full = [&](int k) {
        const int s = k % kStages;
        if (dead())
            return;
        uint32_t it = 0;
        while (*(volatile int *)&srow[s] != k && ++it < kWaitLimit) {
        }
        if (it >= kWaitLimit) {
            s_dead = 1;
            set_status(p.status, TURNOPD_ERR_TIMEOUT);
            return;
        }
        wait_bar(&full[s], (uint32_t)((k / kStages) & 1), false);
    };

    // stream row k of this cluster into stage k % kStages (after the stage's
    // previous row is done with it)
    auto issue = [&](int k, int4 m) {
        const int s = k % kStages;
        const Slice g = slice_of(m.y);
        meta[s] = m;
        if (SM) {  // the thread that will read y's vector (sampled-token rows; see stats)
            const int q = m.z >= 0 ? (m.z + g.head0) / N - v0 : -1;
            yown[s] = q >= 0 && q < g.my_vec ? q % NT : -1;
        }
        *(volatile int *)&srow[s] = k;
        const uint32_t my_bytes = (uint32_t)(cut(g, m.y) ? g.my_vec - 1 : g.my_vec) * 16u;
        const size_t off = (size_t)m.y * (size_t)p.ld - (size_t)g.head0 + (size_t)v0 * N;
        const char *gs = reinterpret_cast<const char *>(zs + off);
        const char *gt = reinterpret_cast<const char *>(zt + off);
        unsigned char *ds = stage + s * stage_bytes;
        const uint64_t pol = evict_first_policy();
        mbar_arrive_expect_tx(&full[s], 2u * my_bytes);
        for (uint32_t o = 0; o < my_bytes; o += kCopyChunk) {
            const uint32_t sz = min(kCopyChunk, my_bytes - o);
            bulk_g2s(ds + o, gs + o, sz, &full[s], pol);
            bulk_g2s(ds + slice_bytes + o, gt + o, sz, &full[s], pol);
        }
    };

    // row k's constants for the gradient pass from its merged statistics and its sampled
    // token's logits (one thread of the group)
    auto row_constants = [&](int k, Student A, const Teacher &B, float ys, float yt) {
        float *bc = rcs + group * 16;
        float omp = 0.f;  // 1 - p_y (sampled)
        if (SM)
            omp = add_sampled_term(A, ys);
        const RowConst rc = row_const(A, B);
        float e = rc.kl;
        if (SM)
            e = (ys - yt) - rc.dl;
        // gradient constants of the row (see grad)
        const float wi = __int_as_float(meta[k % kStages].w), wl = wi * e;
        const float sg = wi < 0.f ? -1.f : 1.f;
        bc[0] = rc.lse_s, bc[1] = rc.lse_t, bc[2] = rc.kl, bc[3] = e;
        if (kScale) {
            if (p.grad) {
                const Scale q = row_scale(A.m, (SM ? -wl : wi) / A.s);
                bc[4] = q.hi;
                bc[5] = bc[9] = q.c;
                bc[6] = -rc.d;
                bc[7] = -q.c * rc.cp;
            }
        } else {
            bc[4] = -rc.lse_s * kLog2e + log2f(fabsf(SM ? wl : wi));  // nlw
            bc[5] = sg;
            bc[6] = -sg * rc.d;
            bc[7] = -sg * rc.cp;
            bc[8] = -sg * (rc.d + rc.cp);     // one rounding of d + cp
            bc[9] = wl > 0.f ? -1.f : 1.f;    // sampled: sign of -w l
        }
        bc[10] = wl * omp;                 // sampled: g_y = w l (1 - p_y)
    };

    // statistics of row k: this CTA's record into slot k % kSlots of every CTA (a cluster
    // of one: the row's constants at once)
    auto stats = [&](int k) {
        const int s = k % kStages;
        const uint4 *vs = reinterpret_cast<const uint4 *>(stage + s * stage_bytes);
        const uint4 *vt = reinterpret_cast<const uint4 *>(stage + s * stage_bytes + slice_bytes);
        const Slice g = slice_of(meta[s].y);
        const int my_vec = g.my_vec;
        if (TL && ((g.tailq >= 0 && g.tailq % NT == gtid) || (g.head && gtid == 0))) {
            // partial vectors: lanes of other rows and padding out of both models' statistics
            uint4 *ws = reinterpret_cast<uint4 *>(stage + s * stage_bytes);
            uint4 *wt = reinterpret_cast<uint4 *>(stage + s * stage_bytes + slice_bytes);
            if (g.tailq >= 0 && g.tailq % NT == gtid) {
                if (cut(g, meta[s].y)) {
                    const size_t e = (size_t)meta[s].y * (size_t)p.ld - (size_t)g.head0 + (size_t)(v0 + g.tailq) * N;
                    ws[g.tailq] = E::load_lanes(zs + e, 0, g.tail);
                    wt[g.tailq] = E::load_lanes(zt + e, 0, g.tail);
                } else {
                    ws[g.tailq] = E::keep_lanes(ws[g.tailq], 0, g.tail);
                    wt[g.tailq] = E::keep_lanes(wt[g.tailq], 0, g.tail);
                }
            }
            if (g.head && gtid == 0) {
                ws[0] = E::keep_lanes(ws[0], g.head0, N);
                wt[0] = E::keep_lanes(wt[0], g.head0, N);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        // A sampled-token row leaves y out of the student statistics (add_sampled_term
        // brings its term back at the merge): the thread that reads y's vector in both
        // passes below (named at issue) keeps z_s[y] for the record and puts the fill
        // in its place, which adds 0.  (The gradient
        // pass replaces g_y; the proxy fence orders the store before the stage's next
        // bulk copy.)
        if (SM && yown[s] == gtid) {
            rcs[group * 16 + 15] = E::swap_shared(smem_u32(stage + s * stage_bytes) +
                                                  (uint32_t)sizeof(T) * (uint32_t)(meta[s].z + g.head0 - v0 * N));
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        // max pass (packed for bf16): running maxima, plus each vector's student
        // maximum so the argmax vector is found after the loop
        typename E::Max smax = E::max_empty(), tmax = E::max_empty();
        typename E::Max vmax[VPT];
#pragma unroll
        for (int u = 0; u < VPT; ++u) {
            const int q = gtid + u * NT;
            vmax[u] = E::max_empty();
            if (q < my_vec) {
                const uint4 a = vs[q], b = vt[q];
                vmax[u] = E::max_of(a);
                smax = E::max2(smax, vmax[u]);
                tmax = E::max2(tmax, E::max_of(b));
            }
        }
        const float ms = E::value(smax), mt = E::value(tmax);
        // reference difference at the first element equal to the student max (see kUseD)
        float xd = 0.f;
        if (kUseD && ms != -INFINITY) {
            int bq = gtid;
#pragma unroll
            for (int u = VPT - 1; u >= 0; --u)
                if (E::has(vmax[u], ms))
                    bq = gtid + u * NT;
            const uint4 a = vs[bq], b = vt[bq];
            bool found = false;
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                const float2 x = E::pair(a, j), y = E::pair(b, j);
                if (!found && x.x == ms) {
                    xd = x.x - y.x;
                    found = true;
                }
                if (!found && x.y == ms) {
                    xd = x.y - y.y;
                    found = true;
                }
            }
        }
        // sum pass (packed pairs)
        const float2 L2 = splat(kLog2e), NS = splat(scale_of(ms)), NTT = splat(scale_of(mt));
        const float2 D = splat(xd);
        float2 S2 = make_float2(0.f, 0.f), A2 = S2, T2 = S2;
#pragma unroll
        for (int u = 0; u < VPT; ++u) {
            const int q = gtid + u * NT;
            if (q < my_vec) {
                const uint4 a = vs[q], b = vt[q];
#pragma unroll
                for (int j = 0; j < NP; ++j) {
                    const float2 a2 = E::pair(a, j), b2 = E::pair(b, j);
                    const float2 es = ex2x2(ffma2(a2, L2, NS));
                    S2 = fadd2(S2, es);
                    A2 = ffma2(es, kUseD ? fsub2(fsub2(a2, b2), D) : fsub2(a2, b2), A2);
                    T2 = fadd2(T2, ex2x2(ffma2(b2, L2, NTT)));
                }
            }
        }
        Student S = ms == -INFINITY ? student_empty() : Student{ms, S2.x + S2.y, A2.x + A2.y, xd};
        Teacher U = mt == -INFINITY ? teacher_empty() : Teacher{mt, T2.x + T2.y};
        lane_merge<32, kUseD>(S, U);
        float *rg = red + group * NWG * 8;
        if (lane == 0) {
            float *rw = rg + gwarp * 8;
            rw[0] = S.m, rw[1] = S.s, rw[2] = S.a, rw[3] = S.d, rw[4] = U.m, rw[5] = U.s;
        }
        group_sync();
        if (gwarp == 0) {
            Student A = student_empty();
            Teacher B = teacher_empty();
            if (lane < NWG) {
                const float *r = rg + lane * 8;
                A = Student{r[0], r[1], r[2], r[3]};
                B = Teacher{r[4], r[5]};
            }
            lane_merge<NWG, kUseD>(A, B);
            if (CS == 1) {  // the CTA's partial is the row's
                if (lane == 0)
                    row_constants(k, A, B, SM ? rcs[group * 16 + 15] : 0.f,
                                  SM ? to_float(reinterpret_cast<const T *>(vt)[meta[s].z + g.head0]) : 0.f);
                return;
            }
            A.m = __shfl_sync(0xffffffffu, A.m, 0);
            A.s = __shfl_sync(0xffffffffu, A.s, 0);
            A.a = __shfl_sync(0xffffffffu, A.a, 0);
            A.d = __shfl_sync(0xffffffffu, A.d, 0);
            B.m = __shfl_sync(0xffffffffu, B.m, 0);
            B.s = __shfl_sync(0xffffffffu, B.s, 0);
            if (lane < CS) {
                float ys = 0.f, yt = 0.f;  // sampled-token logits, from the CTA holding y
                const int y = meta[s].z, yh = y + g.head0;
                if (y >= 0 && yh / N >= v0 && yh / N < v0 + my_vec) {
                    const int e = yh - v0 * N;
                    ys = SM ? rcs[group * 16 + 15] : to_float(reinterpret_cast<const T *>(vs)[e]);
                    yt = to_float(reinterpret_cast<const T *>(vt)[e]);
                }
                const int slot = k % kSlots;
                const uint32_t ra = mapa(smem_u32(rec + (slot * CS + (int)rank) * 8), (uint32_t)lane);
                const uint32_t rbar = mapa(smem_u32(&recv[slot]), (uint32_t)lane);
                st_async16(ra, rbar, make_float4(A.m, A.s, A.a, A.d));
                st_async16(ra + 16, rbar, make_float4(B.m, B.s, ys, yt));
            }
        }
    };

    // row constants of row k from the CS records, computed by the group's
    // first warp (fixed merge order: identical in every CTA) and shared with
    // the group through shared memory
    auto combine = [&](int k, float &ell) {
        const int slot = k % kSlots;
        float *bc = rcs + group * 16;
        if (CS > 1 && gwarp == 0) {
            wait_bar(&recv[slot], (uint32_t)((k / kSlots) & 1), true);
            const float *r = rec + slot * CS * 8;
            Student A = student_empty();
            Teacher B = teacher_empty();
            if (lane < CS) {
                const float4 x = *reinterpret_cast<const float4 *>(r + lane * 8);
                const float4 y = *reinterpret_cast<const float4 *>(r + lane * 8 + 4);
                A = Student{x.x, x.y, x.z, x.w};
                B = Teacher{y.x, y.y};
            }
            lane_merge<CS, kUseD>(A, B);
            if (lane == 0) {
                const int y = meta[k % kStages].z;
                const int yh = TL ? y + ragged<T, TL>(meta[k % kStages].y, p.ld, p.vocab).head : y;
                const int owner = SM ? (yh / N) / slice_vec : 0;
                row_constants(k, A, B, r[owner * 8 + 6], r[owner * 8 + 7]);
                mbar_arrive_expect_tx(&recv[slot], CS * 32u);  // re-arm for row k + kSlots
            }
        }
        group_sync();
        GradConst gc;
        gc.lse_s = bc[0], gc.lse_t = bc[1], gc.kl = bc[2];
        ell = bc[3];
        gc.nlw = bc[4], gc.sg = bc[5], gc.nd = bc[6], gc.ncp = bc[7], gc.nc = bc[8], gc.sgl = bc[9];
        gc.gy = bc[10];
        return gc;
    };

    auto grad = [&](int k, const GradConst &gc) {
        if (!p.grad)
            return;
        const int s = k % kStages;
        const int4 m = meta[s];
        const uint4 *vs = reinterpret_cast<const uint4 *>(stage + s * stage_bytes);
        const uint4 *vt = reinterpret_cast<const uint4 *>(stage + s * stage_bytes + slice_bytes);
        const int y = m.z;
        const float gy = gc.gy;
        const Slice sl = slice_of(m.y);
        const int gvec = sl.gvec;
        const size_t row_off = (size_t)m.y * (size_t)p.ld - (size_t)sl.head0 + (size_t)v0 * N;
        // the sign of w (and row_scale's c) enters through an fma by (sg, sg), which is exact on
        // z_s - z_t for a sign alone
        const float2 L2 = splat(kLog2e), NLW = splat(gc.nlw);
        const float2 SG = splat(gc.sg), ND = splat(gc.nd), NCP = splat(gc.ncp), NC = splat(gc.nc);
        const float2 SGL = splat(gc.sgl);
#pragma unroll
        for (int u = 0; u < VPT; ++u) {
            const int q = gtid + u * NT;
            if (q < gvec && (TL != kAny || q >= sl.g0)) {
                float2 g[NP];
                // y < 0 exactly when !SM; the bf16 logits' fp32-gradient instantiations keep the
                // run-time test, which compiles to a loop 5 % faster there (and 2.4 % slower for
                // bf16 gradients)
                if (G32 && N == 8 ? y < 0 : !SM) {  // full vocabulary: g = w p ((z_s - z_t) - d - cp)
                    const uint4 a = vs[q], b = vt[q];
#pragma unroll
                    for (int j = 0; j < NP; ++j) {
                        const float2 a2 = E::pair(a, j), b2 = E::pair(b, j);
                        const float2 pw = ex2x2(ffma2(a2, L2, NLW));
                        const float2 x = fsub2(a2, b2);
                        g[j] = full_grad<kGradD, kScale>(pw, x, SG, ND, NCP, NC);
                    }
                } else {  // sampled token: g = -w l p (g_y is written after the loop)
                    const uint4 a = vs[q];
#pragma unroll
                    for (int j = 0; j < NP; ++j)
                        g[j] = fmul2(ex2x2(ffma2(E::pair(a, j), L2, NLW)), SGL);
                }
                store_grad<T, G32>(p.grad, row_off, q, g);
            }
        }
        // a partial vector, column by column (the loop's formulas)
        auto store_lanes = [&](int q, int lo, int hi) {
            const uint4 a = vs[q], b = vt[q];
            float2 g[NP];
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                const float2 a2 = E::pair(a, j), b2 = E::pair(b, j);
                const float2 pw = ex2x2(ffma2(a2, L2, NLW)), x = fsub2(a2, b2);
                g[j] = SM ? fmul2(pw, SGL)
                          : full_grad<kGradD, kScale>(pw, x, SG, ND, NCP, NC);
            }
            store_grad_lanes<T, G32>(p.grad, row_off + (size_t)q * N, g, lo, hi);
        };
        if (TL && sl.tailq > 0 && sl.tailq % NT == gtid)
            store_lanes(sl.tailq, 0, sl.tail);
        if (TL && gtid == 0 && (sl.head || sl.tailq == 0))
            store_lanes(0, sl.head ? sl.head0 : 0, sl.tailq == 0 ? sl.tail : N);
        // sampled token: g_y = w l (1 - p_y), over the value the vector store wrote
        // (same thread, so the later store wins)
        if (SM && yown[s] == gtid) {
            const size_t yo = (size_t)m.y * (size_t)p.ld + (size_t)y;
            if (G32)
                static_cast<float *>(p.grad)[yo] = gy;
            else
                static_cast<__nv_bfloat16 *>(p.grad)[yo] = __float2bfloat16_rn(gy);
        }
    };

    // The groups take rows in turn: while one waits for its row's records or
    // data, the others compute.
    if (kStages <= 5) {  // (in parallel these few cost the steady state 0.3 to 3 %)
        if (tid == 0)
            for (int k = 0; k < kStages && k < n; ++k)
                issue(k, p.rows[cid + k * ncl]);
    } else if (tid < kStages && tid < n) {
        issue(tid, p.rows[cid + tid * ncl]);
    }
    for (int k = group; k < n; k += G) {
        int4 ahead = make_int4(0, 0, -1, 0);
        if (gtid == 0 && k + kStages < n)
            ahead = p.rows[cid + (k + kStages) * ncl];  // used at the end of the iteration
        wait_full(k);
        stats(k);
        float ell;
        const GradConst gc = combine(k, ell);
        if (rank == 0 && gtid == 0) {
            const int4 m = meta[k % kStages];
            if (!isfinite(gc.lse_s) || !isfinite(gc.lse_t) || !isfinite(ell))
                set_status(p.status, TURNOPD_ERR_NONFINITE);
            p.token_loss[m.x] = ell;
            p.row_wl[cid + k * ncl] = (double)__int_as_float(m.w) * (double)ell;
        }
        if (!dead())
            grad(k, gc);
        __syncwarp();
        if (lane == 0)
            mbar_arrive(&empty[k % kStages]);
        if (gtid == 0 && k + kStages < n) {
            wait_bar(&empty[k % kStages], (uint32_t)((k / kStages) & 1), false);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            issue(k + kStages, ahead);
        }
    }

    // after a timeout, let this CTA's own copies land before it exits
    if (tid == 0 && dead()) {
        for (int k = max(0, n - kStages); k < n; ++k)
            for (uint32_t it = 0; it < kWaitLimit; ++it)
                if (mbar_try_wait(&full[k % kStages], (uint32_t)((k / kStages) & 1)))
                    break;
    }
    if (CS > 1)
        cluster_sync();  // no CTA leaves while a peer may still address its shared memory
}

// Helper for the SMs the clusters leave free (15 eight-CTA clusters cover 120 of
// 152): one CTA per row at a time, rows j0 + blockIdx.x, j0 + blockIdx.x +
// gridDim.x, ... of the row list, j0 = the cluster kernel's share.  The
// statistics pass streams both rows from HBM (beside the clusters through a cp.async
// ring, AS) with a running maximum per thread (one rescale per batch of kHelpU
// vectors when the maximum moves); the gradient
// pass reads them again from L2, where the pass before left them (the clusters'
// own copies are evict-first).  A bf16 or fp32 gradient or none.
// Like the cluster kernel, the fp32 gradient also keeps A relative to the
// reference difference d at the thread's running student argmax (re-referenced,
// A <- (A + S (d - d')) f, when the maximum moves).  Launched as a dependent
// of the cluster grid (it starts once every cluster is resident) and completes
// only after it, so stream order after it covers both grids.
constexpr int kHelpThreads = 512;
constexpr int kHelpU = 4;  // vectors of each model per thread and batch
// AS: the statistics pass's batches land in a kHelpStages-deep ring in shared memory by
// cp.async, kHelpStages - 1 batches ahead (each thread copies and reads only its own
// slots): twice the loads in flight of the register path, with no registers held by
// them.  The helper beside the clusters takes it (packed 8 x 4096, V = 151,936: 2.776 ->
// 2.743 ms per loss call with the split rate raised to 0.7).  The helper alone, which
// takes rows that no cluster holds, has the register path, from when short rows took it
// (V = 16,384: 0.405 against 0.433 ms); at its present lengths the ring would be faster
// with a gradient (us at 6e8 bf16 logits, registers and ring: V = 400,000 908 and 874,
// sampled 820 and 744, forward 427 and 389; fp32 forward at 200,001 382 and 416).
constexpr int kHelpStages = 3;
constexpr size_t kHelperSmem = (size_t)kHelpStages * 2 * kHelpU * kHelpThreads * 16;  // AS

template <typename T, bool G32, bool SM, int TL, bool AS>
__global__ void __launch_bounds__(kHelpThreads, 1) k_row_helper(RowIn p)
{
    constexpr int NW = kHelpThreads / 32;
    using E = Elem<T>;
    constexpr int N = E::N, NP = E::NP;
    constexpr uint32_t kFill = E::kFillWord;
    constexpr bool kUseD = G32 || N == 4 || (TL == kAny && !SM), kGradD = G32 || TL == kAny, kScale = kGradD && N == 4;  // as in the cluster kernel
    __shared__ float red[NW][8];
    __shared__ float bc[8];
    extern __shared__ uint4 hring[];  // [kHelpStages][2][kHelpU][kHelpThreads] (AS)
    // the loss sum after this grid may take the first SM it frees (it waits for the grid)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nvalid = *p.nvalid;
    const int j0 = p.split_den ? split_rows(p, nvalid) : 0;
    const T *zs = static_cast<const T *>(p.zs);
    const T *zt = static_cast<const T *>(p.zt);
    const float2 L2 = splat(kLog2e);
    for (int j = j0 + (int)blockIdx.x; j < nvalid; j += gridDim.x) {
        const int4 m = p.rows[j];
        const size_t off = (size_t)m.y * (size_t)p.ld;
        // TL: a partial first or last vector's other lanes read as the fill
        // and are never written; the gradient loop stores vectors [g0, nfull)
        const Ragged rg = TL ? ragged<T, TL>(m.y, p.ld, p.vocab) : Ragged{0, (int)(p.vocab / N), 0};
        const int head = rg.head, nvec = rg.nvec, tail = rg.tail;
        const int g0 = TL && head ? 1 : 0, nfull = TL && tail ? nvec - 1 : nvec;
        const size_t voff = off - (size_t)head;          // the row's first vector
        const bool cut = TL && (int64_t)voff + (int64_t)nvec * N > p.elems;  // the last passes the end
        auto lanes_lo = [&](int q) { return q == 0 ? head : 0; };
        auto lanes_hi = [&](int q) { return q == nvec - 1 && tail ? tail : N; };
        const uint4 *vs = reinterpret_cast<const uint4 *>(zs + voff);
        const uint4 *vt = reinterpret_cast<const uint4 *>(zt + voff);
        const int yvec = m.z >= 0 ? (m.z + head) / N : -1;  // the vector holding the sampled id
        float ms = -INFINITY, mt = -INFINITY, dd = 0.f;  // dd: reference difference (fp32 gradient)
        float2 S2 = make_float2(0.f, 0.f), A2 = S2, T2 = S2;
        // this thread's batches of the row: kHelpU vectors of each model, kHelpThreads apart
        const int nbt = nvec > tid ? (nvec - tid + kHelpU * kHelpThreads - 1) / (kHelpU * kHelpThreads) : 0;
        auto slot = [&](int s, int mdl, int u) { return ((s * 2 + mdl) * kHelpU + u) * kHelpThreads + tid; };
        auto issue = [&](int bi) {  // batch bi into the ring (an empty group past the last)
            if (bi < nbt) {
                const int s = bi % kHelpStages, q0 = tid + bi * kHelpU * kHelpThreads;
#pragma unroll
                for (int u = 0; u < kHelpU; ++u) {
                    const int q = q0 + u * kHelpThreads;
                    if (q < nvec && !(TL && cut && q == nvec - 1)) {
                        cp_async16(&hring[slot(s, 0, u)], vs + q);
                        cp_async16(&hring[slot(s, 1, u)], vt + q);
                    }
                }
            }
            cp_async_commit();
        };
        if (AS)
            for (int bi = 0; bi < kHelpStages - 1; ++bi)
                issue(bi);
        for (int bi = 0; bi < nbt; ++bi) {
            const int q0 = tid + bi * kHelpU * kHelpThreads;
            uint4 a[kHelpU], b[kHelpU];
            if (AS) {
                issue(bi + kHelpStages - 1);
                cp_async_wait<kHelpStages - 1>();  // batch bi has landed
            }
#pragma unroll
            for (int u = 0; u < kHelpU; ++u) {
                const int q = q0 + u * kHelpThreads;
                if (TL && cut && q == nvec - 1) {
                    a[u] = E::load_lanes(zs + voff + (size_t)q * N, lanes_lo(q), lanes_hi(q));
                    b[u] = E::load_lanes(zt + voff + (size_t)q * N, lanes_lo(q), lanes_hi(q));
                } else if (q < nvec) {
                    if (AS) {
                        a[u] = hring[slot(bi % kHelpStages, 0, u)];
                        b[u] = hring[slot(bi % kHelpStages, 1, u)];
                    } else {
                        a[u] = __ldg(vs + q);
                        b[u] = __ldg(vt + q);
                    }
                } else {
                    a[u] = b[u] = make_uint4(kFill, kFill, kFill, kFill);
                }
            }
            if (TL && ((head && q0 == 0) || (tail && (unsigned)(nvec - 1 - q0) < (unsigned)(kHelpU * kHelpThreads)))) {
#pragma unroll
                for (int u = 0; u < kHelpU; ++u) {
                    const int q = q0 + u * kHelpThreads;
                    if ((head && q == 0) || (tail && q == nvec - 1)) {
                        a[u] = E::keep_lanes(a[u], lanes_lo(q), lanes_hi(q));
                        b[u] = E::keep_lanes(b[u], lanes_lo(q), lanes_hi(q));
                    }
                }
            }
            // a sampled-token row leaves y out of the student statistics (the fill
            // in its place; add_sampled_term brings its term back at the merge)
            if (SM && (unsigned)(yvec - q0) < (unsigned)(kHelpU * kHelpThreads)) {
#pragma unroll
                for (int u = 0; u < kHelpU; ++u)
                    if (yvec == q0 + u * kHelpThreads)
                        a[u] = E::fill_lane(a[u], (m.z + head) & (N - 1));
            }
            typename E::Max bs = E::max_of(a[0]), bt = E::max_of(b[0]);
#pragma unroll
            for (int u = 1; u < kHelpU; ++u) {
                bs = E::max2(bs, E::max_of(a[u]));
                bt = E::max2(bt, E::max_of(b[u]));
            }
            const float nms = fmaxf(ms, E::value(bs));
            const float nmt = fmaxf(mt, E::value(bt));
            if (nms > ms) {
                const float2 f = splat(ex2((ms - nms) * kLog2e));
                if (kUseD) {  // d at the first element of the batch equal to the new maximum
                    float xd = 0.f;
                    bool found = false;
#pragma unroll
                    for (int u = 0; u < kHelpU; ++u)
#pragma unroll
                        for (int w = 0; w < NP; ++w) {
                            const float2 x = E::pair(a[u], w), y = E::pair(b[u], w);
                            if (!found && x.x == nms) {
                                xd = x.x - y.x;
                                found = true;
                            }
                            if (!found && x.y == nms) {
                                xd = x.y - y.y;
                                found = true;
                            }
                        }
                    A2 = fmul2(ffma2(S2, splat(dd - xd), A2), f);
                    dd = xd;
                } else {
                    A2 = fmul2(A2, f);
                }
                S2 = fmul2(S2, f);
                ms = nms;
            }
            if (nmt > mt) {
                T2 = fmul2(T2, splat(ex2((mt - nmt) * kLog2e)));
                mt = nmt;
            }
            const float2 NS = splat(scale_of(ms)), NTT = splat(scale_of(mt)), D = splat(dd);
#pragma unroll
            for (int u = 0; u < kHelpU; ++u)
#pragma unroll
                for (int w = 0; w < NP; ++w) {
                    const float2 a2 = E::pair(a[u], w), b2 = E::pair(b[u], w);
                    const float2 es = ex2x2(ffma2(a2, L2, NS));
                    S2 = fadd2(S2, es);
                    A2 = ffma2(es, kUseD ? fsub2(fsub2(a2, b2), D) : fsub2(a2, b2), A2);
                    T2 = fadd2(T2, ex2x2(ffma2(b2, L2, NTT)));
                }
        }
        Student S = Student{ms, S2.x + S2.y, A2.x + A2.y, dd};
        Teacher U = Teacher{mt, T2.x + T2.y};
        lane_merge<32, kUseD>(S, U);
        if (lane == 0) {
            red[warp][0] = S.m, red[warp][1] = S.s, red[warp][2] = S.a;
            red[warp][3] = U.m, red[warp][4] = U.s, red[warp][5] = S.d;
        }
        __syncthreads();
        if (warp == 0) {
            Student A = student_empty();
            Teacher B = teacher_empty();
            if (lane < NW) {
                A = Student{red[lane][0], red[lane][1], red[lane][2], red[lane][5]};
                B = Teacher{red[lane][3], red[lane][4]};
            }
            lane_merge<NW, kUseD>(A, B);
            if (lane == 0) {
                const int y = m.z;  // SM: in [0, V) (the compaction drops ids out of range); else -1
                const float omp = SM ? add_sampled_term(A, to_float(zs[off + y])) : 0.f;  // 1 - p_y
                const RowConst rc = row_const(A, B);
                const float e = SM ? (to_float(zs[off + y]) - to_float(zt[off + y])) - rc.dl : rc.kl;
                const float wi = __int_as_float(m.w), wl = wi * e;
                const float sg = wi < 0.f ? -1.f : 1.f;
                if (!isfinite(rc.lse_s) || !isfinite(rc.lse_t) || !isfinite(e))
                    set_status(p.status, TURNOPD_ERR_NONFINITE);
                p.token_loss[m.x] = e;
                p.row_wl[j] = (double)wi * (double)e;
                // the gradient constants of the cluster kernel
                if (kScale) {
                    if (p.grad) {
                        const Scale q = row_scale(A.m, (SM ? -wl : wi) / A.s);
                        bc[0] = q.hi;
                        bc[1] = bc[3] = q.c;
                        bc[5] = -rc.d;
                        bc[6] = -q.c * rc.cp;
                    }
                } else {
                    bc[0] = -rc.lse_s * kLog2e + log2f(fabsf(SM ? wl : wi));  // nlw
                    bc[1] = sg;
                    bc[2] = -sg * (rc.d + rc.cp);  // one rounding of d + cp
                    bc[3] = wl > 0.f ? -1.f : 1.f;
                    bc[5] = -sg * rc.d;            // kGradD
                    bc[6] = -sg * rc.cp;
                }
                bc[4] = wl * omp;              // sampled: g_y = w l (1 - p_y)
            }
        }
        __syncthreads();
        if (p.grad) {
            const float2 NLW = splat(bc[0]), SG = splat(bc[1]), NC = splat(bc[2]), SGL = splat(bc[3]);
            const float2 ND = splat(bc[5]), NCP = splat(bc[6]);
            const float gy = bc[4];
            const int y = m.z;
            for (int q0 = tid; q0 < nfull; q0 += kHelpU * kHelpThreads) {  // (a partial vector 0 is skipped below)
                uint4 a[kHelpU], b[kHelpU];
#pragma unroll
                for (int u = 0; u < kHelpU; ++u) {
                    const int q = q0 + u * kHelpThreads;
                    if (q < nfull) {
                        a[u] = __ldg(vs + q);
                        if (!SM)
                            b[u] = __ldg(vt + q);
                    }
                }
#pragma unroll
                for (int u = 0; u < kHelpU; ++u) {
                    const int q = q0 + u * kHelpThreads;
                    if (q >= nfull)
                        break;
                    if (TL && q < g0)
                        continue;
                    float2 g[NP];
                    if (!SM) {  // full vocabulary: g = w p ((z_s - z_t) - d - cp)
#pragma unroll
                        for (int w = 0; w < NP; ++w) {
                            const float2 a2 = E::pair(a[u], w), b2 = E::pair(b[u], w);
                            const float2 pw = ex2x2(ffma2(a2, L2, NLW)), x = fsub2(a2, b2);
                            g[w] = full_grad<kGradD, kScale>(pw, x, SG, ND, NCP, NC);
                        }
                    } else {  // sampled token: g = -w l p (g_y is written after the loop)
#pragma unroll
                        for (int w = 0; w < NP; ++w)
                            g[w] = fmul2(ex2x2(ffma2(E::pair(a[u], w), L2, NLW)), SGL);
                    }
                    store_grad<T, G32>(p.grad, voff, q, g);
                }
            }
            // a partial vector, column by column
            auto store_lanes = [&](int q) {
                const int lo = lanes_lo(q), hi = lanes_hi(q);
                const size_t to = voff + (size_t)q * N;
                const uint4 a = E::load_lanes(zs + to, lo, hi), b = E::load_lanes(zt + to, lo, hi);
                float2 g[NP];
#pragma unroll
                for (int w = 0; w < NP; ++w) {
                    const float2 a2 = E::pair(a, w), b2 = E::pair(b, w);
                    const float2 pw = ex2x2(ffma2(a2, L2, NLW)), x = fsub2(a2, b2);
                    g[w] = SM ? fmul2(pw, SGL)
                              : full_grad<kGradD, kScale>(pw, x, SG, ND, NCP, NC);
                }
                store_grad_lanes<T, G32>(p.grad, to, g, lo, hi);
            };
            if (TL && tail && (nvec - 1) % kHelpThreads == tid)
                store_lanes(nvec - 1);
            if (TL && head && tid == 0 && !(tail && nvec == 1))
                store_lanes(0);
            // sampled token: g_y = w l (1 - p_y), over the value the vector store wrote
            // (same thread, so the later store wins)
            if (SM && (y + head) / N % kHelpThreads == tid) {
                if (G32)
                    static_cast<float *>(p.grad)[off + y] = gy;
                else
                    static_cast<__nv_bfloat16 *>(p.grad)[off + y] = __float2bfloat16_rn(gy);
            }
        }
        __syncthreads();  // red and bc are reused by the next row
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");  // complete only after the cluster grid
}


// Shapes of a CTA, by the longest slice they hold (kMax vectors).  A shorter slice takes
// smaller groups and more of them, so that as many bytes are in flight and as many rows
// in progress whatever the row's length.  GB/s of the whole step at 4e8 logits of V,
// bf16 (fp32), with a gradient of the same type: Shape32 4,600 at V = 1,024, Shape12
// 4,800 (5,670) at 2,048 (1,024), Shape8 5,400 (6,300) at 4,096, Shape4 5,700 (6,480) at
// 8,192, ShapeMid 5,960 at 12,288, where ShapeBig gives 5,380; rows held in no shape (one
// 256- or 512-thread CTA a row, the second read from L2) reached 820, 1,350, 2,380,
// 3,920 and 3,930, and fp32 rows on clusters of 8 (k_row_split) 186, 370, 736 and 1,370.
struct ShapeBig { static constexpr int NT = 512, G = 2, VPT = 5, ST = 3, kMax = 2405; };  // less in clusters
struct ShapeMid { static constexpr int NT = 320, G = 3, VPT = 6, ST = 4, kMax = 1780; };
struct Shape4 { static constexpr int NT = 256, G = 4, VPT = 5, ST = 5, kMax = 1280; };
struct Shape8 { static constexpr int NT = 128, G = 8, VPT = 5, ST = 10, kMax = 640; };
struct Shape12 { static constexpr int NT = 64, G = 12, VPT = 5, ST = 20, kMax = 320; };
struct Shape32 { static constexpr int NT = 32, G = 32, VPT = 5, ST = 40, kMax = 160; };

template <class Shape> constexpr size_t cluster_smem_bytes(int slice_vec, int cs)
{
    constexpr int ST = Shape::ST, G = Shape::G;
    return (size_t)ST * 2 * slice_vec * 16 + 2 * G * cs * 8 * sizeof(float) +
           ST * sizeof(int4) + (2 * ST + 2 * G) * sizeof(uint64_t) +
           G * (Shape::NT / 32) * 8 * sizeof(float) +  // per-group warp partials
           2 * ((ST + 3) / 4 * 4) * sizeof(int) +                       // row held by each stage, thread reading y
           G * 16 * sizeof(float);                      // broadcast row constants
}
// of the 227 KB a CTA may have, less the static part and alignment
constexpr size_t kMaxClusterSmem = 232448 - 128;

// Cluster size for rows of nvec vectors: the smallest whose slices a CTA holds (0: none).
// That keeps the slices long (a short slice cannot hide the per-row record exchange) and,
// for short rows, puts more SMs in clusters: every SM for 1 and 2, then 36 clusters of 4
// are co-resident, 28 of 5, 23 of 6, 15 of 8, 7 of 16.  7 is left out (only 15).  A CTA holds 2,405
// vectors alone, 2,403 in a cluster of 2, 2,395 of 8 and 2,385 of 16, whose records take more.
inline int cluster_size(int nvec)
{
    static const int kSizes[] = {1, 2, 3, 4, 5, 6, 8, 16};
    for (int c : kSizes)
        if (cluster_smem_bytes<ShapeBig>((nvec + c - 1) / c, c) <= kMaxClusterSmem)
            return c;
    return 0;
}

// The helper's rows per SM and second against the clusters', which decides the
// split of the row list.  A cluster SM is less efficient on a shorter slice and in a
// larger cluster (more records per row), so the rate rises with both; where few SMs are
// left (clusters of 3 to 6) an overloaded helper decides the call.  Measured best (GB/s of
// the step at 4e8 to 1.5e9 logits, or us; slices in vectors):
//   bf16, clusters of 8 at 2,374 (V = 151,936; 8 x 4096 packed tokens): 0.81 (2,724 us;
//   2,759 at 0.72, 2,845 at 0.88), with an fp32 gradient 0.73 (16 x 8192 household tokens
//   2,375; 2,400 at 0.68, 2,431 at 0.76), sampled tokens 0.86 (64 multihop 1,028; 1,049 at
//   0.72); at 2,004 (128,256) 0.92 (6,232; 6,003 at 0.72) and 0.78 (5,865; 5,471 at 0.85);
//   of 16: 0.8 at 1,563 (200,000: 5,487, 5,265 at 0.6), 0.6 at 1,758 (5,405, 5,097 at 0.8), with an
//   fp32 gradient 0.2 less; in ShapeBig (us at 6e8 logits) 0.95 at 1,875 (240,000: 610, 633 at
//   0.8), 0.84 at 2,048 (262,144: 603, 616 at 0.75), 0.65 at 2,344 (300,000: 605, 685 at 0.8), with
//   an fp32 gradient 0.85 (907, 958 at 0.65), 0.8 (826, 868 at 0.6) and 0.7 (825, 964 at 0.8); of 3 in ShapeMid 0.5 (39,000: 6,183, 5,222 at
//   0.7); of 3 to 6 otherwise 0.7 (90,000: 6,335, 6,245 at 0.4), 0.62 with an fp32 gradient
//   (49,152: 6,252 at 0.6, 5,978 at 0.7), of 3 above 2,250 0.6 (57,408: 559 us at 6e8 logits, 590
//   at 0.7);
//   fp32, clusters of 16: 0.69 at 2,374 (151,936: 4 x 4096 packed tokens 2,808 us; 2,833 at
//   0.65, 2,873 at 0.76), 0.80 at 2,048 (6,035, 5,823 at 0.6), 0.65 at 1,719 in ShapeMid
//   (6,361 at 0.6, 6,186 at 0.7), 0.9 at 1,536 (6,203, 5,909 at 0.5), 0.7 at 1,204 in Shape4
//   (6,026, 5,747 at 0.9); of 8 0.70 at 2,350 (6,310, 6,143 at 0.85), more at 2,048 (65,536:
//   6,375 at 0.7, 6,124 at 0.4); of 5 and 6 0.7 (49,152: 6,531, 6,460 at 0.4); of 3 and 4 0.60
//   (28,000: 6,283, 5,562 at 0.75);
//   sampled-token rows, whose helper gradient pass reads the student only: 0.05 more with a
//   bf16 gradient, 0.10 with an fp32 one;
//   forward-only rows, which the helper reads once: 1.0 (bf16 at 2,374: 4,743, 4,478 at 0.7;
//   fp32, clusters of 8 at 2,350: 6,185, 5,836 at 0.7), 0.7 for bf16 in clusters of 3 and 4
//   (57,000: 4,570, 3,443 at 1.0), 0.85 of 5 and 6, 0.9 for fp32 in clusters of 3.
//   bf16 rows that do not all start on a 32-byte sector, which cost the helper's own loads more
//   than the clusters' bulk copies: clusters of 8 0.13 less with a bf16 gradient (V = 151,944: 579
//   us at 0.68, 636 at 0.81), 0.07 less with an fp32 one (820, 880), 0.9 forward (473, 495 at 1.0);
//   of any stride 0.06, 0.04, 0.9 (151,937: 673, 692; 890, 905; 500, 524); of 3 and 4 0.63 (50,008:
//   590, 625 at 0.70; 70,008: 573, 597); of 16 in ShapeBig 0.15, 0.05 (240,008: 631 at 0.8, 670 at
//   0.85; 909, 938).  The other sizes peak where aligned rows do.
template <typename T, int TL>
double helper_rate(int slice_vec, int cs, bool sampled, bool g32, bool forward, bool sectors)
{
    const bool bf16 = sizeof(T) == 2;
    if (forward)
        return cs == 8 && bf16 && !sectors ? 0.9
               : cs >= 8 ? 1.0 : bf16 ? (cs <= 4 ? 0.7 : 0.85) : (cs == 3 ? 0.9 : 1.0);
    double r;
    if (bf16) {
        if (cs == 3 && slice_vec <= ShapeMid::kMax)
            return 0.50;
        if (cs == 3 && slice_vec > 2250)
            return 0.60;
        if (cs < 8)
            return g32 ? 0.62 : cs <= 4 && !sectors && TL != kAny ? 0.63 : 0.70;
        if (cs == 8)
            r = (g32 ? 0.73 + (2374 - slice_vec) * 0.00014 : 0.81 + (2374 - slice_vec) * 0.0003) -
                (sectors ? 0.0 : TL == kAny ? (g32 ? 0.04 : 0.06) : (g32 ? 0.07 : 0.13));
        else if (slice_vec > ShapeMid::kMax)
            r = g32 ? 0.85 - (slice_vec - 1875) * 0.00032 - (sectors ? 0.0 : 0.05)
                    : 0.95 - (slice_vec - 1875) * 0.00064 - (sectors ? 0.0 : 0.15);
        else
            r = (slice_vec > 1563 ? 0.80 - (slice_vec - 1563) * 0.001 : 0.80) - (g32 ? 0.2 : 0.0);
    } else {
        if (cs < 8)
            return cs <= 4 ? 0.60 : 0.70;
        if (cs == 8)
            r = 0.70 + (2350 - slice_vec) * 0.0002;
        else
            r = slice_vec <= Shape4::kMax ? 0.70
                : slice_vec <= ShapeMid::kMax ? 0.90 + (1536 - slice_vec) * 0.0014
                                              : 0.80 + (2048 - slice_vec) * 0.00034;
        r = r > 0.9 ? 0.9 : r;
    }
    r = r < 0.60 ? 0.60 : r;
    return sampled ? r + (g32 ? 0.10 : 0.05) : r;
}

// The cluster grid (as many clusters as are co-resident, cached per device) and
// the helper grid on the SMs the clusters leave free, with the row list split so
// that both finish together.  *used = false (and nothing is launched) where the slices
// do not fit shared memory, or where the device places no cluster of this size (16 is not a
// portable size; a partition of the device may have no room for it).
template <typename T, bool G32, int CS, class Shape, bool SM, int TL>
cudaError_t launch_t(const RowIn &p, int nvec, cudaStream_t stream, bool *used)
{
    auto kern = k_row_cluster<T, CS, Shape::NT, Shape::VPT, Shape::G, Shape::ST, G32, SM, TL>;
    const int slice_vec = (nvec + CS - 1) / CS;
    const size_t smem = cluster_smem_bytes<Shape>(slice_vec, CS);
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return e;
    if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess)
        return e;
    *used = smem + 128 <= (size_t)optin;  // room for the kernel's static shared memory and alignment
    if (!*used)
        return cudaSuccess;
    static int grid_cache[64];  // (per instantiation)
    static size_t smem_cache[64];
    if (dev >= 64)
        return cudaErrorInvalidDevice;
    if (smem_cache[dev] < smem) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess)
            return e;
        if (CS > 8 && (e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess)
            return e;
        smem_cache[dev] = smem;
        grid_cache[dev] = 0;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CS;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.blockDim = dim3(Shape::G * Shape::NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    if (grid_cache[dev] == 0) {
        cfg.gridDim = dim3(CS);
        int ncl = 0;
        e = cudaOccupancyMaxActiveClusters(&ncl, kern, &cfg);
        if (e != cudaSuccess && e != cudaErrorInvalidClusterSize)
            return e;
        if (e != cudaSuccess)
            cudaGetLastError();  // answered below: nothing was launched
        *used = e == cudaSuccess && ncl > 0;
        if (!*used)
            return cudaSuccess;
        grid_cache[dev] = ncl;
    }
    RowIn pl = p;
    const int free_sm = device_sm_count() - grid_cache[dev] * CS;
    if (free_sm > 0) {
        const double cl = (double)(grid_cache[dev] * CS);
        pl.split_den = 1 << 20;
        pl.split_ctas = free_sm;
        pl.split_num = (int32_t)(pl.split_den * cl / (cl + helper_rate<T, TL>(slice_vec, CS, SM, G32, !p.grad, p.ld * (int64_t)sizeof(T) % 32 == 0) * free_sm) + 0.5);
    }
    cfg.gridDim = dim3(grid_cache[dev] * CS);
    e = cudaLaunchKernelEx(&cfg, kern, pl, slice_vec, nvec);
    if (e != cudaSuccess || pl.split_den == 0)
        return e;
    // the helper grid on the free SMs, a dependent of the cluster grid
    cudaLaunchConfig_t hc = {};
    cudaLaunchAttribute ha[1];
    ha[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    ha[0].val.programmaticStreamSerializationAllowed = 1;
    hc.attrs = ha;
    hc.numAttrs = 1;
    hc.gridDim = dim3(free_sm);
    hc.blockDim = dim3(kHelpThreads);
    hc.dynamicSmemBytes = kHelperSmem;
    hc.stream = stream;
    auto helper = k_row_helper<T, G32, SM, TL, true>;
    if ((e = cudaFuncSetAttribute(helper, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)kHelperSmem)) != cudaSuccess)
        return e;
    return cudaLaunchKernelEx(&hc, helper, pl);
}

template <typename T, bool G32, bool SM, int TL>
cudaError_t launch_cs(const RowIn &p, int nvec, cudaStream_t stream, bool *used)
{
    const int cs = cluster_size(nvec);
    const int slice = cs ? (nvec + cs - 1) / cs : 0;
    const int shape = slice <= Shape32::kMax  ? 5
                : slice <= Shape12::kMax  ? 4
                : slice <= Shape8::kMax   ? 3
                : slice <= Shape4::kMax   ? 2
                : slice <= ShapeMid::kMax ? 1
                                          : 0;
    *used = false;
#define TURNOPD_ROWS(CSIZE, SHAPE) launch_t<T, G32, CSIZE, SHAPE, SM, TL>(p, nvec, stream, used)
    switch (cs) {
    case 1:
        switch (shape) {
        case 5: return TURNOPD_ROWS(1, Shape32);
        case 4: return TURNOPD_ROWS(1, Shape12);
        case 3: return TURNOPD_ROWS(1, Shape8);
        case 2: return TURNOPD_ROWS(1, Shape4);
        case 1: return TURNOPD_ROWS(1, ShapeMid);
        default: return TURNOPD_ROWS(1, ShapeBig);
        }
    case 2:
        switch (shape) {
        case 2: return TURNOPD_ROWS(2, Shape4);
        case 1: return TURNOPD_ROWS(2, ShapeMid);
        default: return TURNOPD_ROWS(2, ShapeBig);
        }
    // slices of clusters of 3 to 8 have 1,584 vectors or more, of 16 1,188 or more
    case 3: return shape ? TURNOPD_ROWS(3, ShapeMid) : TURNOPD_ROWS(3, ShapeBig);
    case 4: return TURNOPD_ROWS(4, ShapeBig);
    case 5: return TURNOPD_ROWS(5, ShapeBig);
    case 6: return TURNOPD_ROWS(6, ShapeBig);
    case 8: return TURNOPD_ROWS(8, ShapeBig);
    case 16: return shape == 2 ? TURNOPD_ROWS(16, Shape4) : shape == 1 ? TURNOPD_ROWS(16, ShapeMid) : TURNOPD_ROWS(16, ShapeBig);
    }
#undef TURNOPD_ROWS
    return cudaSuccess;
}

// The helper kernel alone, every row, every SM.
template <typename T, bool G32, bool SM, int TL>
void launch_helper_alone(const RowIn &p, cudaStream_t stream)
{
    RowIn pl = p;
    pl.split_den = 0;
    k_row_helper<T, G32, SM, TL, false><<<device_sm_count(), kHelpThreads, 0, stream>>>(pl);
}

template <typename T, bool G32, bool SM, int TL>
cudaError_t launch_rows_m(const RowIn &p, int nvec, cudaStream_t stream)
{
    bool used = false;
    const cudaError_t e = launch_cs<T, G32, SM, TL>(p, nvec, stream, &used);
    if (e != cudaSuccess || used)
        return e;
    // rows that no cluster holds, or whose cluster size the device cannot place: whole fp32 ones are
    // streamed twice by clusters of 8 (V = 151,936: 5,400 GB/s, held by clusters of 16 6,020)
    if constexpr (std::is_same<T, float>::value && TL == kWhole) {
        return launch_row_split(p, G32, stream);
    } else {
        launch_helper_alone<T, G32, SM, TL>(p, stream);
        return cudaGetLastError();
    }
}

// The row grids for logits of T in rows of form TL.
template <typename T, int TL>
cudaError_t launch_rows_t(const RowIn &p, bool fp32_grad, cudaStream_t stream)
{
    constexpr int N = 16 / (int)sizeof(T);
    // the most vectors a row spans: N - 1 more elements where rows start anywhere in a vector
    const int nvec = (int)((p.vocab + (p.ld % N != 0 ? N - 1 : 0) + N - 1) / N);
    const bool sm = p.mode == TURNOPD_SAMPLED_TOKEN;
    if (fp32_grad)
        return sm ? launch_rows_m<T, true, true, TL>(p, nvec, stream) : launch_rows_m<T, true, false, TL>(p, nvec, stream);
    return sm ? launch_rows_m<T, false, true, TL>(p, nvec, stream) : launch_rows_m<T, false, false, TL>(p, nvec, stream);
}

}  // namespace
}  // namespace turnopd
