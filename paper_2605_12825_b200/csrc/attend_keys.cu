// Block attention for units of few query rows (M = G*K; up to 32, and up to 64 where the wide kernel's plan does
// not suit the number of units) at head_dim 128, and of any number at head_dim 64 (in tiles of up to 128 rows), bf16, both
// views, on tcgen05 with the KEYS on the MMA's rows:
//     S^T [128 keys x NR rows] = K_tile . Q^T        O^T [d x NR rows] = V_tile^T . P^T
// NR = M rounded up to 16, 32, 64 or 128 is the MMA's N.  With the query rows there instead, an M of 4 to 64
// is padded to 128, and only the threads that own real rows take part in the softmax and the
// read-out; here all 128 lanes of the tensor memory hold keys (or head columns), every thread of
// a softmax warpgroup works whatever M is, and a width-1 call costs a quarter of the exponentials.
//
// What bounds it: calls of this size move a few MB, so the chain of one CTA counts: query rows in,
// scores, softmax, P.V, the merge of the cluster's partial results.  Hence 128-key tiles (few steps),
// two softmax warpgroups that take alternate tiles into accumulators and running references of their
// own (no tile waits for another one's maximum), row maxima by redux.sync on the whole warp, and
// addresses worked out ahead of the wait for the preceding kernel.  Per call, chained in a graph,
// against what served these shapes before: 16 units of 4 rows and 2700 keys 16.4 -> 8.5 us; head_dim 64,
// which ran on mma.sync with a second launch for the merge, 10 units of 49 rows and 800 keys 10.9 ->
// 7.0 us, one unit of 128 rows and 4000 keys 15.1 -> 9.4, 256 of 2000 keys 103 -> 68.  A batch of 256
// units of 64 rows at 4000 keys streams at 6.4 TB/s.  From 33 rows at head_dim 128 the kernel for wide
// units, whose tiles are half as long and whose threads hold a row each, takes less from the first score to
// the last product (8 units of 64 rows and 4096 keys 12.4 against 10.1 us; the rule is in api.cu, wide_better).
//
// One CTA (320 threads, up to 64 rows at most 113 KB of shared memory and 256 TMEM columns: two fit an SM, so that
// with programmatic dependent launch the next call's CTAs are resident and, if the caller promised
// a quiescent cache, load their first tiles while this call computes):
//   warps 0-3, 4-7  softmax of tiles 0, 2, 4, ... and 1, 3, 5, ...; thread = key; also the query
//                   rows' way into shared memory, the read-out and the merge
//   warp 8          producer: K and V tiles into a ring of 128-key slots, in the order of their use
//   warp 9          TMEM allocation, both products
// A tile is two 64-key halves, each a box of the cache or the block's own keys, so that a short
// block shares its tile with prefix keys.
//
// Softmax of a tile: the scores are reduced per row over the warp (redux.sync), over the four warps
// through shared memory, and the running reference of a row is raised only when a tile exceeds it
// by more than 2^8 (then O^T's column is rescaled in TMEM); the result is the exact softmax because
// numerator and denominator use the same reference.  References are integers: another reference
// scales a probability by a power of two, so that its rounding to bf16, and with it the result of this kernel up to
// the order of fp32 sums, does not depend on how the keys were cut.  Probabilities are written as
// bf16 rows [key][row], which is the MN-major B operand of the second product; their sums are taken
// over the same rounded values, while that product runs.  (attend_tc.cu rounds the same probabilities but sums
// them before rounding: a call that moves from one kernel to the other keeps its numerators and changes its
// denominators by up to the mean rounding of the probabilities, 2^-9 at most.)
//
// Merge of the S CTAs of a cluster (one unit).  A thread of the read-out holds its head column of four
// query rows per 16 bytes.  Where the CTAs have much to tell one another (`exchanges`), it sends them into
// the ring of the CTA that sums up that column; a cluster barrier before that (every ring is idle; the
// CTAs arrive ahead of the read-out, which hides it), one behind it.  Else through the workspace, which
// stays in L2: a warp's store is 512 contiguous bytes; a cluster barrier publishes them; each CTA then
// sums its share of the (row group, column) elements over the S partials, a lane every fourth partial.
//
// Every mbarrier wait is bounded: on expiry the CTA raises ORTHRUS_DEV_WAIT_TIMEOUT, its warps go
// on through their barriers with void results, the MMAs and copies in flight are waited for, and it ends.
#include <cuda.h>
#include <atomic>
#include <mutex>
#include "common.cuh"
#include "tc_ptx.cuh"

namespace orthrus {
namespace {

constexpr int KT = 128;                    // keys per tile (the MMA's M)
constexpr int HALF = 64;                   // keys per TMA box
constexpr int SW = 8, ST = 256;            // softmax warps and threads
constexpr int PRODUCER_WARP = 8, MMA_WARP = 9, NTHREADS = 320;
constexpr int PANEL = KT * 128;            // bytes of [128 keys][64 columns]
constexpr int MAX_CLUSTER = 16;
constexpr float RAISE = 8.f;               // log2 units

struct KeysMaps { CUtensorMap k, v, kb, vb; };
struct KeysArgs {
    int S, quiescent, ranked;
    uint32_t inv_g;            // ceil(2^16 / G): r / G = r * inv_g >> 16 for r < 128
    int slice;                 // elements of the merge per CTA, a multiple of 8
    int width;                 // XCH: columns that each CTA sums up
    int kb_rows;               // block positions per query tile (blockIdx.z counts the tiles of a unit)
};

template <int HD, int NR> struct KeysShape {
    static constexpr int PANELS = HD / 64;
    static constexpr int KV_BYTES = PANELS * PANEL;
    // up to 64 rows two CTAs share an SM; 128 rows take all of its tensor memory
    static constexpr int CTAS = NR <= 64 ? 2 : 1;
    static constexpr int NSLOT = HD == 128 && NR <= 64 ? 2 : 4;
    static constexpr int Q_BYTES = NR * HD * 2;
    static constexpr int P_PANELS = (NR + 63) / 64, P_BYTES = P_PANELS * PANEL;   // probabilities of a tile
    static constexpr int OFF_RING = 0;
    static constexpr int OFF_P = NSLOT * KV_BYTES;             // per warpgroup [panel][128 keys][128 bytes]
    static constexpr int OFF_Q = OFF_P + 2 * P_BYTES;
    static constexpr int END_Q = OFF_Q + (Q_BYTES > 6144 ? Q_BYTES : 6144);   // (later the tables of the read-out)
    // merge through distributed shared memory, in the ring: partial sums [CTA][row group][column], maxima and
    // sums [CTA][row], weights [CTA][row]
    static constexpr int OFF_XML = 40 * 1024, OFF_XW = OFF_XML + 16 * NR * 8;
    static_assert(HD / 4 * NR * 19 <= OFF_XML && OFF_XW + 16 * NR * 4 <= NSLOT * KV_BYTES, "exchange buffer");
    static constexpr int OFF_REF = END_Q;                      // float [2][NR]: references of the current tiles
    static constexpr int OFF_BAR = OFF_REF + 2 * NR * 4;
    static constexpr int BAR_FULL = 0, BAR_Q = NSLOT, BAR_S = BAR_Q + 1, BAR_P = BAR_S + 2, BAR_PV = BAR_P + 2,
                         BAR_QKALL = BAR_PV + 2, BAR_ALL = BAR_QKALL + 1, BAR_DRAIN = BAR_ALL + 1,
                         NUM_BARS = BAR_DRAIN + 1;
    static constexpr int OFF_MISC = OFF_BAR + NUM_BARS * 8;    // TMEM address, abort flag, sequence
    static constexpr int SMEM_BYTES = OFF_MISC + 16;
    static constexpr uint32_t TM_COLS = 4 * NR;                // two score buffers, two accumulators
    static constexpr uint32_t tm_s(int w) { return (uint32_t)(w * NR); }
    static constexpr uint32_t tm_o(int w) { return (uint32_t)(2 * NR + w * NR); }
    static_assert(CTAS * (SMEM_BYTES + 1024) <= 228 * 1024, "shared memory of an SM");
};

__device__ inline float warp_max(float x) {
    float y;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(y) : "f"(x));
    return y;
}
__device__ inline void store_lane0(uint32_t addr, const float4 &v, int lane) {
    asm volatile("{\n .reg .pred p;\n setp.eq.s32 p, %5, 0;\n @p st.shared.v4.f32 [%0], {%1, %2, %3, %4};\n}"
                 ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(lane) : "memory");
}
// barriers 1 and 2 (a warpgroup of 128 threads each) and 3 (both)
__device__ inline void bar_pair() { asm volatile("bar.sync 3, 256;" ::: "memory"); }
__device__ inline void bar_group(int wg) {
    if (wg == 0) asm volatile("bar.sync 1, 128;" ::: "memory");
    else asm volatile("bar.sync 2, 128;" ::: "memory");
}
// the same, telling whether any of the threads brought `pred`
__device__ inline bool bar_group_or(int wg, bool pred) {
    uint32_t r;
    if (wg == 0)
        asm volatile("{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n barrier.cta.red.or.pred q, 1, 128, p;\n"
                     " selp.u32 %0, 1, 0, q;\n}" : "=r"(r) : "r"((uint32_t)pred) : "memory");
    else
        asm volatile("{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n barrier.cta.red.or.pred q, 2, 128, p;\n"
                     " selp.u32 %0, 1, 0, q;\n}" : "=r"(r) : "r"((uint32_t)pred) : "memory");
    return r != 0;
}
// D fp32, A and B bf16, M = 128, N = n; bit 15 / 16: A / B is MN-major
__host__ __device__ constexpr uint32_t keys_idesc(uint32_t n, uint32_t a_mn, uint32_t b_mn) {
    return make_idesc(n, b_mn) | (a_mn << 15);
}

// A CTA's share [e, e_end) of the merge of S <= 4 U partial results, an element being a head column of
// a group of four rows; called by each softmax warp, no barrier.  A warp takes eight columns at a time,
// its lane groups every fourth partial, a lane U of them; all loads of 8 / U such steps are requested
// together (a step waits for L2 once, about 0.9 us; two CTAs had sixteen steps of two for 128 rows).
template <int HD, int NR, int U, class RowOff>
__device__ inline void merge(const float4 *po, const float2 *pml, float *wt, int e, const int e_end, int M, int S,
                             __nv_bfloat16 *out, const RowOff &row_off)
{
    constexpr int MX = 8 / U, MSTEP = 8 * SW, JS = U == 4 ? 16 : 8, R4 = NR / 4 * HD;
    const int lane = threadIdx.x & 31, el = lane & 7, jg = lane >> 3, r = lane >> 3, j0 = lane & 7;
    e += (threadIdx.x >> 5) * 8;
    po += el + (long long)jg * R4;
    for (; e < e_end; e += MX * MSTEP) {
        float2 ml[MX][U == 4 ? 2 : 1];
        float4 v[MX][U];
        int at[MX];                           // where this lane's result goes (-1: no such row)
#pragma unroll
        for (int x = 0; x < MX; ++x) {
            // rows 4g..4g+3 of the element's group g: lane = (row, partial), with U = 4 twice
            const int ex = e + x * MSTEP, row = ex / HD * 4 + r;
            const bool live = ex < e_end;
#pragma unroll
            for (int w = 0; w < (U == 4 ? 2 : 1); ++w)
                ml[x][w] = live && row < M && j0 + 8 * w < S ? __ldcg(pml + (j0 + 8 * w) * NR + row) : make_float2(-INFINITY, 0.f);
#pragma unroll
            for (int u = 0; u < U; ++u)
                v[x][u] = live && jg + 4 * u < S ? __ldcg(po + ex + u * (4 * R4)) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int x = 0; x < MX; ++x) {
            const int ex = e + x * MSTEP, row = ex / HD * 4 + jg;
            at[x] = ex < e_end && row < M ? row_off(row) + ex % HD + el : -1;
        }
#pragma unroll
        for (int x = 0; x < MX; ++x) {
            if (e + x * MSTEP >= e_end) break;
            float m = ml[x][0].x;
            if constexpr (U == 4) m = fmaxf(m, ml[x][1].x);
#pragma unroll
            for (int off = 4; off; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
            const float w0 = ml[x][0].y > 0.f ? ex2(ml[x][0].x - m) : 0.f;
            float w1 = 0.f, L = w0 * ml[x][0].y;
            if constexpr (U == 4) {
                w1 = ml[x][1].y > 0.f ? ex2(ml[x][1].x - m) : 0.f;
                L = fmaf(w1, ml[x][1].y, L);
            }
#pragma unroll
            for (int off = 4; off; off >>= 1) L += __shfl_xor_sync(0xffffffffu, L, off);
            const float inv = L > 0.f ? 1.f / L : 0.f;
            float *wx = wt + x * (JS * 4);    // weights [partial][row]
            wx[j0 * 4 + r] = w0 * inv;
            if constexpr (U == 4) wx[(j0 + 8) * 4 + r] = w1 * inv;
            __syncwarp();
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const float4 w = *reinterpret_cast<const float4 *>(wx + (jg + 4 * u) * 4);
                acc.x = fmaf(w.x, v[x][u].x, acc.x); acc.y = fmaf(w.y, v[x][u].y, acc.y);
                acc.z = fmaf(w.z, v[x][u].z, acc.z); acc.w = fmaf(w.w, v[x][u].w, acc.w);
            }
            // the four lane groups add up and end with a row each
            const float2 send = jg & 1 ? make_float2(acc.x, acc.z) : make_float2(acc.y, acc.w);
            float2 keep = jg & 1 ? make_float2(acc.y, acc.w) : make_float2(acc.x, acc.z);
            keep.x += __shfl_xor_sync(0xffffffffu, send.x, 8);
            keep.y += __shfl_xor_sync(0xffffffffu, send.y, 8);
            const float give = jg & 2 ? keep.x : keep.y;
            const float y = (jg & 2 ? keep.y : keep.x) + __shfl_xor_sync(0xffffffffu, give, 16);
            if (at[x] >= 0) out[at[x]] = __float2bfloat16_rn(y);
        }
        __syncwarp();
    }
}

// XCH: the merge goes through distributed shared memory
template <int HD, int NR, bool XCH>
__global__ void __launch_bounds__(NTHREADS, KeysShape<HD, NR>::CTAS)
attend_keys_kernel(const AttnParams p, const __grid_constant__ KeysMaps tm, const KeysArgs args)
{
    using C = KeysShape<HD, NR>;
    constexpr int NSLOT = C::NSLOT, PANELS = C::PANELS, QPANEL = NR * 128;
    extern __shared__ __align__(1024) unsigned char smem[];
    const uint32_t sbase = smem_u32(smem);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + C::OFF_MISC);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + C::OFF_MISC + 4);
    volatile int *seq_slot = reinterpret_cast<volatile int *>(smem + C::OFF_MISC + 8);
    auto bar = [&](int i) { return sbase + C::OFF_BAR + i * 8; };
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = blockIdx.x, S = args.S, quiescent = args.quiescent;
    // query tile: block positions [i0, i0 + kb_rows) of the unit, M rows
    const int zt = blockIdx.z, i0 = zt * args.kb_rows, M = min(p.K - i0, args.kb_rows) * p.G;
    // element offset of query row r within the tensor rows of this unit's sequence and head group
    auto row_off = [&](int r) {
        const int i = (int)((uint32_t)r * args.inv_g >> 16);
        return (i * p.Hq + (r - i * p.G)) * HD;
    };

    // ------------------------------------------------------------------ prologue
    if (warp == PRODUCER_WARP && lane == 0) {
        *abort_flag = (sbase & 1023u) == 0 ? 0 : 1;           // swizzled tiles need 1 KB alignment
        *seq_slot = 0;
        for (int i = 0; i < NSLOT; ++i) mbar_init(bar(C::BAR_FULL + i), 1);
        mbar_init(bar(C::BAR_Q), SW);
        for (int w = 0; w < 2; ++w) {
            mbar_init(bar(C::BAR_S + w), 1);
            mbar_init(bar(C::BAR_P + w), 4);
            mbar_init(bar(C::BAR_PV + w), 1);
        }
        mbar_init(bar(C::BAR_QKALL), 1);
        mbar_init(bar(C::BAR_ALL), 1);
        mbar_init(bar(C::BAR_DRAIN), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async();
        prefetch_map(&tm.k); prefetch_map(&tm.v); prefetch_map(&tm.kb); prefetch_map(&tm.vb);
    } else if (warp == MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(C::TM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // Everything that needs no data of earlier kernels is worked out here, ahead of the wait for them:
    // behind it every instruction of a warp's chain counts.
    // where this thread's query chunks (16 bytes each) come from; rows past M are zero
    constexpr int QCH = HD / 8, QN = (NR * QCH + ST - 1) / ST;
    int q_src[QN];
    if (warp < SW) {
#pragma unroll
        for (int u = 0; u < QN; ++u) {
            const int e = tid + u * ST, r = e / QCH;
            q_src[u] = r < M ? row_off(r) / 8 + e % QCH : -1;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    if (!quiescent) griddep_wait();

    // which unit: when the clusters do not all fit at once they go out longest prefix first
    int b = blockIdx.y / p.Hkv;
    const int h = blockIdx.y % p.Hkv;
    const int len_hi = (int)p.len_cap;
    if (args.ranked) {
        for (int i = tid; i < p.B; i += NTHREADS) {
            const int Pi = min(max(__ldg(p.cache_len + i), 0), len_hi);
            int before = 0;
            for (int j = 0; j < p.B; ++j) {
                const int Pj = min(max(__ldg(p.cache_len + j), 0), len_hi);
                before += (Pj > Pi) || (Pj == Pi && j < i);
            }
            if (before == b) *seq_slot = i;
        }
        __syncthreads();
        b = *seq_slot;
    }
    int P = p.cache_len[b];
    if (P < 0 || P > len_hi) {
        if (tid == 0 && rank == 0 && p.status) atomicOr(p.status, ORTHRUS_DEV_BAD_CACHE_LEN);
        P = P < 0 ? 0 : len_hi;
    }
    // the unit's halves: n_pre of 64 prefix keys, then the block's keys, shared out evenly
    const int n_pre = (P + HALF - 1) / HALF, n_all = n_pre + 1;
    const int a0 = (int)((long long)rank * n_all / S), a1 = (int)((long long)(rank + 1) * n_all / S);
    const int nh = a1 - a0, n_mine = max(0, min(nh, n_pre - a0));     // halves of this CTA, prefix halves among them
    const int n_tiles = (nh + 1) >> 1;
    const int row_base = (int)(((long long)(b / p.nb) * p.Hkv + h) * p.capacity);
    // keys of half a (CTA-local): 0 past the end
    auto half_keys = [&](int a) { return a >= nh ? 0 : (a < n_mine ? min(HALF, P - (a0 + a) * HALF) : p.K); };

    // ring items in the order of their use: K0, K1, V0, K2, V1, ..., K(n-1), V(n-2), V(n-1); item i in slot i % NSLOT
    auto item_of_k = [&](int t) { return t == 0 ? 0 : 2 * t - 1; };
    auto item_of_v = [&](int t) { return min(2 * t + 2, 2 * n_tiles - 1); };
    auto is_v = [&](int i) { return i == 2 * n_tiles - 1 || (i > 0 && (i & 1) == 0); };
    auto tile_of = [&](int i) { return is_v(i) ? (i == 2 * n_tiles - 1 ? n_tiles - 1 : i / 2 - 1) : (i + 1) / 2; };
    const uint64_t policy = policy_evict_first();
    auto load_item = [&](int i) {
        const bool v = is_v(i);
        const int t = tile_of(i), slot = i % NSLOT, halves = min(2, nh - 2 * t);
        const uint32_t dst = sbase + C::OFF_RING + slot * C::KV_BYTES, fb = bar(C::BAR_FULL + slot);
        mbar_expect_tx(fb, (uint32_t)(halves * PANELS * HALF * 128));
        for (int a = 2 * t; a < 2 * t + halves; ++a) {
#pragma unroll
            for (int s = 0; s < PANELS; ++s) {
                const uint32_t d = dst + s * PANEL + (a & 1) * (HALF * 128);
                if (a < n_mine || p.blk_in_cache)  // (rows behind the keys hold anything: masked, cleared in V)
                    tma_load_2d(d, v ? &tm.v : &tm.k, s * 64, row_base + (a < n_mine ? (a0 + a) * HALF : P), fb, policy);
                else                                          // rows >= K are out of bounds and arrive as zeros
                    tma_load_4d(d, v ? &tm.vb : &tm.kb, s * 64, h, 0, b, fb);
            }
        }
    };
    const long long unit_row = (((long long)b * p.K + i0) * p.Hq + h * p.G) * HD;
    const uint4 *q = reinterpret_cast<const uint4 *>(static_cast<const __nv_bfloat16 *>(p.q) + unit_row);
    __nv_bfloat16 *out = static_cast<__nv_bfloat16 *>(p.out) + unit_row;
    int produced = 0;
    if (quiescent) {
        // cache rows below cache_len are not being written by the preceding kernel
        if (warp == PRODUCER_WARP && lane == 0)
            while (produced < 2 * n_tiles && produced < NSLOT && min(2 * tile_of(produced) + 2, nh) <= n_mine) {
                load_item(produced); ++produced;
            }
        griddep_wait();
    }
    griddep_launch();

    if (warp < SW) {
        // ------------------------------------------------------------------ query rows
        uint4 qv[QN];
#pragma unroll
        for (int u = 0; u < QN; ++u) qv[u] = q_src[u] >= 0 ? q[q_src[u]] : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < QN; ++u) {
            const int e = tid + u * ST;
            if (e < NR * QCH) *reinterpret_cast<uint4 *>(smem + C::OFF_Q + sw_off(e / QCH, e % QCH, QPANEL)) = qv[u];
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(C::BAR_Q));

        // ------------------------------------------------------------------ softmax, thread = key
        const int wg = warp >> 2, wq = warp & 3, kt = tid & 127;
        const uint32_t lane_base = tmem + ((uint32_t)(wq * 32) << 16);
        const uint32_t TS = lane_base + C::tm_s(wg), TO = lane_base + C::tm_o(wg);
        unsigned char *p_buf = smem + C::OFF_P + wg * C::P_BYTES, *p_row = p_buf + kt * 128;
        float *red = reinterpret_cast<float *>(p_buf);        // [4 warps][NR] until the probabilities take its place
        float *ref = reinterpret_cast<float *>(smem + C::OFF_REF) + wg * NR;
        const float sc = p.scale_log2;
        float m_run = -INFINITY;                              // of row kt (threads kt < NR)
        constexpr int PP = C::P_PANELS, RP = NR / 2 / PP, LG = 32 / RP;   // row pairs of a panel, lane groups that share a warp's keys
        float2 l_run[PP];                                     // of row pair lane % RP of each panel over this warp's keys
#pragma unroll
        for (int x = 0; x < PP; ++x) l_run[x] = make_float2(0.f, 0.f);
        for (int t = wg, u = 0; t < n_tiles; t += 2, ++u) {
            const int a = 2 * t + (kt >> 6), j = kt & 63;     // this thread's half and key in it
            // rows below lo do not see the key (all, if the key does not exist)
            const int lo = j >= half_keys(a) ? NR : (a >= n_mine && p.causal ? (j - i0) * p.G : 0);
            const bool masks = __any_sync(0xffffffffu, lo > 0);
            mbar_wait_warp(bar(C::BAR_S + wg), u & 1, abort_flag);
            if (u > 0) mbar_wait_warp(bar(C::BAR_PV + wg), (u - 1) & 1, abort_flag);   // P buffer and O^T at rest
            tc_fence_after();
            uint32_t s[NR];
            tmem_ld<NR>(TS, s);
            tmem_ld_wait();
            if (masks) {
#pragma unroll
                for (int i = 0; i < NR; ++i) if (i < lo) s[i] = 0xff800000u;
            }
            {   // (each store one step behind its maxima: a warp issues in order and would wait for them)
                const uint32_t red_w = smem_u32(red + wq * NR);
                float4 prev;
#pragma unroll
                for (int i = 0; i < NR + 4; i += 4) {
                    float4 m;
                    if (i < NR)
                        m = make_float4(warp_max(__uint_as_float(s[i])), warp_max(__uint_as_float(s[i + 1])),
                                        warp_max(__uint_as_float(s[i + 2])), warp_max(__uint_as_float(s[i + 3])));
                    if (i > 0) store_lane0(red_w + (i - 4) * 4, prev, lane);
                    prev = m;
                }
            }
            bar_group(wg);
            bool raised = false;
            if (kt < NR) {
                const float m = ceilf(fmaxf(fmaxf(red[kt], red[NR + kt]), fmaxf(red[2 * NR + kt], red[3 * NR + kt])) * sc);
                raised = m > m_run + RAISE;                   // also the first finite maximum
                if (raised) {
                    red[kt] = ex2(m_run - m);                 // the factor of what row kt has summed up so far
                    m_run = m;
                } else {
                    red[kt] = 1.f;
                }
                ref[kt] = m_run == -INFINITY ? 0.f : -m_run;
            }
            if (bar_group_or(wg, raised && u > 0)) {
                // rescale what the earlier tiles have added up
#pragma unroll
                for (int x = 0; x < PP; ++x) {
                    const float2 al = *reinterpret_cast<const float2 *>(red + x * 64 + 2 * (lane % RP));
                    l_run[x].x *= al.x; l_run[x].y *= al.y;
                }
#pragma unroll 1
                for (int c = 0; c < NR; c += 16) {
                    uint32_t o[16];
                    tmem_ld<16>(TO + c, o);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * red[c + i]);
                    tmem_st16(TO + c, o);
                }
                tmem_st_wait();
                bar_group(wg);                                // the factors have been read
            }
            // (a masked score is -inf: its probability is 0.  The references of the next eight columns are
            //  read ahead of the use of these.)
            const float2 sc2 = make_float2(sc, sc);
            float4 ra = *reinterpret_cast<const float4 *>(ref), rb = *reinterpret_cast<const float4 *>(ref + 4);
#pragma unroll
            for (int c = 0; c < NR; c += 8) {
                float2 x[4];
                x[0] = __ffma2_rn(make_float2(__uint_as_float(s[c]), __uint_as_float(s[c + 1])), sc2, make_float2(ra.x, ra.y));
                x[1] = __ffma2_rn(make_float2(__uint_as_float(s[c + 2]), __uint_as_float(s[c + 3])), sc2, make_float2(ra.z, ra.w));
                x[2] = __ffma2_rn(make_float2(__uint_as_float(s[c + 4]), __uint_as_float(s[c + 5])), sc2, make_float2(rb.x, rb.y));
                x[3] = __ffma2_rn(make_float2(__uint_as_float(s[c + 6]), __uint_as_float(s[c + 7])), sc2, make_float2(rb.z, rb.w));
                if (c + 8 < NR) {
                    ra = *reinterpret_cast<const float4 *>(ref + c + 8);
                    rb = *reinterpret_cast<const float4 *>(ref + c + 12);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) s[(c >> 1) + i] = pack_bf16(ex2(x[i].x), ex2(x[i].y));
            }
#pragma unroll
            for (int c = 0; c < NR / 8; ++c)
                *reinterpret_cast<uint4 *>(p_row + (c >> 3) * PANEL + (((c & 7) ^ (kt & 7)) << 4)) =
                    make_uint4(s[4 * c], s[4 * c + 1], s[4 * c + 2], s[4 * c + 3]);
            fence_proxy_async();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(C::BAR_P + wg));
            // while the product runs: the sums of this warp's 32 keys, lane = row pair
#pragma unroll
            for (int pn = 0; pn < PP; ++pn) {
                const int rp = lane % RP;
                float2 l0 = make_float2(0.f, 0.f), l1 = l0;
#pragma unroll 8
                for (int k = lane / RP; k < 32; k += 2 * LG) {
                    const uint32_t x = *reinterpret_cast<const uint32_t *>(p_buf + pn * PANEL + (wq * 32 + k) * 128 +
                                                                           (((rp >> 2) ^ (k & 7)) << 4) + (rp & 3) * 4);
                    const int k2 = k + LG;
                    const uint32_t y = *reinterpret_cast<const uint32_t *>(p_buf + pn * PANEL + (wq * 32 + k2) * 128 +
                                                                           (((rp >> 2) ^ (k2 & 7)) << 4) + (rp & 3) * 4);
                    l0.x += __uint_as_float(x << 16); l0.y += __uint_as_float(x & 0xffff0000u);
                    l1.x += __uint_as_float(y << 16); l1.y += __uint_as_float(y & 0xffff0000u);
                }
                l_run[pn].x += l0.x + l1.x; l_run[pn].y += l0.y + l1.y;
            }
        }
        // ------------------------------------------------------------------ weights of the two warpgroups
#pragma unroll
        for (int off = RP; off < 32; off <<= 1)
#pragma unroll
            for (int x = 0; x < PP; ++x) {
                l_run[x].x += __shfl_xor_sync(0xffffffffu, l_run[x].x, off);
                l_run[x].y += __shfl_xor_sync(0xffffffffu, l_run[x].y, off);
            }
        // the query rows have served: their place takes the tables
        float *t_l = reinterpret_cast<float *>(smem + C::OFF_Q);              // [8 warps][NR] sums
        float *t_m = t_l + 8 * NR, *t_w = t_m + 2 * NR;                       // [2][NR] references, weights
        static_assert((8 + 4) * NR * 4 <= C::END_Q - C::OFF_Q, "tables");
        const int n4 = (M + 3) >> 2;                          // groups of four rows
        const long long cta0 = ((long long)zt * gridDim.y + blockIdx.y) * S, cta = cta0 + rank;
        if (n_tiles > 0) mbar_wait_warp(bar(C::BAR_QKALL), 0, abort_flag);
        else bar_pair();                                      // (no product reads them: every warp has written its own)
        if (lane < RP)
#pragma unroll
            for (int x = 0; x < PP; ++x) *reinterpret_cast<float2 *>(t_l + warp * NR + x * 64 + 2 * lane) = l_run[x];
        if (kt < NR) t_m[wg * NR + kt] = m_run;
        bar_pair();
        float2 ml_row = make_float2(-INFINITY, 0.f);          // of row tid
        if (tid < NR) {
            const float la = (t_l[tid] + t_l[NR + tid]) + (t_l[2 * NR + tid] + t_l[3 * NR + tid]);
            const float lb = (t_l[4 * NR + tid] + t_l[5 * NR + tid]) + (t_l[6 * NR + tid] + t_l[7 * NR + tid]);
            const float ma = t_m[tid], mb = t_m[NR + tid], M = fmaxf(ma, mb);
            float wa = la > 0.f ? ex2(ma - M) : 0.f, wb = lb > 0.f ? ex2(mb - M) : 0.f;
            const float L = wa * la + wb * lb;
            ml_row = make_float2(M, L);
            if (S == 1) { wa /= L; wb /= L; }
            else if (!XCH) __stcg(reinterpret_cast<float2 *>(p.part_ml) + cta * NR + tid, make_float2(M, L));
            t_w[tid] = wa; t_w[NR + tid] = wb;
        }
        if (n_tiles > 0) mbar_wait_warp(bar(C::BAR_ALL), 0, abort_flag);
        if constexpr (XCH) cluster_arrive();                     // the ring is idle
        bar_pair();
        tc_fence_after();
        // ------------------------------------------------------------------ read-out: lane = head column
        const int d = wq * 32 + lane;
        float4 *part = reinterpret_cast<float4 *>(p.part_o) + cta * (NR / 4 * HD) + d;
        if (wq * 32 < HD) {
            constexpr int CW = NR / 2;
            const int c = wg * CW;
            uint32_t oa[CW], ob[CW];
            if (n_tiles > 0) tmem_ld<CW>(lane_base + C::tm_o(0) + c, oa);
            if (n_tiles > 1) tmem_ld<CW>(lane_base + C::tm_o(1) + c, ob);
            tmem_ld_wait();
            // (sums first, stores behind them: the compiler moves no table read over a store)
            float4 x[CW / 4];
#pragma unroll
            for (int i = 0; i < CW; i += 4) {
                x[i / 4] = make_float4(0.f, 0.f, 0.f, 0.f);        // (a CTA without keys contributes zeros)
                if (n_tiles > 0) {
                    const float4 w = *reinterpret_cast<const float4 *>(t_w + c + i);
                    x[i / 4] = make_float4(w.x * __uint_as_float(oa[i]), w.y * __uint_as_float(oa[i + 1]),
                                           w.z * __uint_as_float(oa[i + 2]), w.w * __uint_as_float(oa[i + 3]));
                }
            }
            if (n_tiles > 1) {
#pragma unroll
                for (int i = 0; i < CW; i += 4) {
                    const float4 w = *reinterpret_cast<const float4 *>(t_w + NR + c + i);
                    float4 &y = x[i / 4];
                    y.x = fmaf(w.x, __uint_as_float(ob[i]), y.x); y.y = fmaf(w.y, __uint_as_float(ob[i + 1]), y.y);
                    y.z = fmaf(w.z, __uint_as_float(ob[i + 2]), y.z); y.w = fmaf(w.w, __uint_as_float(ob[i + 3]), y.w);
                }
            }
            if constexpr (XCH) {
                const int q = d / args.width;                 // the CTA that sums up column d
                const uint32_t dst = map_to_rank(sbase, q) + ((rank * (NR / 4) + c / 4) * args.width + d - q * args.width) * 16;
                cluster_wait();
#pragma unroll
                for (int i = 0; i < CW / 4; ++i)
                    if (c / 4 + i < n4) st_cluster(dst + i * args.width * 16, x[i]);
            } else if (S > 1) {
#pragma unroll
                for (int i = 0; i < CW / 4; ++i)
                    if (c / 4 + i < n4) __stcg(part + (c / 4 + i) * HD, x[i]);
            } else {
#pragma unroll
                for (int i = 0; i < CW; ++i) {
                    const float4 y = x[i / 4];
                    if (c + i < M)
                        out[row_off(c + i) + d] = __float2bfloat16_rn(i % 4 == 0 ? y.x : i % 4 == 1 ? y.y : i % 4 == 2 ? y.z : y.w);
                }
            }
        } else if constexpr (XCH) {
            cluster_wait();
        }
        tc_fence_before();
        if constexpr (XCH) {
            if (tid < M)
                for (int q = 0; q < S; ++q) st_cluster(map_to_rank(sbase + C::OFF_XML + (rank * NR + tid) * 8, q), ml_row.x, ml_row.y);
            cluster_sync_all();
            float *wt = reinterpret_cast<float *>(smem + C::OFF_XW);
            if (tid < M) {
                const float2 *ml = reinterpret_cast<const float2 *>(smem + C::OFF_XML) + tid;
                float m = -INFINITY, L = 0.f;
                for (int j = 0; j < S; ++j) m = fmaxf(m, ml[j * NR].x);
                for (int j = 0; j < S; ++j) {
                    const float2 y = ml[j * NR];
                    const float w = y.y > 0.f ? ex2(y.x - m) : 0.f;
                    L = fmaf(w, y.y, L);
                    wt[j * NR + tid] = w;
                }
                const float inv = L > 0.f ? 1.f / L : 0.f;
                for (int j = 0; j < S; ++j) wt[j * NR + tid] *= inv;
            }
            bar_pair();
            const int w0 = rank * args.width, wn = min(args.width, HD - w0);
            for (int e = tid; e < n4 * wn; e += ST) {
                const int g = e / wn, col = e - g * wn;
                const float4 *v = reinterpret_cast<const float4 *>(smem) + g * args.width + col;
                float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
                for (int j = 0; j < S; ++j) {
                    const float4 a = v[j * (NR / 4) * args.width], w = *reinterpret_cast<const float4 *>(wt + j * NR + 4 * g);
                    acc.x = fmaf(w.x, a.x, acc.x); acc.y = fmaf(w.y, a.y, acc.y);
                    acc.z = fmaf(w.z, a.z, acc.z); acc.w = fmaf(w.w, a.w, acc.w);
                }
                const float y[4] = {acc.x, acc.y, acc.z, acc.w};
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (4 * g + k < M) out[row_off(4 * g + k) + w0 + col] = __float2bfloat16_rn(y[k]);
            }
            return;
        } else if (S > 1) {
            float *wt = reinterpret_cast<float *>(smem) + warp * 256;
            const float4 *po = reinterpret_cast<const float4 *>(p.part_o) + cta0 * (NR / 4 * HD);
            const float2 *pml = reinterpret_cast<const float2 *>(p.part_ml) + cta0 * NR;
            cluster_sync_all();
            const int e0 = rank * args.slice, e1 = min(n4 * HD, e0 + args.slice);
            if (S <= 4) merge<HD, NR, 1>(po, pml, wt, e0, e1, M, S, out, row_off);
            else if (S <= 8) merge<HD, NR, 2>(po, pml, wt, e0, e1, M, S, out, row_off);
            else merge<HD, NR, 4>(po, pml, wt, e0, e1, M, S, out, row_off);
            return;
        }
    } else if (warp == PRODUCER_WARP) {
        // ------------------------------------------------------------------ producer
        if (lane == 0) {
            bool ok = !*abort_flag;
            while (produced < 2 * n_tiles && ok) {
                if (produced >= NSLOT) {
                    // the slot is free once the product that read it has retired (which its tile's
                    // softmax, or the accumulator's next user, is told anyway)
                    const int i = produced - NSLOT, t = tile_of(i);
                    ok = mbar_wait(bar((is_v(i) ? C::BAR_PV : C::BAR_S) + (t & 1)), (t >> 1) & 1, abort_flag);
                }
                if (ok) { load_item(produced); ++produced; }
            }
            if (*abort_flag)                                  // copies in flight land before the CTA ends
                for (int i = max(0, produced - NSLOT); i < produced; ++i) {
                    int dummy = 0;
                    mbar_wait(bar(C::BAR_FULL + i % NSLOT), (i / NSLOT) & 1, &dummy);
                }
        }
        __syncwarp();
        if (XCH) cluster_sync_all();
        if (S > 1) cluster_sync_all();
    } else {
        // ------------------------------------------------------------------ MMA issue
        constexpr uint32_t IDESC_QK = keys_idesc(NR, 0, 0);   // A = K tile, B = query rows, both K-major
        constexpr uint32_t IDESC_PV = keys_idesc(NR, 1, 1);   // A = V tile, B = P, both MN-major
        bool ok = __all_sync(0xffffffffu, !*abort_flag);
        auto issue_qk = [&](int t) -> bool {
            const int i = item_of_k(t), slot = i % NSLOT;
            if (!mbar_wait_warp(bar(C::BAR_FULL + slot), (i / NSLOT) & 1, abort_flag)) return false;
            if (t == 0 && !mbar_wait_warp(bar(C::BAR_Q), 0, abort_flag)) return false;
            tc_fence_after();
            if (elect_one()) {
                const uint32_t k_addr = sbase + C::OFF_RING + slot * C::KV_BYTES;
#pragma unroll
                for (int kk = 0; kk < HD / 16; ++kk)
                    umma_ss(tmem + C::tm_s(t & 1), make_desc(k_addr + (kk >> 2) * PANEL + (kk & 3) * 32, 16, 1024),
                            make_desc(sbase + C::OFF_Q + (kk >> 2) * QPANEL + (kk & 3) * 32, 16, 1024), IDESC_QK, kk > 0);
                umma_commit(bar(C::BAR_S + (t & 1)));
                if (t == n_tiles - 1) umma_commit(bar(C::BAR_QKALL));
            }
            __syncwarp();
            return true;
        };
        auto issue_pv = [&](int t) -> bool {
            const int i = item_of_v(t), slot = i % NSLOT, w = t & 1;
            if (!mbar_wait_warp(bar(C::BAR_FULL + slot), (i / NSLOT) & 1, abort_flag)) return false;
            // only the 16-key groups that hold keys are multiplied; V rows behind the keys in the last
            // group may hold anything where they come from the cache, and 0 * NaN would poison the product
            const int k0 = half_keys(2 * t), k1 = half_keys(2 * t + 1);
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                const int n = a ? k1 : k0, pad = -n & 15;
                if (pad && (2 * t + a < n_mine || p.blk_in_cache)) {
                    unsigned char *vt = smem + C::OFF_RING + slot * C::KV_BYTES + a * (HALF * 128);
                    for (int e = lane; e < pad * (HD / 8); e += 32)
                        *reinterpret_cast<uint4 *>(vt + sw_off(n + e / (HD / 8), e % (HD / 8), PANEL)) = make_uint4(0, 0, 0, 0);
                    fence_proxy_async();
                    __syncwarp();
                }
            }
            if (!mbar_wait_warp(bar(C::BAR_P + w), (t >> 1) & 1, abort_flag)) return false;
            tc_fence_after();
            if (elect_one()) {
                const uint32_t v_addr = sbase + C::OFF_RING + slot * C::KV_BYTES, p_addr = sbase + C::OFF_P + w * C::P_BYTES;
                const int g0 = (k0 + 15) >> 4, g1 = (k1 + 15) >> 4;
#pragma unroll
                for (int g = 0; g < 8; ++g)
                    if (g < 4 ? g < g0 : g - 4 < g1)
                        // (head_dim 64: lanes 64-127 take another panel and are not read)
                        umma_ss(tmem + C::tm_o(w), make_desc(v_addr + g * 2048, PANEL, 1024),
                                make_desc(p_addr + g * 2048, PANEL, 1024), IDESC_PV, t > 1 || g > 0);
                if (t == n_tiles - 1) umma_commit(bar(C::BAR_ALL));
                umma_commit(bar(C::BAR_PV + w));
            }
            __syncwarp();
            return true;
        };
        if (ok && n_tiles > 0) ok = issue_qk(0);
        for (int t = 0; t < n_tiles && ok; ++t) {
            if (t + 1 < n_tiles) ok = issue_qk(t + 1);
            if (ok) ok = issue_pv(t);
        }
        if (ok && n_tiles > 0) ok = mbar_wait_warp(bar(C::BAR_ALL), 0, abort_flag);
        if (!ok) {                                            // the MMAs in flight end before TMEM is freed
            if (elect_one()) umma_commit(bar(C::BAR_DRAIN));
            __syncwarp();
            int dummy = 0;
            mbar_wait_warp(bar(C::BAR_DRAIN), 0, &dummy);
        }
        tc_fence_before();
        if (S > 1) {
            if (XCH) cluster_sync_all();
            cluster_sync_all();                               // every warp of this CTA has read its TMEM
            tc_fence_after();
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::TM_COLS) : "memory");
            if (lane == 0 && *abort_flag && p.status) atomicOr(p.status, ORTHRUS_DEV_WAIT_TIMEOUT);
        }
    }
    if (S == 1) {
        __syncthreads();
        tc_fence_after();
        if (warp == MMA_WARP) {
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::TM_COLS) : "memory");
            if (lane == 0 && *abort_flag && p.status) atomicOr(p.status, ORTHRUS_DEV_WAIT_TIMEOUT);
        }
    }
}

// function attributes belong to a device: set them once on each device that launches
template <int HD, int NR, bool XCH> cudaError_t configure(int *dev)
{
    constexpr int kMaxDevices = 64;
    static std::mutex mu;
    static bool configured[kMaxDevices] = {};
    cudaError_t e = cudaGetDevice(dev);
    if (e != cudaSuccess) return e;
    if (*dev < 0 || *dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (!configured[*dev]) {
        auto kern = attend_keys_kernel<HD, NR, XCH>;
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, KeysShape<HD, NR>::SMEM_BYTES);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
        configured[*dev] = true;
    }
    return cudaSuccess;
}

// Clusters of S CTAs the current device keeps resident at once.  Two CTAs fit an SM, and a cluster
// stays within a GPC, so that this is less than 2 x 148 / S.  The query counts one CTA per SM for
// kernels that allocate tensor memory: asked for clusters of S / 2 (rounded up) it tells how many
// groups of that many SMs there are (33 of 4, 15 of 8 on a B200; 32 clusters of 8 CTAs were measured
// to run in one wave, 16 of 16 not).  Asked once per device and size.
template <int HD, int NR> int resident_clusters(int S)
{
    constexpr int kMaxDevices = 64;
    static std::atomic<int> cached[kMaxDevices][MAX_CLUSTER + 1];
    int dev = 0;
    constexpr int CTAS = KeysShape<HD, NR>::CTAS;
    if (configure<HD, NR, false>(&dev) != cudaSuccess) { (void)cudaGetLastError(); return CTAS * kDefaultSMs / S; }
    int n = cached[dev][S].load(std::memory_order_relaxed);
    if (n != 0) return n > 0 ? n : 0;
    cudaLaunchConfig_t cfg = {};
    const int sms = (S + CTAS - 1) / CTAS;
    cfg.gridDim = dim3(sms, 1);
    cfg.blockDim = dim3(NTHREADS);
    cfg.dynamicSmemBytes = KeysShape<HD, NR>::SMEM_BYTES;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = sms; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, attend_keys_kernel<HD, NR, false>, &cfg) != cudaSuccess || n < 1) {
        (void)cudaGetLastError();
        n = sms <= 8 ? num_sms() / sms : 0;       // a size the device cannot schedule is not chosen
    }
    if (S == 1) n *= CTAS;
    cached[dev][S].store(n < 1 ? -1 : n, std::memory_order_relaxed);
    return n;
}

// Clusters of up to four CTAs that exchange 4 KB or more with each other merge through distributed shared
// memory.  Measured per call, through L2 against exchanged: d = 128, 32 rows: 128 units of 1000 keys (2 CTAs) 17.5 and
// 16.2 us, of 400 10.9 and 9.4, 64 of 2000 (4) 15.8 and 15.1; 64 rows: 128 of 1000 (2) 22.1 and 18.4, 64 of 2000 (4)
// 19.2 and 17.8; d = 64, 128 rows: 64 of 2000 (2) 26.3 and 23.6; but d = 128, 32 rows: 32 units of 1000 keys (8) 8.3 and 8.8,
// 8 of 4000 (16) 8.3 and 9.7; d = 64, 64 rows: 32 of 1000 (8) 8.8 and 9.5.
constexpr bool exchanges(int d, int nr, int S) { return S > 1 && S <= 4 && nr >= 32 && nr * d >= 1024 * S; }

// CTAs per unit.  A CTA's time is that of its tiles one after the other; a merge costs as much as one
// tile and, for what it moves, up to two more; a second wave of clusters costs more than any split
// gains.  So: the cheapest by that count among the sizes at which all units are resident together.
// Of sizes that cost the same the largest up to 8 (lengths are often below the bound the plan is
// made for, and then the larger size has fewer tiles), else the smallest; above 10 a single tile per
// CTA gains nothing over two.  Measured per call, chained in a graph, lengths 0.7 to 1 times the bound:
// d = 128, 32 rows: 8 units, bound 150, 5.1 us at 1 CTA, 5.8 at 2; bound 2000, 6.6 us at 10, 8.1 at 8; bound 4000,
// 8.2 us at 16, 10.4 at 8; 32 units, bound 2000, 10.1 at 8, 16.8 at 9 (not all resident); 128 units, bound 400, 9.5 us at 2, 10.7 at 1;
// 256 units, bound 2000, 43 us at 1, 49 at 2; 4 rows: 8 units, bound 400, 4.6 us at 5, 7.2 at 1; bound 4000, 7.2 at 16,
// 9.4 at 8; 64 rows: 12 units, bound 8000, 15.2 us at 16, 19.5 at 8; 42 units, bound 6000, 27.1 at 6, 31.6 at 4, 38.0 at 7 (not
// all resident); 256 units, bound 2000, 45 us at 1, 54 at 2; d = 64, 32 rows: 2 units, bound 1000, 4.5 us at 10, 5.0 at 8, 10.8 at 1.
template <int HD, int NR> int choose_splits(int units, int halves)
{
    int best = 1, best_cost = 1 << 30;
    for (int S = 1; S <= MAX_CLUSTER && S <= halves; ++S) {
        const int tiles = max(S <= 10 ? 1 : 2, ((halves + S - 1) / S + 1) / 2);
        const int cost = 2 * tiles + (S > 1 ? 2 + NR * HD / 2048 : 0);
        if (S <= 8 ? cost > best_cost : cost >= best_cost) continue;
        if (S > 1 && units > resident_clusters<HD, NR>(S)) continue;
        best = S;
        best_cost = cost;
    }
    return best;
}

template <int HD, int NR, bool XCH = false>
cudaError_t launch_shape(const AttnParams &p, const KeysMaps &tm, int flags, cudaStream_t st)
{
    using C = KeysShape<HD, NR>;
    if constexpr (!XCH && exchanges(HD, NR, 2))
        if (exchanges(HD, NR, p.n_splits)) return launch_shape<HD, NR, true>(p, tm, flags, st);
    auto kern = attend_keys_kernel<HD, NR, XCH>;
    int dev = 0;
    cudaError_t e = configure<HD, NR, XCH>(&dev);
    if (e != cudaSuccess) return e;
    const int S = p.n_splits, units = p.B * p.Hkv, kb = tc_kb_rows(p.G, p.K), tiles = (p.K + kb - 1) / kb;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(S, units, tiles);
    cfg.blockDim = dim3(NTHREADS);
    cfg.dynamicSmemBytes = C::SMEM_BYTES;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int n_attr = 0;
    if (S > 1) {
        attr[n_attr].id = cudaLaunchAttributeClusterDimension;
        attr[n_attr].val.clusterDim.x = S; attr[n_attr].val.clusterDim.y = 1; attr[n_attr].val.clusterDim.z = 1;
        ++n_attr;
    }
    if (p.early) {
        attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n_attr].val.programmaticStreamSerializationAllowed = 1;
        ++n_attr;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n_attr;
    KeysArgs args;
    args.S = S;
    args.quiescent = (flags & ORTHRUS_LAYER_CACHE_QUIESCENT) ? 1 : 0;
    args.ranked = units * tiles * S > C::CTAS * num_sms() && p.B > 1 && p.B <= 128;
    args.inv_g = (65536u + p.G - 1) / p.G;
    args.slice = (((kb * p.G + 3) / 4 * HD + S - 1) / S + 7) & ~7;
    args.kb_rows = kb;
    args.width = (HD + S - 1) / S;
    e = cudaLaunchKernelEx(&cfg, kern, p, tm, args);
    count_launch();
    return e;
}

template <int HD>
cudaError_t launch_rows(const AttnParams &p, const KeysMaps &tm, int flags, cudaStream_t st)
{
    switch (keys_rows(HD, p.G, p.K)) {
    case 16: return launch_shape<HD, 16>(p, tm, flags, st);
    case 32: return launch_shape<HD, 32>(p, tm, flags, st);
    case 64: return launch_shape<HD, 64>(p, tm, flags, st);
    }
    if constexpr (HD == 64) return launch_shape<HD, 128>(p, tm, flags, st);
    return cudaErrorInvalidValue;
}

}  // namespace

// columns of the MMA that a unit's query rows take (0: not a shape of this kernel)
int keys_rows(int d, int G, int K)
{
    const int M = G * K;
    if (d == 64 && M > 64) return G <= 128 ? 128 : 0;
    return M <= 16 ? 16 : M <= 32 ? 32 : M <= 64 ? 64 : 0;
}

int keys_splits(int d, int G, int K, int units, int max_keys)
{
    // the layers of a pass ask the same question: the last answer of this thread is kept
    struct Key { int dev, d, nr, units, halves, S; };
    static thread_local Key last = {-1, 0, 0, 0, 0, 0};
    Key k = {-1, d, keys_rows(d, G, K), units, (max_keys + HALF - 1) / HALF + 1, 0};   // (prefix and block in halves of their own)
    if (cudaGetDevice(&k.dev) != cudaSuccess) { (void)cudaGetLastError(); k.dev = -2; }
    if (k.dev == last.dev && k.d == last.d && k.nr == last.nr && k.units == last.units && k.halves == last.halves) return last.S;
    switch (k.nr) {
    case 16: k.S = d == 64 ? choose_splits<64, 16>(units, k.halves) : choose_splits<128, 16>(units, k.halves); break;
    case 32: k.S = d == 64 ? choose_splits<64, 32>(units, k.halves) : choose_splits<128, 32>(units, k.halves); break;
    case 64: k.S = d == 64 ? choose_splits<64, 64>(units, k.halves) : choose_splits<128, 64>(units, k.halves); break;
    default: k.S = choose_splits<64, 128>(units, k.halves);
    }
    last = k;
    return k.S;
}

int keys_resident_clusters(int S) { return resident_clusters<128, 64>(S); }

cudaError_t launch_attend_keys(const AttnParams &p, int flags, cudaStream_t st)
{
    KeysMaps tm;
    const unsigned long long rows = (unsigned long long)(p.B / p.nb) * p.Hkv * p.capacity;
    if (!tensor_map(p.k_cache, p.d, rows, 0, 0, HALF, 0, &tm.k) || !tensor_map(p.v_cache, p.d, rows, 0, 0, HALF, 0, &tm.v))
        return cudaErrorInvalidValue;
    if (p.blk_in_cache) {
        tm.kb = tm.k; tm.vb = tm.v;           // unused: the block's keys come through the cache maps
    } else if (!tensor_map(p.k_blk, p.d, p.Hkv, p.K, p.B, 1, HALF, &tm.kb) ||
               !tensor_map(p.v_blk, p.d, p.Hkv, p.K, p.B, 1, HALF, &tm.vb)) {
        return cudaErrorInvalidValue;
    }
    return p.d == 64 ? launch_rows<64>(p, tm, flags, st) : launch_rows<128>(p, tm, flags, st);
}

}  // namespace orthrus
