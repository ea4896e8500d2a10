// Block attention for units of few query rows (M = G*K; up to 64, up to 128 in two tiles where latency counts; the lines are in
// api.cu) at head_dim 128, and of any number at head_dim 64 (in tiles of up to 128 rows), bf16, both
// views, on tcgen05 with the KEYS on the MMA's rows:
//     S^T [128 keys x NR rows] = K_tile . Q^T        O^T [d x NR rows] = V_tile^T . P^T
// NR = M rounded up to 16, 32, 64 or 128 is the MMA's N.  With the query rows there instead, an M of 4 to 64
// is padded to 128, and only the threads that own real rows take part in the softmax and the
// read-out; here all 128 lanes of the tensor memory hold keys (or head columns), every thread of
// a softmax warpgroup works whatever M is, and a width-1 call costs a quarter of the exponentials.
//
// What bounds it: calls of this size move a few MB, so the chain of one CTA counts: query rows in,
// scores, softmax, P.V, the merge of the cluster's partial results.  Measured for the steps of that chain (cycles): eight MMAs
// of 128 keys 470 to 550 with 16 to 64 query rows (the A operand's way through shared memory), a named barrier 17,
// an mbarrier 54 from the arrival to a waiting thread, the arrival at a cluster barrier 330 with its release and 18
// without, 32 KB to the other CTAs of a cluster 2000 to 3000 whatever the instruction, and the instruction cache: 32 KB, up
// to which straight code runs at an instruction a cycle, beyond at a third of that and with hundreds of cycles for a jump.
// Hence short code, 128-key tiles (few steps), two softmax warpgroups that take alternate tiles into
// accumulators and references of their own, references of zero, loads that are under way before anything else is set up,
// one cluster barrier without a release, and a merge that waits for the messages themselves.
// Per call, chained in a graph, against this kernel with 104 to 122 KB of code, row maxima by redux.sync for every tile and
// the merge through L2 or with two cluster barriers: 16 units of 4 rows and 2700 keys 7.4 -> 6.3 us, 8 of 4 rows and
// 4000 keys 7.2 -> 5.7, 8 of 64 rows and 4000 keys 10.2 -> 8.6, 32 of 64 rows and 1900 keys 12.0 -> 10.5, at head_dim 64 one
// unit of 128 rows and 4000 keys 9.4 -> 7.2 (2 units of 112 rows), 10 of 49 rows and 800 keys 6.5 -> 4.7, 2 of 32 rows and 512 keys
// 4.5 -> 3.5; 256 units of 64 rows and 2000 keys 45 -> 46.
//
// One CTA (320 threads, up to 64 rows at most 113 KB of shared memory and 256 TMEM columns: two fit an SM, so that
// with programmatic dependent launch the next call's CTAs are resident and, if the caller promised
// a quiescent cache, load their first tiles while this call computes):
//   warps 0-3, 4-7  softmax of tiles 0, 2, 4, ... and 1, 3, 5, ...; thread = key; also the query
//                   rows' way into shared memory, the read-out and the merge
//   warp 8          producer: K and V tiles into a ring of 128-key slots, in the order of their use
//   warp 9          TMEM allocation, both products, the loads of the block's own keys
// A tile is two 64-key halves, each a box of the cache or the block's own keys, so that a short
// block shares its tile with prefix keys.
//
// Softmax of a tile: a row's reference starts at 0 and is left alone as long as no probability exceeds 2^40 and, in a
// warpgroup's first tile, no probability of its first key, which every row sees, is below 2^-60: floating-point numbers keep their
// relative precision whatever the reference, so that the maximum itself is not needed.  Otherwise (a vote of the warpgroup) the
// references are raised to the rows' maxima (redux.sync over the warp, shared memory over the four warps) and what
// earlier tiles have added up is rescaled.  The result is the exact softmax because
// numerator and denominator use the same reference.  A tile that moves them takes its exponentials twice: 8 units of 64 rows, 4000 keys, with
// all scores about +60 or -60 10.4 us a call instead of 8.6 (9.9 in a kernel that took every tile's maxima), 128 rows 13.4 instead of
// 11.2 (12.2), 4 rows 6.5 instead of 6.2; scores of standard deviation 3 cost nothing.  (The first key's scores as
// references before the maxima gained 0.1 us of it where all scores are alike and lost 1 where they are not.)  References are integers: another reference
// scales a probability by a power of two, so that its rounding to bf16, and with it the result of this kernel up to
// the order of fp32 sums, does not depend on how the keys were cut.  Probabilities are written as
// bf16 rows [key][row], which is the MN-major B operand of the second product; their sums are taken
// over the same rounded values, while that product runs.  (attend_tc.cu rounds the same probabilities but sums
// them before rounding: a call that moves from one kernel to the other keeps its numerators and changes its
// denominators by up to the mean rounding of the probabilities, 2^-9 at most.)
//
// Merge of the S CTAs of a cluster (one unit), through distributed shared memory.  Four query rows by 32 head columns are a task;
// task i belongs to CTA i mod S.  Every CTA sends its part of a task, with its references and sums, into the owner's ring (a
// cluster barrier says that it is idle; the CTAs arrive ahead of the read-out, which hides it) by stores that the
// owner's mbarrier counts; the owner's warps wait for that count and add up.  Nothing goes through L2: the
// workspace of a call holds its header only.
//
// Every mbarrier wait is bounded: on expiry the CTA raises ORTHRUS_DEV_WAIT_TIMEOUT, its warps go
// on through their barriers with void results, the MMAs and copies in flight are waited for, and it ends.
#include <cuda.h>
#include <float.h>
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
constexpr uint32_t P_HIGH = 0x5380, P_LOW = 0x2180;   // 2^40 and 2^-60 as bf16: what an unshifted probability may be
constexpr int MSG = 512 + 32;              // a message of the merge: 32 columns of four rows, their references, their sums

struct KeysMaps { CUtensorMap k, v, kb, vb; };
struct KeysArgs {
    int S, quiescent, ranked;
    uint32_t inv_g;            // ceil(2^16 / G): r / G = r * inv_g >> 16 for r < 128
    uint32_t inv_s;            // ceil(2^16 / S), likewise
    uint32_t inv_s32;          // ceil(2^32 / S): n / S = n * inv_s32 >> 32 for n < 2^25
    int kb_rows;               // block positions per query tile
    int tiles;                 // query tiles of a unit; blockIdx.y = tile * KV heads + head
};

template <int HD, int NR> struct KeysShape {
    static constexpr int PANELS = HD / 64;
    static constexpr int KV_BYTES = PANELS * PANEL;
    // up to 64 rows two CTAs share an SM; 128 rows take all of its tensor memory
    static constexpr int CTAS = NR <= 64 ? 2 : 1;
    static constexpr int Q_BYTES = NR * HD * 2;
    static constexpr int P_PANELS = (NR + 63) / 64, P_BYTES = P_PANELS * PANEL;   // probabilities of a tile
    // Ring of K and V tiles, behind it the probabilities of the two warpgroups [panel][128 keys][128 bytes].  At
    // head_dim 128 a CTA of two tiles, the usual one where latency counts, puts them where K0 was and has a third slot
    // instead: K0, K1 and V0 arrive ahead of the query rows, and V1 takes the place of K1.
    static constexpr int NSLOT = HD == 128 ? 2 : 4;
    static constexpr bool FOLD = HD == 128;
    static constexpr int OFF_RING = 0;
    static constexpr int OFF_P = NSLOT * KV_BYTES;
    static constexpr int OFF_Q = OFF_P + 2 * P_BYTES;
    static_assert(!FOLD || 2 * P_BYTES == KV_BYTES, "the third slot is the place of the probabilities");
    static constexpr int END_Q = OFF_Q + (Q_BYTES > 6144 ? Q_BYTES : 6144);   // (later the tables of the read-out)
    static constexpr int OFF_REF = END_Q;                      // float [2][NR]: minus the references of the current tiles
    static constexpr int OFF_BAR = OFF_REF + 2 * NR * 4;
    static constexpr int BAR_FULL = 0, BAR_Q = NSLOT + FOLD, BAR_S = BAR_Q + 1, BAR_P = BAR_S + 2, BAR_PV = BAR_P + 2,
                         BAR_QKALL = BAR_PV + 2, BAR_ALL = BAR_QKALL + 1, BAR_DRAIN = BAR_ALL + 1,
                         BAR_X = BAR_DRAIN + 1, NUM_BARS = BAR_X + 1;
    static constexpr int OFF_MISC = OFF_BAR + NUM_BARS * 8;    // TMEM address, abort flag, sequence
    static constexpr int SMEM_BYTES = OFF_MISC + 16;
    // the merge, in the ring: [task of this CTA][CTA] messages, then weights [warp][CTA][row]
    static constexpr int TASKS = NR / 4 * (HD / 32);
    static constexpr int OFF_XW = (TASKS + MAX_CLUSTER) * MSG;
    static constexpr int OFF_XB = OFF_XW + SW * (MAX_CLUSTER + 1) * 16;       // a task's part from the block's own keys [warp][row][column]
    static_assert(OFF_XB + SW * 512 <= OFF_Q, "exchange buffer");
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
    asm volatile("{\n .reg .pred p;\n setp.eq.s32 p, %5, 0;\n@p st.shared.v4.f32 [%0], {%1, %2, %3, %4};\n}"
                 ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(lane) : "memory");
}
// barriers 1 and 2 (a warpgroup of 128 threads each), 3 (both), 4 (both and the MMA warp), 5 (all), 6 (MMA warp and producer)
__device__ inline void bar_pair() { asm volatile("bar.sync 3, 256;" ::: "memory"); }
__device__ inline void bar_group(int wg) {
    if (wg == 0) asm volatile("bar.sync 1, 128;" ::: "memory");
    else asm volatile("bar.sync 2, 128;" ::: "memory");
}
__device__ inline void bar_tmem_arrive() { asm volatile("bar.arrive 4, 288;" ::: "memory"); }
__device__ inline void bar_tmem_wait() { asm volatile("bar.sync 4, 288;" ::: "memory"); }
__device__ inline void bar_start_arrive() { asm volatile("bar.arrive 5, 320;" ::: "memory"); }
__device__ inline void bar_start_wait() { asm volatile("bar.sync 5, 320;" ::: "memory"); }
__device__ inline void bar_issue_arrive() { asm volatile("bar.arrive 6, 64;" ::: "memory"); }
__device__ inline void bar_issue_wait() { asm volatile("bar.sync 6, 64;" ::: "memory"); }
// bar_group, telling whether any of the threads brought `pred`
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

// A block's own keys apart from the tiles (APART): what a unit's query rows 4 g to 4 g + 3 get from them in 32 head columns, by the
// warp that merges these.  Sixteen keys at a time by mma.sync, query rows (four of the sixteen) on its rows, the 128 head columns of the
// first product in an order of their own, the same for both sides; probabilities, references and sums as a tile's.
struct BlockPart { float m, l, o[4][2]; };                   // of row lane / 4 (lanes below 16); columns 8 t + 2 (lane % 4), + 1
__device__ inline void mma_16x8x16(float *d, uint32_t a0, uint32_t a2, uint32_t b0, uint32_t b1) {      // (rows 8 to 15 of A are zero)
    float x = 0.f, y = 0.f;
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(x), "+f"(y) : "r"(a0), "r"(0u), "r"(a2), "r"(0u), "r"(b0), "r"(b1));
}
__device__ inline uint32_t transposed_8x8(uint32_t x) {
    uint32_t y;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}
// q: query row lane / 4 (any where there is none); k, v: row 0 of the block's keys and of the 32 columns of its values, `stride`
// elements apart; sees: keys that the row sees
__device__ inline BlockPart block_part(const __nv_bfloat16 *q, const __nv_bfloat16 *k, const __nv_bfloat16 *v, long long stride, int K,
                                       int sees, float sc, int lane)
{
    constexpr int HD = 128;
    BlockPart r = {-INFINITY, 0.f, {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}}};
    const int part = (lane & 3) * 8, key = lane >> 2, j0 = (lane & 3) * 2;
    uint4 qv[HD / 32];
#pragma unroll
    for (int x = 0; x < HD / 32; ++x) qv[x] = *reinterpret_cast<const uint4 *>(q + x * 32 + part);
#pragma unroll 1
    for (int k0 = 0; k0 < K; k0 += 16) {
        // (rows behind the block's last are that one again: their probabilities are zero)
        const long long row0 = min(k0 + key, K - 1) * stride, row1 = min(k0 + key + 8, K - 1) * stride;
        uint4 ka[HD / 32], kb[HD / 32];
        uint32_t va[4], vb[4];
#pragma unroll
        for (int x = 0; x < HD / 32; ++x) {
            ka[x] = *reinterpret_cast<const uint4 *>(k + row0 + x * 32 + part);
            kb[x] = *reinterpret_cast<const uint4 *>(k + row1 + x * 32 + part);
        }
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            va[t] = *reinterpret_cast<const uint32_t *>(v + row0 + t * 8 + j0);
            vb[t] = *reinterpret_cast<const uint32_t *>(v + row1 + t * 8 + j0);
        }
        float d[2][2] = {{0.f, 0.f}, {0.f, 0.f}};             // keys k0 + j0, + 1 and those 8 on
#pragma unroll
        for (int x = 0; x < HD / 32; ++x) {
            mma_16x8x16(d[0], qv[x].x, qv[x].y, ka[x].x, ka[x].y);
            mma_16x8x16(d[1], qv[x].x, qv[x].y, kb[x].x, kb[x].y);
            mma_16x8x16(d[0], qv[x].z, qv[x].w, ka[x].z, ka[x].w);
            mma_16x8x16(d[1], qv[x].z, qv[x].w, kb[x].z, kb[x].w);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) if (k0 + j0 + (i & 1) + (i & 2) * 4 >= sees) d[i >> 1][i & 1] = -INFINITY;
        float top = fmaxf(fmaxf(d[0][0], d[0][1]), fmaxf(d[1][0], d[1][1]));
        top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, 1));
        top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, 2));
        const float m = fmaxf(r.m, ceilf(top * sc)), ref = m == -INFINITY ? 0.f : m, al = ex2(r.m - ref);     // (of nothing so far: 0)
        r.m = m;
        const uint32_t wa = pack_bf16(ex2(fmaf(d[0][0], sc, -ref)), ex2(fmaf(d[0][1], sc, -ref)));
        const uint32_t wb = pack_bf16(ex2(fmaf(d[1][0], sc, -ref)), ex2(fmaf(d[1][1], sc, -ref)));
        r.l = fmaf(r.l, al, (__uint_as_float(wa << 16) + __uint_as_float(wa & 0xffff0000u)) + (__uint_as_float(wb << 16) + __uint_as_float(wb & 0xffff0000u)));
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            r.o[t][0] *= al; r.o[t][1] *= al;
            mma_16x8x16(r.o[t], wa, wb, transposed_8x8(va[t]), transposed_8x8(vb[t]));
        }
    }
    r.l += __shfl_xor_sync(0xffffffffu, r.l, 1);
    r.l += __shfl_xor_sync(0xffffffffu, r.l, 2);
    return r;
}

// XCH: several CTAs share a unit and exchange their partial results.
// APART: the tiles hold prefix keys only; the block's own, which would be one CTA's third tile, are left to the warps that merge, while
// they wait for messages (8 units of 64 rows, 4096 keys and blocks of 16: sixteen CTAs of two tiles each).
// The code is kept short on purpose (loops not unrolled, one place for each wait, copy and product): the warps' roles are
// run through once or twice per call, and an SM's instruction cache holds 32 KB.
template <int HD, int NR, bool XCH, bool APART>
__device__ __forceinline__ void attend_keys(const AttnParams &p, const KeysMaps &tm, const KeysArgs &args)
{
    using C = KeysShape<HD, NR>;
    constexpr int PANELS = C::PANELS, QPANEL = NR * 128;
    extern __shared__ __align__(1024) unsigned char smem[];
    const uint32_t sbase = smem_u32(smem);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + C::OFF_MISC);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + C::OFF_MISC + 4);
    auto bar = [&](int i) { return sbase + C::OFF_BAR + i * 8; };
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = XCH ? blockIdx.x : 0, S = XCH ? args.S : 1, quiescent = args.quiescent;
    // query tile: block positions [i0, i0 + kb_rows) of the unit, M rows
    const int zt = args.tiles > 1 ? blockIdx.y / (unsigned)p.Hkv : 0, i0 = zt * args.kb_rows, M = min(p.K - i0, args.kb_rows) * p.G;
    // element offset of query row r within the tensor rows of this unit's sequence and head group
    auto row_off = [&](int r) {
        const int i = (int)((uint32_t)r * args.inv_g >> 16);
        return (i * p.Hq + (r - i * p.G)) * HD;
    };
    // A task of the merge: four query rows, 32 head columns.  Task i belongs to CTA i % S of the cluster.
    const int n4 = (M + 3) >> 2, n_tasks = n4 * (HD / 32);
    const int my_tasks = (int)((uint32_t)(n_tasks - rank + S - 1) * args.inv_s >> 16);

    // ------------------------------------------------------------------ prologue
    int b = blockIdx.z, P = 0;
    const bool len_first = quiescent && !args.ranked;         // the length is on its way while the barriers are set up
    if (len_first) P = p.cache_len[b];
    // The producer is to ask for its first tiles as early as can be: it sets up the barriers of the ring and waits for nobody.
    if (warp == PRODUCER_WARP) {
        if (lane == 0) {
#pragma unroll
            for (int i = 0; i < C::NSLOT + C::FOLD; ++i) mbar_init(bar(C::BAR_FULL + i), 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            fence_proxy_async();
        }
        __syncwarp();
        bar_start_arrive();
    } else if (warp == MMA_WARP) {
        if (lane == 0) {
            *abort_flag = (sbase & 1023u) == 0 ? 0 : 1;   // swizzled tiles need 1 KB alignment
#pragma unroll
            for (int i = C::BAR_Q; i < C::NUM_BARS; ++i) mbar_init(bar(i), i == C::BAR_Q ? SW : 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            fence_proxy_async();
            if (XCH) mbar_expect_tx(bar(C::BAR_X), (uint32_t)(my_tasks * S * MSG));
            if (!APART) { prefetch_map(&tm.kb); prefetch_map(&tm.vb); }
        }
        __syncwarp();
        bar_issue_arrive();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(C::TM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    } else if (tid < 2 * NR) {
        reinterpret_cast<float *>(smem + C::OFF_REF)[tid] = 0.f;
    }
    // which unit: when the clusters do not all fit at once they go out longest prefix first (every warp finds out by itself)
    if (__builtin_expect(!quiescent, 0)) griddep_wait();
    const int h = blockIdx.y - zt * p.Hkv;
    const int len_hi = (int)p.len_cap;
    if (__builtin_expect(args.ranked, 0)) b = rank_by_length(p, b, len_hi, lane);
    if (!len_first) P = p.cache_len[b];
    if (warp != PRODUCER_WARP) {
        tc_fence_before();
        bar_start_wait();
        tc_fence_after();
    }
    if (P < 0 || P > len_hi) {
        if (tid == 0 && rank == 0 && p.status) atomicOr(p.status, ORTHRUS_DEV_BAD_CACHE_LEN);
        P = P < 0 ? 0 : len_hi;
    }
    // the unit's halves: n_pre of 64 prefix keys, then the block's keys, shared out evenly
    const int n_pre = (P + HALF - 1) / HALF, n_all = n_pre + !APART;
    const int share = XCH ? (int)__umulhi((unsigned)n_all, args.inv_s32) : n_all, rest = n_all - share * S;
    auto first_half = [&](int k) { return XCH ? k * share + (int)((uint32_t)(k * rest) * args.inv_s >> 16) : k * share; };  // k * n_all / S
    const int a0 = first_half(rank), a1 = first_half(rank + 1);
    const int nh = a1 - a0, n_mine = max(0, min(nh, n_pre - a0));     // halves of this CTA, prefix halves among them
    const int n_tiles = (nh + 1) >> 1;
    // keys of half a (CTA-local): 0 past the end
    auto half_keys = [&](int a) { return a >= nh ? 0 : (a < n_mine ? min(HALF, P - (a0 + a) * HALF) : p.K); };

    // ring items in the order of their use: K0, K1, V0, K2, V1, ..., K(n-1), V(n-2), V(n-1); item i in slot i % NSLOT, or,
    // folded, K0, K1, V0 in slots 0 to 2 and V1 in slot 1
    const bool fold = C::FOLD && n_tiles == 2;
    auto slot_of = [&](int i) { return fold ? (i == 3 ? 1 : i) : i % C::NSLOT; };
    auto use_of = [&](int i) { return fold ? (int)(i == 3) : i / C::NSLOT; };     // earlier items of its slot
    const int off_p = fold ? C::OFF_RING : C::OFF_P;
    auto item_of_k = [&](int t) { return t == 0 ? 0 : 2 * t - 1; };
    auto item_of_v = [&](int t) { return min(2 * t + 2, 2 * n_tiles - 1); };
    const int n_slots = C::NSLOT + fold;
    const int row_base = (int)(((long long)(b / p.nb) * p.Hkv + h) * p.capacity);
    // half a (CTA-local) of a K or V tile, to its place in `slot`
    const uint64_t policy = policy_evict_first();
    auto load_half = [&](bool v, int a, int slot) {
        const uint32_t d = sbase + C::OFF_RING + slot * C::KV_BYTES + (a & 1) * (HALF * 128), fb = bar(C::BAR_FULL + slot);
#pragma unroll
        for (int s = 0; s < PANELS; ++s) {
            if (APART || a < n_mine || p.blk_in_cache)        // (rows behind the keys hold anything: masked, cleared in V)
                tma_load_2d(d + s * PANEL, v ? &tm.v : &tm.k, s * 64, row_base + (a < n_mine ? (a0 + a) * HALF : P), fb, policy);
            else                                              // rows >= K are out of bounds and arrive as zeros
                tma_load_4d(d + s * PANEL, v ? &tm.vb : &tm.kb, s * 64, h, 0, b, fb);
        }
    };
    constexpr int HALF_BYTES = PANELS * HALF * 128;

    if (warp < SW) {
        // ------------------------------------------------------------------ query rows
        const long long unit_row = (((long long)b * p.K + i0) * p.Hq + h * p.G) * HD;
        const uint4 *q = reinterpret_cast<const uint4 *>(static_cast<const __nv_bfloat16 *>(p.q) + unit_row);
        __nv_bfloat16 *out = static_cast<__nv_bfloat16 *>(p.out) + unit_row;
        // the block's own keys and values, where they are kept apart from the tiles
        const long long blk0 = APART && !p.blk_in_cache ? ((long long)b * p.K * p.Hkv + h) * HD : ((long long)row_base + P) * HD;
        const __nv_bfloat16 *bk = static_cast<const __nv_bfloat16 *>(APART && !p.blk_in_cache ? p.k_blk : p.k_cache) + blk0;
        const __nv_bfloat16 *bv = static_cast<const __nv_bfloat16 *>(APART && !p.blk_in_cache ? p.v_blk : p.v_cache) + blk0;
        const long long blk_stride = p.blk_in_cache ? HD : (long long)p.Hkv * HD;
        if (APART && tid < 4 * p.K) prefetch_l2((tid & 1 ? bv : bk) + (tid >> 2) * blk_stride + (tid >> 1 & 1) * 64);
        {
            // where this thread's chunks (16 bytes each) come from; rows past M are zero
            constexpr int QCH = HD / 8, QN = (NR * QCH + ST - 1) / ST;
            int q_src[QN];
#pragma unroll
            for (int u = 0; u < QN; ++u) {
                const int e = tid + u * ST, r = e / QCH;
                q_src[u] = r < M ? row_off(r) / 8 + e % QCH : -1;
                // (a line that the preceding kernel is writing may be asked into L2: that is where it is written)
                if (q_src[u] >= 0 && (lane & 7) == 0) prefetch_l2(q + q_src[u]);
            }
            if (quiescent) griddep_wait();
            griddep_launch();
            uint4 qv[QN];
#pragma unroll
            for (int u = 0; u < QN; ++u) qv[u] = q_src[u] >= 0 ? q[q_src[u]] : make_uint4(0, 0, 0, 0);
            const uint32_t q_dst = sbase + C::OFF_Q + sw_off(tid / QCH, tid % QCH, QPANEL);
#pragma unroll
            for (int u = 0; u < QN; ++u)                      // (ST / QCH rows on, a multiple of eight: the same swizzle)
                if (NR * QCH >= ST || tid < NR * QCH)
                    *reinterpret_cast<uint4 *>(smem + (q_dst - sbase) + u * (ST / QCH) * 128) = qv[u];
            static_assert(ST / QCH % 8 == 0 && (NR * QCH >= ST ? NR * QCH % ST == 0 : true), "query rows");
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(C::BAR_Q));

        // ------------------------------------------------------------------ softmax, thread = key
        const int wg = warp >> 2, wq = warp & 3, kt = tid & 127;
        const uint32_t lane_base = *tmem_slot + ((uint32_t)(wq * 32) << 16);
        const uint32_t TS = lane_base + C::tm_s(wg), TO = lane_base + C::tm_o(wg);
        unsigned char *p_buf = smem + off_p + wg * C::P_BYTES, *p_row = p_buf + kt * 128;
        float *ref = reinterpret_cast<float *>(smem + C::OFF_REF) + wg * NR;
        const float sc = p.scale_log2;
        constexpr int CH = NR < 32 ? NR : 32;                 // columns at a time
        constexpr int PP = C::P_PANELS, RP = NR / 2 / PP, LG = 32 / RP;   // row pairs of a panel, lane groups that share a warp's keys
        float2 l_run[PP];                                     // of row pair lane % RP of each panel over this warp's keys
#pragma unroll
        for (int x = 0; x < PP; ++x) l_run[x] = make_float2(0.f, 0.f);
#pragma unroll 1
        for (int t = wg, u = 0; t < n_tiles; t += 2, ++u) {
            const int a = 2 * t + (kt >> 6), j = kt & 63;     // this thread's half and key in it
            // rows below lo do not see the key (all, if the key does not exist)
            const int lo = j >= half_keys(a) ? NR : (!APART && a >= n_mine && p.causal ? (j - i0) * p.G : 0);
            const bool masks = __any_sync(0xffffffffu, lo > 0);
            if (u > 0) mbar_wait_warp_call(bar(C::BAR_PV + wg), (u - 1) & 1, abort_flag);   // P buffer and O^T at rest
            mbar_wait_warp_call(bar(C::BAR_S + wg), u & 1, abort_flag);
            tc_fence_after();
            bool exact = false;                               // the references are at or above the maxima of this tile
#pragma unroll 1
            for (;;) {
                uint32_t top = 0, low = 0x7f807f80;           // the largest and the smallest probabilities, as bit patterns
#pragma unroll 1
                for (int c0 = 0; c0 < NR; c0 += CH) {
                    uint32_t s[CH];
                    tmem_ld<CH>(TS + c0, s);
                    const float4 *rf = reinterpret_cast<const float4 *>(ref + c0);
                    float4 ra = rf[0], rb = rf[1];
                    tmem_ld_wait();
                    if (__builtin_expect(masks, 0)) {
#pragma unroll
                        for (int i = 0; i < CH; ++i) if (i < lo - c0) s[i] = 0xff800000u;
                    }
                    // (a masked score is -inf: its probability is 0.  The references of the next eight columns are
                    //  read ahead of the use of these.)
                    const float2 sc2 = make_float2(sc, sc);
                    unsigned char *row = p_row + (c0 >> 6) * PANEL;
                    const int x0 = (c0 >> 3 & 7) ^ (kt & 7);
#pragma unroll
                    for (int c = 0; c < CH; c += 8) {
                        float2 x[4];
                        x[0] = __ffma2_rn(make_float2(__uint_as_float(s[c]), __uint_as_float(s[c + 1])), sc2, make_float2(ra.x, ra.y));
                        x[1] = __ffma2_rn(make_float2(__uint_as_float(s[c + 2]), __uint_as_float(s[c + 3])), sc2, make_float2(ra.z, ra.w));
                        x[2] = __ffma2_rn(make_float2(__uint_as_float(s[c + 4]), __uint_as_float(s[c + 5])), sc2, make_float2(rb.x, rb.y));
                        x[3] = __ffma2_rn(make_float2(__uint_as_float(s[c + 6]), __uint_as_float(s[c + 7])), sc2, make_float2(rb.z, rb.w));
                        if (c + 8 < CH) { ra = rf[c / 4 + 2]; rb = rf[c / 4 + 3]; }
                        uint32_t w[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) w[i] = pack_bf16(ex2(x[i].x), ex2(x[i].y));
                        top = __vimax3_u16x2(__vimax3_u16x2(top, w[0], w[1]), w[2], w[3]);
                        low = __vimin3_u16x2(__vimin3_u16x2(low, w[0], w[1]), w[2], w[3]);
                        *reinterpret_cast<uint4 *>(row + ((x0 ^ (c >> 3)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
                    }
                }
                fence_proxy_async();
                tc_fence_before();
                // A reference of 0, with which a row starts, will do as long as no probability is out of all proportion and
                // (first tile; its first key is one that every row sees) no row has nothing but tiny ones.
                const bool off = max(top & 0xffffu, top >> 16) > P_HIGH || (u == 0 && kt == 0 && min(low & 0xffffu, low >> 16) < P_LOW);
                if (__builtin_expect(!bar_group_or(wg, off && !exact), 1)) break;
                // ------------------------------------------------ all references are set to the maxima of the tile, or, behind
                // the first, raised to them, and what the earlier tiles have added up is rescaled
                tc_fence_after();
                float *red = reinterpret_cast<float *>(p_buf);            // [4 warps][NR]: the probabilities are void
#pragma unroll 1
                for (int c = 0; c < NR; c += 8) {
                    uint32_t x[8];
                    tmem_ld<8>(TS + c, x);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 8; i += 4) {
                        float4 m;
                        m.x = warp_max(c + i < lo ? -INFINITY : __uint_as_float(x[i]));
                        m.y = warp_max(c + i + 1 < lo ? -INFINITY : __uint_as_float(x[i + 1]));
                        m.z = warp_max(c + i + 2 < lo ? -INFINITY : __uint_as_float(x[i + 2]));
                        m.w = warp_max(c + i + 3 < lo ? -INFINITY : __uint_as_float(x[i + 3]));
                        store_lane0(smem_u32(red + wq * NR + c + i), m, lane);
                    }
                }
                bar_group(wg);
                if (kt < NR) {
                    const float m = ceilf(fmaxf(fmaxf(red[kt], red[NR + kt]), fmaxf(red[2 * NR + kt], red[3 * NR + kt])) * sc);
                    const float m_old = -ref[kt], m_new = u > 0 ? fmaxf(m, m_old) : m;
                    red[kt] = u > 0 ? ex2(m_old - m_new) : 1.f;           // the factor of what row kt has summed up so far
                    // (a row that has met scores of -inf only: a reference so low that the first other score is out of proportion)
                    ref[kt] = m_new == -INFINITY ? FLT_MAX : -m_new;
                }
                bar_group(wg);
                if (u > 0) {
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
                    tc_fence_before();
                }
                bar_group(wg);                                // the factors have been read
                exact = true;
            }
            if (kt == 0) mbar_arrive(bar(C::BAR_P + wg));
            // while the product runs: the sums of this warp's 32 keys, lane = row pair
#pragma unroll
            for (int pn = 0; pn < PP; ++pn) {
                const int rp = lane % RP;
                float2 l0 = make_float2(0.f, 0.f), l1 = l0;
                const unsigned char *src = p_buf + pn * PANEL + wq * 32 * 128 + (rp & 3) * 4;
#pragma unroll 4
                for (int k = lane / RP; k < 32; k += 2 * LG) {
                    const uint32_t x = *reinterpret_cast<const uint32_t *>(src + k * 128 + (((rp >> 2) ^ (k & 7)) << 4));
                    const int k2 = k + LG;
                    const uint32_t y = *reinterpret_cast<const uint32_t *>(src + k2 * 128 + (((rp >> 2) ^ (k2 & 7)) << 4));
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
        float *t_w = t_l + 8 * NR, *t_ml = t_w + 2 * NR;                      // [2][NR] weights, [2][NR] reference and sum of the CTA
        static_assert((8 + 4) * NR * 4 <= C::END_Q - C::OFF_Q, "tables");
        if (n_tiles > 0) mbar_wait_warp_call(bar(C::BAR_QKALL), 0, abort_flag);
        else bar_pair();                                      // (no product reads them: every warp has written its own)
        if (lane < RP)
#pragma unroll
            for (int x = 0; x < PP; ++x) *reinterpret_cast<float2 *>(t_l + warp * NR + x * 64 + 2 * lane) = l_run[x];
        bar_pair();
        if (tid < NR) {
            const float *r = reinterpret_cast<const float *>(smem + C::OFF_REF);
            const float la = (t_l[tid] + t_l[NR + tid]) + (t_l[2 * NR + tid] + t_l[3 * NR + tid]);
            const float lb = (t_l[4 * NR + tid] + t_l[5 * NR + tid]) + (t_l[6 * NR + tid] + t_l[7 * NR + tid]);
            const float ma = la > 0.f ? -r[tid] : -INFINITY, mb = lb > 0.f ? -r[NR + tid] : -INFINITY;
            const float m = fmaxf(ma, mb);
            float wa = la > 0.f ? ex2(ma - m) : 0.f, wb = lb > 0.f ? ex2(mb - m) : 0.f;
            const float L = wa * la + wb * lb;
            if (!XCH) { const float inv = 1.f / L; wa *= inv; wb *= inv; }
            t_w[tid] = wa; t_w[NR + tid] = wb;
            t_ml[tid] = m; t_ml[NR + tid] = L;
        }
        // ------------------------------------------------------------------ read-out: lane = head column
        const int d = wq * 32 + lane;
        const bool reads = HD == 128 || wq * 32 < HD;
        constexpr int CW = NR / 2, CR = CW < 16 ? CW : 16;    // this warpgroup's rows, how many at a time
        // where the messages of rows c..c+CR-1 go (0: nowhere), and the barrier there
        uint32_t to[CR / 4], to_bar[CR / 4];
        auto addresses = [&](int c) {
#pragma unroll
            for (int i = 0; i < CR / 4; ++i) {
                const int g = (c >> 2) + i, task = g * (HD / 32) + wq;
                const int n = (int)((uint32_t)task * args.inv_s >> 16), owner = task - n * S;
                const uint32_t base = map_to_rank(sbase, owner);
                to[i] = g < n4 ? base + (n * S + rank) * MSG + lane * 16 : 0;
                to_bar[i] = base + C::OFF_BAR + C::BAR_X * 8;
            }
        };
        if constexpr (XCH) addresses(wg * CW);
        if (n_tiles > 0) mbar_wait_warp_call(bar(C::BAR_ALL), 0, abort_flag);
        if constexpr (XCH) cluster_arrive_relaxed();                  // the ring is idle
        bar_pair();
        tc_fence_after();
        if constexpr (XCH) { if (!reads) cluster_wait(); }
        if (reads) {
#pragma unroll 1
            for (int c = wg * CW; c < (wg + 1) * CW; c += CR) {
                uint32_t oa[CR], ob[CR];
                if (n_tiles > 0) tmem_ld<CR>(lane_base + C::tm_o(0) + c, oa);
                if (n_tiles > 1) tmem_ld<CR>(lane_base + C::tm_o(1) + c, ob);
                tmem_ld_wait();
                float x[CR];
#pragma unroll
                for (int i = 0; i < CR; ++i) x[i] = 0.f;      // (a CTA without keys contributes zeros)
                if (n_tiles > 0) {
#pragma unroll
                    for (int i = 0; i < CR; i += 4) {
                        const float4 w = *reinterpret_cast<const float4 *>(t_w + c + i);
                        x[i] = w.x * __uint_as_float(oa[i]); x[i + 1] = w.y * __uint_as_float(oa[i + 1]);
                        x[i + 2] = w.z * __uint_as_float(oa[i + 2]); x[i + 3] = w.w * __uint_as_float(oa[i + 3]);
                    }
                }
                if (n_tiles > 1) {
#pragma unroll
                    for (int i = 0; i < CR; i += 4) {
                        const float4 w = *reinterpret_cast<const float4 *>(t_w + NR + c + i);
                        x[i] = fmaf(w.x, __uint_as_float(ob[i]), x[i]); x[i + 1] = fmaf(w.y, __uint_as_float(ob[i + 1]), x[i + 1]);
                        x[i + 2] = fmaf(w.z, __uint_as_float(ob[i + 2]), x[i + 2]); x[i + 3] = fmaf(w.w, __uint_as_float(ob[i + 3]), x[i + 3]);
                    }
                }
                if constexpr (XCH) {
                    if (c == wg * CW) cluster_wait();
#pragma unroll
                    for (int i = 0; i < CR / 4; ++i)
                        if (to[i]) {                          // (the same for the whole warp)
                            st_async_if(true, to[i], make_float4(x[4 * i], x[4 * i + 1], x[4 * i + 2], x[4 * i + 3]), to_bar[i]);
                            st_async_if(lane < 2, to[i] + 512, *reinterpret_cast<const float4 *>(t_ml + (lane & 1) * NR + c + 4 * i), to_bar[i]);
                        }
                    if (CR < CW) addresses(c + CR);
                } else {
#pragma unroll
                    for (int i = 0; i < CR; ++i)
                        if (c + i < M) out[row_off(c + i) + d] = __float2bfloat16_rn(x[i]);
                }
            }
        }
        tc_fence_before();
        bar_tmem_arrive();
        if (XCH && warp < my_tasks) {
            // ---------------------------------------------------------------- merge
            // where this lane's results of task n go: four rows, one column (-1: no such row)
            int at[4];
            auto places = [&](int n) {
                const int task = n * S + rank, g = task / (HD / 32), col = task % (HD / 32) * 32 + lane;
#pragma unroll
                for (int k = 0; k < 4; ++k) at[k] = 4 * g + k < M ? row_off(4 * g + k) + col : -1;
            };
            float *wt = reinterpret_cast<float *>(smem + C::OFF_XW) + warp * ((MAX_CLUSTER + 1) * 4);
            bool got = true;
            auto wait_for_messages = [&]() {
                // (the wait outlasts every other one: a CTA of the cluster that gave one up sends all the same)
                got = __all_sync(0xffffffffu, mbar_wait_long(bar(C::BAR_X), 0));
                if (!got && lane == 0 && p.status) atomicOr(p.status, ORTHRUS_DEV_WAIT_TIMEOUT);
            };
            // (the places of a task are worked out ahead of the wait, or behind the stores of the one before)
            if constexpr (!APART) { places(warp); wait_for_messages(); }
#pragma unroll 1
            for (int n = warp; n < my_tasks && got; n += SW) {
                BlockPart bp;
                if constexpr (APART) {
                    places(n);
                    const int g = (n * S + rank) / (HD / 32), row = min(4 * g + (lane >> 2 & 3), M - 1);
                    bp = block_part(reinterpret_cast<const __nv_bfloat16 *>(q) + row_off(row), bk, bv + (n * S + rank) % (HD / 32) * 32,
                                    blk_stride, p.K, p.causal ? i0 + (int)((uint32_t)row * args.inv_g >> 16) + 1 : p.K, p.scale_log2, lane);
                    if (lane < 16) {
                        float *o = reinterpret_cast<float *>(smem + C::OFF_XB) + warp * 128 + (lane >> 2) * 32 + (lane & 3) * 2;
#pragma unroll
                        for (int t = 0; t < 4; ++t) *reinterpret_cast<float2 *>(o + t * 8) = make_float2(bp.o[t][0], bp.o[t][1]);
                    }
                }
                if (APART && n == warp) {
                    wait_for_messages();
                    if (!got) break;
                }
                const unsigned char *msg = smem + n * S * MSG;
                // weights: lane = (row, CTA and CTA + 8)
                const int r = lane >> 3, j0 = lane & 7, j1 = j0 + 8;
                const float *ml = reinterpret_cast<const float *>(msg + 512) + r;
                float m0 = 0.f, l0 = 0.f, m1 = 0.f, l1 = 0.f;
                if (j0 < S) { m0 = ml[j0 * (MSG / 4)]; l0 = ml[j0 * (MSG / 4) + 4]; }
                if (j1 < S) { m1 = ml[j1 * (MSG / 4)]; l1 = ml[j1 * (MSG / 4) + 4]; }
                float m = fmaxf(l0 > 0.f ? m0 : -INFINITY, l1 > 0.f ? m1 : -INFINITY);
                float mb = 0.f, lb = 0.f;                     // of this lane's row from the block's own keys
                if constexpr (APART) {
                    mb = __shfl_sync(0xffffffffu, bp.m, 4 * r); lb = __shfl_sync(0xffffffffu, bp.l, 4 * r);
                    m = fmaxf(m, lb > 0.f ? mb : -INFINITY);
                }
#pragma unroll
                for (int off = 4; off; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
                // (a sum that is not a number has no order: its row is void with it)
                const float w0 = l0 > 0.f ? ex2(m0 - m) : l0, w1 = l1 > 0.f ? ex2(m1 - m) : l1;
                float L = fmaf(w0, l0, w1 * l1);
#pragma unroll
                for (int off = 4; off; off >>= 1) L += __shfl_xor_sync(0xffffffffu, L, off);
                const float wb = lb > 0.f ? ex2(mb - m) : lb;
                if constexpr (APART) L = fmaf(wb, lb, L);
                const float inv = L == 0.f ? 0.f : __frcp_rn(L);
                wt[j0 * 4 + r] = w0 * inv;
                wt[j1 * 4 + r] = w1 * inv;
                if (APART && j0 == 0) wt[MAX_CLUSTER * 4 + r] = wb * inv;
                __syncwarp();
                float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
                if constexpr (APART) {
                    const float4 w = *reinterpret_cast<const float4 *>(wt + MAX_CLUSTER * 4);
                    const float *o = reinterpret_cast<const float *>(smem + C::OFF_XB) + warp * 128 + lane;
                    acc = make_float4(w.x * o[0], w.y * o[32], w.z * o[64], w.w * o[96]);
                }
#pragma unroll 4
                for (int j = 0; j < S; ++j) {
                    const float4 v = *reinterpret_cast<const float4 *>(msg + j * MSG + lane * 16);
                    const float4 w = *reinterpret_cast<const float4 *>(wt + j * 4);
                    acc.x = fmaf(w.x, v.x, acc.x); acc.y = fmaf(w.y, v.y, acc.y);
                    acc.z = fmaf(w.z, v.z, acc.z); acc.w = fmaf(w.w, v.w, acc.w);
                }
                const float y[4] = {acc.x, acc.y, acc.z, acc.w};
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (at[k] >= 0) out[at[k]] = __float2bfloat16_rn(y[k]);
                if (!APART && n + SW < my_tasks) places(n + SW);
                __syncwarp();
            }
        }
    } else if (warp == PRODUCER_WARP) {
        // ------------------------------------------------------------------ producer
        bar_issue_wait();                                     // the other barriers are set up
        if (lane == 0) {
            const int n_items = 2 * n_tiles;
            bool ok = (sbase & 1023u) == 0;
            // Two rounds.  The first only if the caller promised that the preceding kernel writes no cache row below
            // cache_len: the halves that are made of such rows, into the slots, and the item behind them as far as L2.
            // (The block's own half, where its item is one of those, is left to the MMA warp, which waits for that kernel at once.)
            uint32_t loaded = 0;                              // the first items: which are under way
            int n = 0;
#pragma unroll 1
            for (bool ahead = quiescent; ; ++n) {
                if (ahead && (n >= n_items || n > n_slots)) {
                    griddep_wait();
                    ahead = false; n = 0;
                }
                if (!ahead && (n >= n_items || !ok)) break;
                const bool v = n == n_items - 1 || (n > 0 && (n & 1) == 0);
                const int t = v ? (n == n_items - 1 ? n_tiles - 1 : n / 2 - 1) : (n + 1) / 2;
                const int slot = slot_of(n);
                int last = min(2 * t + 2, nh);                // halves [2 t, last)
                if (ahead) {
                    if (n == n_slots) {                       // (the rows of a tile are contiguous)
                        if (fold && last <= n_mine)
                            prefetch_l2_bulk(static_cast<const __nv_bfloat16 *>(v ? p.v_cache : p.k_cache) + (row_base + (long long)(a0 + 2 * t) * HALF) * HD,
                                             (uint32_t)(min((last - 2 * t) * HALF, P - (a0 + 2 * t) * HALF) * HD * 2));
                        continue;
                    }
                    loaded |= 1u << n;
                    if (2 * t >= n_mine) continue;
                    mbar_expect_tx(bar(C::BAR_FULL + slot), (uint32_t)((last - 2 * t) * HALF_BYTES));
                    last = min(last, n_mine);
                } else {
                    if (n < 32 && (loaded >> n & 1)) continue;
                    if (use_of(n) > 0) {
                        // the slot is free once the product that read it has retired (which its tile's
                        // softmax, or the accumulator's next user, is told anyway)
                        const int i = fold ? 1 : n - C::NSLOT;                // the slot's item before this one
                        const bool iv = i > 0 && (i & 1) == 0;                // (never the last item)
                        // (Item 3 is K2, so that with four slots the barrier of K0 can be two phases on before it is looked
                        // at here.  K1's cannot, and its scores come behind those of K0.)
                        const int it = iv ? i / 2 - 1 : C::NSLOT == 4 && i == 0 ? 1 : (i + 1) / 2;
                        ok = mbar_wait_call(bar((iv ? C::BAR_PV : C::BAR_S) + (it & 1)), (it >> 1) & 1, abort_flag);
                        if (!ok) continue;
                    }
                    if (n < 32) loaded |= 1u << n;
                    mbar_expect_tx(bar(C::BAR_FULL + slot), (uint32_t)((last - 2 * t) * HALF_BYTES));
                }
#pragma unroll 1
                for (int a = 2 * t; a < last; ++a) load_half(v, a, slot);
            }
            if (__builtin_expect(*abort_flag, 0)) {
                // Copies in flight land before the CTA ends: the last of each slot.  (`ok` false: item n - 1 was
                // not asked for, later ones only if they were early.)
                const int end = ok ? n : max(n - 1, 0);
#pragma unroll 1
                for (int i = fold ? 0 : max(0, end - C::NSLOT); i < max(end, n_slots); ++i) {
                    int dummy = 0;
                    if (fold && i == 1 && (loaded >> 3 & 1)) continue;
                    if (i < 32 ? loaded >> i & 1 : i < end) mbar_wait_call(bar(C::BAR_FULL + slot_of(i)), use_of(i) & 1, &dummy);
                }
            }
        }
        __syncwarp();
        if constexpr (XCH) { cluster_arrive_relaxed(); cluster_wait(); }
    } else {
        // ------------------------------------------------------------------ MMA issue
        constexpr uint32_t IDESC_QK = keys_idesc(NR, 0, 0);   // A = K tile, B = query rows, both K-major
        constexpr uint32_t IDESC_PV = keys_idesc(NR, 1, 1);   // A = V tile, B = P, both MN-major
        const uint32_t tmem = *tmem_slot;
        bool ok = __all_sync(0xffffffffu, !*abort_flag);
        if (!APART && quiescent && nh > n_mine) {
            // the block's own half of the last tile, where the producer's first round has left it out
            griddep_wait();
            if (ok && elect_one()) {
                const int bt = n_tiles - 1;
#pragma unroll 1
                for (int v = 0; v < 2; ++v) {
                    const int i = v ? item_of_v(bt) : item_of_k(bt);
                    if (i >= n_slots) continue;
                    if (2 * bt >= n_mine) mbar_expect_tx(bar(C::BAR_FULL + slot_of(i)), HALF_BYTES);
                    load_half(v, nh - 1, slot_of(i));
                }
            }
            __syncwarp();
        }
        // step t: the scores of tile t, then, while its softmax runs, the product of tile t - 1
        int scored = 0;
#pragma unroll 1
        for (int t = 0; t <= n_tiles && n_tiles > 0 && ok; ++t) {
            if (t < n_tiles && t >= scored) {
                const int i = item_of_k(t), slot = slot_of(i);
                ok = mbar_wait_warp_call(bar(C::BAR_FULL + slot), use_of(i) & 1, abort_flag);
                if (ok && t == 0) ok = mbar_wait_warp_call(bar(C::BAR_Q), 0, abort_flag);
                if (!ok) break;
                // (the second tile's scores with the first one's, if its keys are there)
                scored = t + 1;
                if (t == 0 && n_tiles > 1 && __all_sync(0xffffffffu, mbar_test(bar(C::BAR_FULL + slot_of(1)), 0))) scored = 2;
                tc_fence_after();
                if (elect_one()) {
                    const uint64_t qd = make_desc(sbase + C::OFF_Q, 16, 1024);
#pragma unroll 1
                    for (int x = t; x < scored; ++x) {
                        const uint64_t kd = make_desc(sbase + C::OFF_RING + slot_of(item_of_k(x)) * C::KV_BYTES, 16, 1024);
                        const uint32_t dst = tmem + C::tm_s(x & 1);
#pragma unroll
                        for (int kk = 0; kk < HD / 16; ++kk)
                            umma_ss(dst, kd + (((kk >> 2) * PANEL + (kk & 3) * 32) >> 4),
                                    qd + (((kk >> 2) * QPANEL + (kk & 3) * 32) >> 4), IDESC_QK, kk > 0);
                        umma_commit(bar(C::BAR_S + (x & 1)));
                        if (x == n_tiles - 1) umma_commit(bar(C::BAR_QKALL));
                    }
                }
                __syncwarp();
            }
            if (t > 0) {
                const int pt = t - 1, i = item_of_v(pt), slot = slot_of(i), w = pt & 1;
                ok = mbar_wait_warp_call(bar(C::BAR_FULL + slot), use_of(i) & 1, abort_flag);
                if (!ok) break;
                // only the 16-key groups that hold keys are multiplied; V rows behind the keys in the last
                // group may hold anything where they come from the cache, and 0 * NaN would poison the product
                const int k0 = half_keys(2 * pt), k1 = half_keys(2 * pt + 1);
                if (__builtin_expect((k0 | k1) & 15, 0)) {
#pragma unroll 1
                    for (int a = 0; a < 2; ++a) {
                        const int n = a ? k1 : k0, pad = -n & 15;
                        if (pad && (2 * pt + a < n_mine || p.blk_in_cache)) {
                            unsigned char *vt = smem + C::OFF_RING + slot * C::KV_BYTES + a * (HALF * 128);
#pragma unroll 1
                            for (int e = lane; e < pad * (HD / 8); e += 32)
                                *reinterpret_cast<uint4 *>(vt + sw_off(n + e / (HD / 8), e % (HD / 8), PANEL)) = make_uint4(0, 0, 0, 0);
                        }
                    }
                    fence_proxy_async();
                    __syncwarp();
                }
                ok = mbar_wait_warp_call(bar(C::BAR_P + w), (pt >> 1) & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                if (elect_one()) {
                    const uint64_t vd = make_desc(sbase + C::OFF_RING + slot * C::KV_BYTES, PANEL, 1024);
                    const uint64_t pd = make_desc(sbase + off_p + w * C::P_BYTES, PANEL, 1024);
                    const uint32_t dst = tmem + C::tm_o(w);
                    const int g0 = (k0 + 15) >> 4, g1 = (k1 + 15) >> 4;
#pragma unroll
                    for (int g = 0; g < 8; ++g)
                        if (g < 4 ? g < g0 : g - 4 < g1)
                            // (head_dim 64: lanes 64-127 take another panel and are not read)
                            umma_ss(dst, vd + (g * 2048 >> 4), pd + (g * 2048 >> 4), IDESC_PV, pt > 1 || g > 0);
                    if (pt == n_tiles - 1) umma_commit(bar(C::BAR_ALL));
                    umma_commit(bar(C::BAR_PV + w));
                }
                __syncwarp();
            }
        }
        if (ok && n_tiles > 0) ok = mbar_wait_warp_call(bar(C::BAR_ALL), 0, abort_flag);
        if (__builtin_expect(!ok, 0)) {                       // the MMAs in flight end before TMEM is freed
            if (elect_one()) umma_commit(bar(C::BAR_DRAIN));
            __syncwarp();
            int dummy = 0;
            mbar_wait_warp_call(bar(C::BAR_DRAIN), 0, &dummy);
        }
        if constexpr (XCH) cluster_arrive_relaxed();
        bar_tmem_wait();                                      // the softmax warps have read their TMEM
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::TM_COLS) : "memory");
        if (lane == 0 && *abort_flag && p.status) atomicOr(p.status, ORTHRUS_DEV_WAIT_TIMEOUT);
        if constexpr (XCH) cluster_wait();
    }
}

template <int HD, int NR, bool XCH>
__global__ void __launch_bounds__(NTHREADS, KeysShape<HD, NR>::CTAS)
attend_keys_kernel(const AttnParams p, const __grid_constant__ KeysMaps tm, const KeysArgs args)
{
    attend_keys<HD, NR, XCH, false>(p, tm, args);
}
template <int HD, int NR>
__global__ void __launch_bounds__(NTHREADS, KeysShape<HD, NR>::CTAS)
apart_attend_keys_kernel(const AttnParams p, const __grid_constant__ KeysMaps tm, const KeysArgs args)
{
    attend_keys<HD, NR, true, true>(p, tm, args);
}
template <int HD, int NR, bool XCH, bool APART> constexpr auto keys_kernel()
{
    if constexpr (APART) return apart_attend_keys_kernel<HD, NR>;
    else return attend_keys_kernel<HD, NR, XCH>;
}

// function attributes belong to a device: set them once on each device that launches
template <int HD, int NR, bool XCH, bool APART> cudaError_t configure(int *dev)
{
    constexpr int kMaxDevices = 64;
    static std::mutex mu;
    static bool configured[kMaxDevices] = {};
    cudaError_t e = cudaGetDevice(dev);
    if (e != cudaSuccess) return e;
    if (*dev < 0 || *dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (!configured[*dev]) {
        auto kern = keys_kernel<HD, NR, XCH, APART>();
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, KeysShape<HD, NR>::SMEM_BYTES);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
        configured[*dev] = true;
    }
    return cudaSuccess;
}

// CTAs per unit: the cheapest by this count (in 0.1 us) among the sizes at which all units are resident together.
//  - Tiles follow one another.  Two cost little more than one (a warpgroup each; at head_dim 128 both tiles' keys and the
//    first one's values wait in shared memory), from the third on each waits for its slot of the ring: 8 units
//    of 4 rows, 500 keys, 1, 2, 3 and 5 tiles a CTA 3.5, 4.4, 5.9 and 8.6 us; d = 64, 32 rows, 2 units of 500 keys 3.5, 4.2, 5.1, 7.0.
//  - The merge: a warp takes some 0.4 us for a task, and the CTAs share the tasks (64 rows, 8 units of 300 keys, one tile
//    each: 7.2 us at 2 CTAs, 6.2 at 3, 5.7 at 4 to 6).  At 64 rows that is worth CTAs without a key of their own (one unit of 100
//    keys 6.2 us at 3, 5.1 at 8).
//  - From 32 rows on there is much to tell, and CTAs that share an SM share the way to the others: once the clusters of a call do not all
//    find SMs of their own, it takes 1 to 1.5 us more at 33 to 64 rows, 0.5 at 32.  A cluster stays within a GPC, so that this depends on the size of the
//    cluster (a B200 has SMs for 45, 33, 26, 22, 15, 15, 15, 11 and 7 clusters of 3 to 11 CTAs and for 7 of 12 to 16; us a call, 300 keys:
//    clusters of 3, 36 units 6.7 and 48 8.4; of 4, 28 6.3 and 36 8.0; of 5, 24 6.5 and 28 7.6; of 6, 20 6.6 and 24 8.1; of 7, 14
//    6.3 and 16 7.6).  A line at five ninths of the SMs, which stood here before, kept 28 units of 200 keys at 2 CTAs: 7.3 us, 6.3 at 4.
//  - Once they do not fit beside one another at all, the next call starts late (32 units of 1000 keys, 4 rows 5.8 us at 5 CTAs, 6.3
//    at 8), the more so where clusters fill the GPU to the last place (56 units of 32 rows, 3000 keys 17.1 us at 4, 19.9 at 5).
// Of sizes that cost the same the largest up to 8 (lengths are often below the bound the plan is
// made for, and then the larger size has fewer tiles) and beyond where a CTA has three tiles or more, of which the last is only half
// with the larger size (8 units of 64 rows, 4096 keys 10.5 us at 11, 9.8 at 16; but 15 of 4000 keys, eight halves a CTA either way, 11.3 at 8, 11.7 at 9);
// the smallest where a CTA has one tile in any case and half the SMs are taken (16 units of 64 rows, 300 keys 5.8 us at 4, 6.3 at 6; but 8 of 4 rows 3.6 at 3, 3.4 at 6).  A second wave of clusters costs more than any
// split gains (32 units of 64 rows, 1000 keys 9.1 us at 8, 12.8 at 9; 22 of 4000 keys 13.7 at 10, 20.7 at 11; 72 units of 32 rows,
// 1000 keys 10.4 at 3, 17.4 at 4).
// Against sweeps of 1 to 92 units, 64 to 8000 keys and all sizes, the choice is 0.5 to 0.6 % above the best size in the mean at
// 4, 32 and 64 rows and both head sizes, where the count of residents by half-sized clusters and the line at five ninths took 3.8 to 4.9 %.
// Where it misses most: 16 or 17 units of 24 to 26 halves, which get 13 CTAs and are 5 to 12 % faster with 8.
struct Pick { int S, cost; };
template <int HD, int NR> Pick choose_splits(int units, int halves, int rows)
{
    constexpr bool FULL = HD == 128 && NR == 64;
    constexpr int TILE2 = HD == 128 ? 9 : 6, TILE3 = HD == 128 ? 16 : NR == 128 ? 15 : 10;
    constexpr int ALONE = NR >= 64 ? 10 : 6, MERGE = FULL ? 10 : 7;
    const int tasks = FULL ? (rows + 3) / 4 * (HD / 32) : NR / 4 * (HD / 32);
    const int shared = FULL ? (rows > 48 ? 15 : 11) : NR == 64 ? 8 : NR == 32 ? 5 : 0;        // CTAs of a call share SMs
    constexpr int PER_SM = KeysShape<HD, NR>::CTAS;
    const int sms = num_sms();
    int best = 1, best_cost = 1 << 30;
    for (int S = 1; S <= MAX_CLUSTER && S <= (FULL ? max(halves, 8) : halves); ++S) {
        const int chunk = (halves + S - 1) / S, tiles = (chunk + 1) / 2, ctas = units * S;
        int cost = (tiles > 1 ? TILE2 : 0) + (tiles > 2 ? min(tiles - 2, 1 << 20) * TILE3 : 0);
        cost += S == 1 ? ALONE : MERGE + 4 * ((tasks + 8 * S - 1) / (8 * S));
        if (shared && S > (NR == 32 ? 2 : 1) && units > clusters_resident(S, 1)) cost += shared;
        if (S > 1 && ctas > sms) cost += FULL ? 3 + 4 * (ctas - sms) / sms : 5 + min(5 * (ctas - sms) / sms, 10);
        // of two that cost the same
        const bool larger = S <= 8 ? tiles > 1 || 2 * ctas <= sms : HD == 128 && tiles > 2 && chunk < (halves + best - 1) / best;
        if (larger ? cost > best_cost : cost >= best_cost) continue;
        if (S > 1 && (units > clusters_resident(S, PER_SM) || (S > 2 && 16 * ctas > 15 * PER_SM * sms))) continue;
        best = S;
        best_cost = cost;
    }
    return {best, best_cost};
}

template <int HD, int NR, bool XCH = true, bool APART = false>
cudaError_t launch_shape(const AttnParams &p, const KeysMaps &tm, int flags, cudaStream_t st)
{
    if constexpr (XCH && !APART) {
        if (p.n_splits == 1) return launch_shape<HD, NR, false>(p, tm, flags, st);
        if constexpr (HD == 128 && NR == 64)
            if (p.apart) return launch_shape<HD, NR, true, true>(p, tm, flags, st);
    }
    using C = KeysShape<HD, NR>;
    auto kern = keys_kernel<HD, NR, XCH, APART>();
    int dev = 0;
    cudaError_t e = configure<HD, NR, XCH, APART>(&dev);
    if (e != cudaSuccess) return e;
    const int S = p.n_splits, units = p.B * p.Hkv, kb = keys_kb_rows(HD, p.G, p.K), tiles = (p.K + kb - 1) / kb;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(S, p.Hkv * tiles, p.B);
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
    args.inv_s = (65536u + S - 1) / S;
    args.inv_s32 = (uint32_t)(((1ull << 32) + S - 1) / S);
    args.kb_rows = kb;
    args.tiles = tiles;
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
    return M <= 16 ? 16 : M <= 32 ? 32 : M <= 64 || (M <= 128 && G <= 64) ? 64 : 0;
}

// Block positions of a query tile.  At head_dim 128 up to 128 rows are cut into tiles of at most 64, as equal as can be,
// which read the same keys (from L2, but for the first).
int keys_kb_rows(int d, int G, int K)
{
    if (d == 64 || G * K <= 64) return tc_kb_rows(G, K);
    const int most = 64 / G, tiles = (K + most - 1) / most;
    return (K + tiles - 1) / tiles;
}

// `apart`: the block's own keys are left out of the tiles.  That takes a merging warp 1.4 us for each of its tasks and sixteen keys, a
// third of it while it would wait; worth it where those keys alone are a tile more for the longest CTA, no warp has two tasks and
// every CTA an SM (64 rows, 4096 keys: 8 units in sixteen CTAs 10.5 us a call, 9.7 so, 4 units 8.2 and 7.4; but 32 units of 2000 keys in eight
// 11.8 and 13.0, blocks of 32 with 4 units of 128 rows 10.0 and 10.7).
int keys_splits(int d, int G, int K, int units, int max_len, bool *apart)
{
    // the layers of a pass ask the same question: the last answer of this thread is kept
    struct Key { int dev, d, nr, rows, units, halves, S; bool few, apart; };
    static thread_local Key last = {-1, 0, 0, 0, 0, 0, 0, false, false};
    Key k = {-1, d, keys_rows(d, G, K), keys_kb_rows(d, G, K) * G, units, (max_len + HALF - 1) / HALF + 1, 0, K <= 16, false};   // (prefix and block in halves of their own)
    if (cudaGetDevice(&k.dev) != cudaSuccess) { (void)cudaGetLastError(); k.dev = -2; }
    if (!(k.dev == last.dev && k.d == last.d && k.nr == last.nr && k.rows == last.rows && k.units == last.units && k.halves == last.halves &&
          k.few == last.few)) {
        switch (k.nr) {
        case 16: k.S = (d == 64 ? choose_splits<64, 16>(units, k.halves, k.rows) : choose_splits<128, 16>(units, k.halves, k.rows)).S; break;
        case 32: k.S = (d == 64 ? choose_splits<64, 32>(units, k.halves, k.rows) : choose_splits<128, 32>(units, k.halves, k.rows)).S; break;
        case 64:
            if (d == 64) {
                k.S = choose_splits<64, 64>(units, k.halves, k.rows).S;
            } else {
                const Pick with = choose_splits<128, 64>(units, k.halves, k.rows), without = choose_splits<128, 64>(units, k.halves - 1, k.rows);
                k.apart = k.few && without.S >= 8 && without.S * units <= num_sms() && without.cost + 11 < with.cost;      // (64 tasks)
                k.S = k.apart ? without.S : with.S;
            }
            break;
        default: k.S = choose_splits<64, 128>(units, k.halves, k.rows).S;
        }
        last = k;
    }
    *apart = last.apart;
    return last.S;
}

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
