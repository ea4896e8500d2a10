// Split-KV flash-decode block attention on the 5th-generation tensor cores
// (tcgen05.mma with TMEM accumulators), bf16, head_dim 128, both views.
//
// Work decomposition.  A unit is one (sequence, KV head); its query tile is the GQA
// group times the block width, M = G*K logical rows (row r = i*G + g), padded to the
// 128 rows of the MMA.  The S CTAs of a thread-block cluster share one unit: the unit's
// 64-position prefix tiles plus the tile of block keys are shared out evenly.  Clusters are handed out longest sequence first, so that a ragged
// batch packs well onto the SMs.
//
// One CTA (192 threads, 112 KB of shared memory, 256 TMEM columns: two fit on an SM).
//   warps 0-3  softmax.  Thread r owns TMEM lane r = query row r: it reads the 64 scores
//              of a tile, keeps the running max / sum of the online softmax, and writes
//              the bf16 probabilities back into TMEM over the scores, where the P.V
//              product reads them as its A operand.
//   warp 4     producer: one lane issues every TMA load (Q tile, K and V tiles of the
//              cache, the block K/V tile) into a ring of five 16 KB slots, in the order
//              the MMAs consume them.
//   warp 5     TMEM allocation and MMA issue: S = Q.K^T into one of two score buffers
//              (so that QK(t+1) runs under softmax(t)), then O += P.V.  This chain sets the pace
//              of a lone CTA, 1450 cycles per tile: 480 to issue the eight MMAs of QK, 250 for the
//              four of P.V, the rest waits and fences.  (Behind a test of the lane index instead
//              of elect.sync, the descriptors built in the loop: 660, 640 and 2020 per tile.)
// (Units of few rows run on attend_keys.cu; api.cu, keys_usable and wide_better.)
// The output accumulator O stays in TMEM for the whole CTA.  A row's reference starts at 0 and is left alone as long as no
// probability exceeds 2^40 and, in the first tile that shows the row a key, the largest is not below 2^-60: floating-point
// numbers keep their relative precision whatever the reference, so that no tile pays for its row maxima.  Otherwise the
// owner threads set the reference to the tile's maximum, or raise it, and rescale their O rows in TMEM, and the tile takes its
// exponentials twice (8 units of 128 rows, 4000 keys, without the promise below, all scores about +60 or -60: 12.3 us a call instead of
// 11.6, 32 of 1000 keys 13.9 instead of 13.0; 13.1 and 14.2 in a kernel that took every tile's maxima).  The result is the
// exact softmax because the same shift is used for the numerator and the denominator.
//
// Merge of the S partial results of a unit, inside the kernel (there is no second launch), through distributed shared
// memory: a cluster barrier without a release (every query tile and ring are idle), then each row's thread sends the other
// CTAs their columns of its row by stores that the destination's mbarrier counts, and sums up its own columns once its count is
// there.  Nothing goes through the workspace.
//
// The kernel's code matters at its two ends, which every CTA runs through once: an SM's instruction cache holds 32 KB, a taken branch
// costs some 25 cycles, a chain of address arithmetic for each message as much again.  So there is an instance for each size of
// cluster that plans come to, whose merge is straight-line code for that size (merge_fixed); other sizes, and the two-tile CTA, go through
// loops (merge).  Us a call, with one merge for all sizes in loops and now: 8 units of 64 rows and 300 keys 6.4 and 5.3, of 1000
// 7.4 and 6.6, of 4096 11.0 and 10.0; one unit of 2000 keys 8.5 and 7.0; 128 rows, 8 units of 500 keys 7.3 and 6.7.
// Before that the merge went through two cluster barriers with a release, and at clusters of 16 through L2: 5.8, 7.0, 10.2, 6.6 and 7.6.
// (16 is where L2 was the better way still: one unit of 64 rows 6.6 against 7.0, 8 of 128 rows and 4096 keys 12.7 against 13.2; api.cu
// has fewer of them.)
//
// Programmatic dependent launch.  The kernel waits for the preceding kernel of the
// stream (griddepcontrol.wait) before it reads anything that kernel may have written,
// and then lets its own successor start.  With ORTHRUS_LAYER_CACHE_QUIESCENT the prefix
// K/V tiles are requested before that wait, so the next call's loads are in flight
// while this call is still computing.
//
// Every mbarrier wait is bounded: on expiry the CTA records ORTHRUS_DEV_WAIT_TIMEOUT in
// the status word, drains the copies it armed, still takes part in the cluster barriers,
// frees its TMEM and returns.
#include <cuda.h>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <unordered_map>
#include "common.cuh"
#include "tc_ptx.cuh"

namespace orthrus {
namespace {

constexpr int HD = 128;                  // head_dim
constexpr int MROWS = 128;               // MMA M
constexpr int TN = 64;                   // key positions per tile
constexpr int QSUB_BYTES = MROWS * 128;  // a [128 rows][64 cols] bf16 sub-tile of Q
constexpr int SUB_BYTES = TN * 128;      // a [64 rows][64 cols] bf16 sub-tile of K or V
constexpr int SLOT_BYTES = 2 * SUB_BYTES;
constexpr int MAX_BARS = 40;

// Two shapes of CTA.  NT = 1: one 128-row query tile, 192 threads, 112 KB of shared memory and
// 256 TMEM columns, so that two CTAs share an SM.  NT = 2 (units wider than 128 rows): two
// 128-row query tiles of the same unit share ONE ring of K/V tiles, so every cache byte is
// loaded once for both; 320 threads (two softmax warpgroups), 224 KB of shared memory, all
// 512 TMEM columns: one CTA per SM, with a ring twice as deep.
template <int NT> struct Shape {
    static constexpr int NSLOT = NT == 1 ? 5 : 10;             // ring slots, one K or V tile each
    // warps: 4 softmax warps per query tile, the producer, one MMA-issuing warp per query tile
    // (a thread is held for about fifty cycles per tcgen05.mma it issues, whatever the shape: the
    //  two tiles' MMAs of a key tile are issued side by side, not one after the other)
    static constexpr int NTHREADS = 32 * (4 * NT + 1 + NT);
    static constexpr int PRODUCER_WARP = 4 * NT, MMA_WARP = 4 * NT + 1;    // MMA warps: MMA_WARP + ti
    // shared memory map (offsets from a 1024-byte aligned base)
    static constexpr int OFF_Q = 0;                            // NT x [128][128] bf16, 2 sub-tiles each
    static constexpr int OFF_RING = OFF_Q + NT * 2 * QSUB_BYTES;
    static constexpr int OFF_BAR = OFF_RING + NSLOT * SLOT_BYTES;
    static constexpr int OFF_MISC = OFF_BAR + MAX_BARS * 8;    // tmem base, abort flag, unit
    static constexpr int SMEM_BYTES = OFF_MISC + 64;
    // mbarriers: per ring slot, per query tile and score buffer
    static constexpr int BAR_FULL = 0, BAR_EMPTY = NSLOT, BAR_QFULL = 2 * NSLOT;
    static constexpr int BAR_SFULL = BAR_QFULL + 1;            // + ti * 2 + buffer
    static constexpr int BAR_PFULL = BAR_SFULL + 2 * NT;       // + ti * 2 + buffer
    static constexpr int BAR_PVDONE = BAR_PFULL + 2 * NT;      // + ti
    static constexpr int BAR_ALLDONE = BAR_PVDONE + NT;        // + ti
    static constexpr int BAR_DRAIN = BAR_ALLDONE + NT;         // + MMA warp: its MMAs retired, after a wait gave up
    static constexpr int BAR_X = BAR_DRAIN + 2;                // + ti: messages of the merge
    static constexpr int NUM_BARS = BAR_X + NT;
    static_assert(NUM_BARS <= MAX_BARS, "barrier area");
    // TMEM columns: the NT output accumulators, then two score buffers per query tile
    static constexpr uint32_t TM_COLS = 256 * NT;
    static constexpr uint32_t tm_o(int ti) { return (uint32_t)ti * HD; }
    static constexpr uint32_t tm_s(int ti, int sb) { return (uint32_t)(NT * HD + ti * 2 * TN + sb * TN); }
};
static_assert(2 * (Shape<1>::SMEM_BYTES + 1024) <= 228 * 1024, "two CTAs per SM");
static_assert(Shape<2>::SMEM_BYTES <= 227 * 1024, "one CTA per SM");
// The merge takes the place of the query tile and half the ring: [source][8 columns][16 bytes][row], then (reference, sum)
// [source][row], with at most 16 / S (rounded up) times 8 columns from each of S sources
constexpr int EXCHANGE_BYTES = 112 * 1024;
constexpr int exchange_bytes(int S) { return S * ((16 + S - 1) / S) * 4096 + S * MROWS * 8; }
static_assert(exchange_bytes(16) <= EXCHANGE_BYTES && exchange_bytes(12) <= EXCHANGE_BYTES && exchange_bytes(11) <= EXCHANGE_BYTES &&
              exchange_bytes(10) <= EXCHANGE_BYTES && exchange_bytes(9) <= EXCHANGE_BYTES && exchange_bytes(8) <= EXCHANGE_BYTES && exchange_bytes(7) <= EXCHANGE_BYTES &&
              exchange_bytes(6) <= EXCHANGE_BYTES && exchange_bytes(5) <= EXCHANGE_BYTES && exchange_bytes(3) <= EXCHANGE_BYTES, "merge");
static_assert(Shape<1>::OFF_BAR >= EXCHANGE_BYTES && Shape<2>::OFF_BAR >= 2 * EXCHANGE_BYTES, "merge");
constexpr float RESCALE_THRESHOLD = 8.f;                  // log2 units (the persistent kernel)
constexpr uint32_t P_HIGH = 0x5380, P_LOW = 0x2180;       // 2^40 and 2^-60 as bf16: what an unshifted probability may be
struct TcMaps { CUtensorMap k, v, q, kb, vb; };

__device__ inline void bar_start_arrive(int n) { asm volatile("bar.arrive 2, %0;" ::"r"(n) : "memory"); }
__device__ inline void bar_start_wait(int n) { asm volatile("bar.sync 2, %0;" ::"r"(n) : "memory"); }
__device__ inline void bar_tmem_arrive(int n) { asm volatile("bar.arrive 3, %0;" ::"r"(n) : "memory"); }
__device__ inline void bar_tmem_wait(int n) { asm volatile("bar.sync 3, %0;" ::"r"(n) : "memory"); }

// Merge of a cluster, called by the softmax warps that own rows, a thread its row r of the query tile: CTA q ends with the
// eight-column groups [first_group(q), first_group(q + 1)) of all rows.  A thread sends the other CTAs their groups of
// its row with its reference and sum, as 16-byte chunks [source][group][half][row] so that a warp's store is 512
// contiguous bytes, by stores that the destination's barrier counts; then it waits for its own count and sums up, two groups at a time.
// Lanes without a row go the same way with predicated stores: the loads from tensor memory are the whole warp's.  (A branch around
// their stores and a __syncwarp() ahead of each load cost 0.1 us a call.)
__device__ inline int first_group(int q, int S) { return (int)((uint32_t)(16 * q) * ((65536u + S - 1) / (uint32_t)S) >> 16); }
__device__ inline void merge(uint32_t tm_row, unsigned char *smem, uint32_t buf, uint32_t x_bar, int S, int rank, int r, bool valid,
                             bool have_o, float m, float l, __nv_bfloat16 *row, int32_t *status)
{
    const uint32_t sbase = smem_u32(smem);
#pragma unroll 1
    for (int k = 1; k < S; ++k) {
        int q = rank + k;
        if (q >= S) q -= S;
        const int g0 = first_group(q, S), n = first_group(q + 1, S) - g0;
        const uint32_t base = map_to_rank(sbase, q), xb = base + (x_bar - sbase);
        uint32_t dst = base + buf + rank * n * 4096 + r * 16;
        st_async_if(valid, base + buf + S * n * 4096 + (rank * MROWS + r) * 8, m, l, xb);
#pragma unroll 1
        for (int g = g0; g < g0 + n; g += 2, dst += 2 * 4096) {
            uint32_t o[16];                                   // (the second group need not be one of q's)
#pragma unroll
            for (int i = 0; i < 16; ++i) o[i] = 0u;           // (a CTA without keys sends zeros)
            if (have_o) { tmem_ld<16>(tm_row + g * 8, o); tmem_ld_wait(); }
#pragma unroll
            for (int i = 0; i < 4; ++i)
                st_async_if(valid && (i < 2 || g + 1 < g0 + n), dst + i * 2048,
                            make_float4(__uint_as_float(o[4 * i]), __uint_as_float(o[4 * i + 1]),
                                        __uint_as_float(o[4 * i + 2]), __uint_as_float(o[4 * i + 3])), xb);
        }
    }
    // (the wait outlasts every other one: a CTA of the cluster that gave one up sends all the same)
    const bool got = __all_sync(0xffffffffu, mbar_wait_long(x_bar, 0));
    if (!got && (threadIdx.x & 31) == 0 && status) atomicOr(status, ORTHRUS_DEV_WAIT_TIMEOUT);
    const int g0 = first_group(rank, S), n = first_group(rank + 1, S) - g0;
    const unsigned char *src = smem + buf + r * 16;
    float2 *ml = reinterpret_cast<float2 *>(smem + buf + S * n * 4096) + r;
    // weights, in the place of the references
    float mmax = -INFINITY, L = 0.f, own = 0.f;
    ml[rank * MROWS] = make_float2(m, l);
#pragma unroll 8
    for (int j = 0; j < S; ++j) { const float2 x = ml[j * MROWS]; mmax = fmaxf(mmax, x.y > 0.f ? x.x : -INFINITY); }
#pragma unroll 8
    for (int j = 0; j < S; ++j) {
        const float2 x = ml[j * MROWS];
        // (a sum that is not a number has no order: its row is void with it)
        const float w = x.y > 0.f ? ex2(x.x - mmax) : x.y;
        L = fmaf(w, x.y, L);
        if (j == rank) own = w;
        ml[j * MROWS].x = w;
    }
    const float inv = 1.f / L;
#pragma unroll 1
    for (int g = 0; g < n; g += 2) {
        const bool two = g + 1 < n;
        uint32_t o[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) o[i] = 0u;
        if (have_o) { tmem_ld<16>(tm_row + (g0 + g) * 8, o); tmem_ld_wait(); }
        float acc[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) acc[i] = own * __uint_as_float(o[i]);
#pragma unroll 4
        for (int k = 0; k < S - 1; ++k) {
            const int j = k + (k >= rank);
            const float w = ml[j * MROWS].x;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i < 2 || two) {
                    const float4 x = *reinterpret_cast<const float4 *>(src + (j * n + g) * 4096 + i * 2048);
                    acc[4 * i] = fmaf(w, x.x, acc[4 * i]); acc[4 * i + 1] = fmaf(w, x.y, acc[4 * i + 1]);
                    acc[4 * i + 2] = fmaf(w, x.z, acc[4 * i + 2]); acc[4 * i + 3] = fmaf(w, x.w, acc[4 * i + 3]);
                }
        }
#pragma unroll
        for (int i = 0; i < 16; i += 8)
            st_global_if(valid && (i == 0 || two), row + (g0 + g) * 8 + i,
                         make_uint4(pack_bf16(acc[i] * inv, acc[i + 1] * inv), pack_bf16(acc[i + 2] * inv, acc[i + 3] * inv),
                                    pack_bf16(acc[i + 4] * inv, acc[i + 5] * inv), pack_bf16(acc[i + 6] * inv, acc[i + 7] * inv)));
    }
}

// The same for the sizes that plans come to, straight through: no loop, no branch, no address that depends on one.  The
// merge is run through once per call, and what it takes is its chains of instructions and not its bytes (a taken branch alone some 25
// cycles): per call, merge() and this, 64 rows: a unit of 200 keys in a cluster of 2, 6.8 and 5.8 us, 8 units of 300 keys in 4, 6.4 and
// 5.3, of 1000 in 8, 7.4 and 6.6, of 4096 in 16, 11.0 and 10.0; 128 rows, 8 units of 500 keys in 8, 7.3 and 6.7.
template <int SP>
__device__ inline void merge_fixed(uint32_t tm_row, unsigned char *smem, uint32_t buf, uint32_t x_bar, int rank, int r, bool valid, bool have_o,
                                   float m, float l, __nv_bfloat16 *row, int32_t *status)
{
    constexpr bool EVEN = 16 % SP == 0;                       // every CTA has as many groups; else one more here, one fewer there
    constexpr int NG = (16 + SP - 1) / SP, W = 8 * NG, SRC = NG * 4096;       // groups and columns of a CTA at most, bytes of a source
    // destinations whose columns are read together (at eight CTAs five and two: three at a time were level on short prefixes and 1 % of
    // a call slower on long ones, 32 units of 128 rows, 32768 keys)
    constexpr int AT_ONCE = W == 8 || W == 16 ? 5 : W == 32 ? 2 : 1;
    const uint32_t mine = smem_u32(smem) + buf;
    auto next = [&](int k) { return (SP & (SP - 1)) == 0 ? (rank + k) & (SP - 1) : rank + k - (rank + k >= SP ? SP : 0); };
    auto full = [&](int q) { return EVEN || first_group(q + 1, SP) - first_group(q, SP) == NG; };
#pragma unroll
    for (int k0 = 1; k0 < SP; k0 += AT_ONCE) {
        uint32_t o[AT_ONCE][W];
#pragma unroll
        for (int i = 0; i < AT_ONCE; ++i)
#pragma unroll
            for (int x = 0; x < W; ++x) o[i][x] = 0u;         // (a CTA without keys sends zeros)
        if (have_o) {
#pragma unroll
            for (int i = 0; i < AT_ONCE; ++i)                 // (of a CTA with a group fewer the last one is another's)
                if (k0 + i < SP) tmem_ld<W>(tm_row + first_group(next(k0 + i), SP) * 8, o[i]);
            tmem_ld_wait();
        }
#pragma unroll
        for (int i = 0; i < AT_ONCE; ++i) {
            if (k0 + i >= SP) continue;
            const int q = next(k0 + i);
            const uint32_t dst = map_to_rank(mine, q), xb = map_to_rank(x_bar, q);
            st_async_if(valid, dst + SP * SRC + (rank * MROWS + r) * 8, m, l, xb);
#pragma unroll
            for (int c = 0; c < W; c += 4)
                st_async_if(valid && (c < W - 8 || full(q)), dst + rank * SRC + (c / 4 * MROWS + r) * 16,
                            make_float4(__uint_as_float(o[i][c]), __uint_as_float(o[i][c + 1]), __uint_as_float(o[i][c + 2]), __uint_as_float(o[i][c + 3])), xb);
        }
    }
    const int g0 = first_group(rank, SP);
    float acc[W];
    {
        uint32_t o[W];
#pragma unroll
        for (int x = 0; x < W; ++x) o[x] = 0u;
        if (have_o) { tmem_ld<W>(tm_row + g0 * 8, o); tmem_ld_wait(); }
#pragma unroll
        for (int x = 0; x < W; ++x) acc[x] = __uint_as_float(o[x]);
    }
    // (the wait outlasts every other one: a CTA of the cluster that gave one up sends all the same)
    const bool got = __all_sync(0xffffffffu, mbar_wait_long(x_bar, 0));
    if (!got && (threadIdx.x & 31) == 0 && status) atomicOr(status, ORTHRUS_DEV_WAIT_TIMEOUT);
    const unsigned char *src = smem + buf + r * 16;
    const float2 *ml = reinterpret_cast<const float2 *>(smem + buf + SP * SRC) + r;
    float2 x[SP];
    float mmax = -INFINITY, L = 0.f, own = 0.f;
#pragma unroll
    for (int j = 0; j < SP; ++j) { x[j] = ml[j * MROWS]; if (j == rank) x[j] = make_float2(m, l); }
#pragma unroll
    for (int j = 0; j < SP; ++j) mmax = fmaxf(mmax, x[j].y > 0.f ? x[j].x : -INFINITY);
#pragma unroll
    for (int j = 0; j < SP; ++j) {
        const float w = ex2(x[j].x - mmax);
        x[j].x = x[j].y > 0.f ? w : x[j].y;                   // (a sum that is not a number has no order: its row is void with it)
        L = fmaf(x[j].x, x[j].y, L);
        own = j == rank ? x[j].x : own;
    }
#pragma unroll
    for (int i = 0; i < W; ++i) acc[i] *= own;
#pragma unroll
    for (int k = 1; k < SP; ++k) {                            // (source j's slot; a CTA's own, which holds nothing, is passed over)
        const int j = k - 1 + (k - 1 >= rank);
        const float w = k - 1 >= rank ? x[k].x : x[k - 1].x;
#pragma unroll
        for (int c = 0; c < W; c += 4) {                      // (of a group that is not there anything: it is not stored)
            const float4 v = *reinterpret_cast<const float4 *>(src + j * SRC + c / 4 * (MROWS * 16));
            acc[c] = fmaf(w, v.x, acc[c]); acc[c + 1] = fmaf(w, v.y, acc[c + 1]);
            acc[c + 2] = fmaf(w, v.z, acc[c + 2]); acc[c + 3] = fmaf(w, v.w, acc[c + 3]);
        }
    }
    const float inv = 1.f / L;
#pragma unroll
    for (int i = 0; i < W; i += 8)
        st_global_if(valid && (i < W - 8 || full(rank)), row + g0 * 8 + i,
                     make_uint4(pack_bf16(acc[i] * inv, acc[i + 1] * inv), pack_bf16(acc[i + 2] * inv, acc[i + 3] * inv),
                                pack_bf16(acc[i + 4] * inv, acc[i + 5] * inv), pack_bf16(acc[i + 6] * inv, acc[i + 7] * inv)));
}

// Thread r of a softmax warpgroup owns query row r of its tile (TMEM lane r) and all 64 columns of
// a key tile.  blockIdx.z counts groups of NT query tiles; warpgroup ti works on tile z * NT + ti.
//
// PACK (multi-block mask, Eq. 6): the p.nb blocks of a sequence, p.kb_width positions each, lie
// back to back on the position axis (p.K = nb * kb_width), so a 128-row query tile holds the rows
// of several blocks and the prefix is streamed once for all of them.  Row i belongs to block
// j = i / kb_width, sees the prefix below its own anchor cache_len[b * nb + j] and the keys of its
// own block only; the CTA streams up to the largest anchor among the blocks of its query tile,
// then the 64-key tiles of the block axis that hold those blocks' keys.
//
// SC: the size of the cluster where it is 1, 2, 4, 8, 10, 12 or 16, else 0 (then it is an argument).  An instance each, because the end of the
// kernel is straight-line code for its size and none of another's.
template <int NT, bool PACK, int SC>
__global__ void __launch_bounds__(Shape<NT>::NTHREADS, NT == 1 ? 2 : 1)
attend_tc_kernel(const AttnParams p, const __grid_constant__ TcMaps tm, const int s_arg, const int kb_rows,
                 const int quiescent, const int ranked)
{
    using C = Shape<NT>;
    const int S = SC ? SC : s_arg;
    constexpr int W = TN;                     // score columns per softmax thread
    constexpr int NSLOT = C::NSLOT, NTHREADS = C::NTHREADS, NSOFT = 128 * NT;
    constexpr int OFF_Q = C::OFF_Q, OFF_RING = C::OFF_RING, OFF_BAR = C::OFF_BAR, OFF_MISC = C::OFF_MISC;
    constexpr int BAR_FULL = C::BAR_FULL, BAR_EMPTY = C::BAR_EMPTY, BAR_QFULL = C::BAR_QFULL;
    extern __shared__ __align__(1024) unsigned char smem[];
    const uint32_t sbase = smem_u32(smem);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + OFF_MISC + 8);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + OFF_MISC);
    auto bar = [&](int i) { return sbase + OFF_BAR + i * 8; };

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = S > 1 ? (int)cluster_rank() : 0;
    const int order = blockIdx.y;
    // query tile ti of this CTA: kb_rows block positions x G heads (at most 128 rows); the last
    // group of a unit may hold fewer than NT tiles
    // (packed form: anchors usually grow along a sequence, so the last query tiles, which stream the
    //  longest prefixes, are handed out first)
    const int zt = PACK ? (int)(gridDim.z - 1 - blockIdx.z) : (int)blockIdx.z;
    auto tile_i0 = [&](int ti) { return (zt * NT + ti) * kb_rows; };
    auto tile_rows = [&](int ti) { return max(0, min(p.K - tile_i0(ti), kb_rows)) * p.G; };
    const bool aligned = (sbase & 1023u) == 0;                // swizzled tiles need 1 KB alignment

    // ------------------------------------------------------------------ prologue
    // The producer is to ask for its first tiles as early as can be: it sets up the barriers of the ring and waits for nobody.
    if (warp == C::PRODUCER_WARP) {
        if (lane == 0) {
            *abort_flag = aligned ? 0 : 1;                    // (here, as this warp reads it without having waited for another)
            int n_tiles_q = 0;                                // query tiles with rows = MMA warps at work
            for (int ti = 0; ti < NT; ++ti) n_tiles_q += tile_rows(ti) > 0;
#pragma unroll 1
            for (int i = 0; i < NSLOT; ++i) {
                mbar_init(bar(BAR_FULL + i), 1);
                mbar_init(bar(BAR_EMPTY + i), max(1, n_tiles_q));  // every MMA warp releases a slot
            }
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            fence_proxy_async();
        }
        __syncwarp();
        bar_start_arrive(NTHREADS);
    } else if (warp == C::MMA_WARP) {
        if (lane == 0) {
            mbar_init(bar(BAR_QFULL), 1);
            for (int x = 0; x < NT; ++x) {
                const int rows = tile_rows(x), n_act = max(1, (rows + 31) >> 5);      // softmax warps with rows
                for (int sb = 0; sb < 2; ++sb) {
                    mbar_init(bar(C::BAR_SFULL + x * 2 + sb), 1);
                    mbar_init(bar(C::BAR_PFULL + x * 2 + sb), n_act);
                }
                mbar_init(bar(C::BAR_PVDONE + x), 1);
                mbar_init(bar(C::BAR_ALLDONE + x), 1);
                mbar_init(bar(C::BAR_X + x), 1);
            }
            mbar_init(bar(C::BAR_DRAIN), 1);
            mbar_init(bar(C::BAR_DRAIN + 1), 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            fence_proxy_async();
            if (S > 1) {
                const int n = first_group(rank + 1, S) - first_group(rank, S);
                for (int x = 0; x < NT; ++x) mbar_expect_tx(bar(C::BAR_X + x), (uint32_t)(tile_rows(x) * (S - 1) * (n * 32 + 8)));
            }
        }
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(C::TM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // Nothing written by earlier work of the stream has been read so far.
    if (!quiescent) griddep_wait();

    // ------------------------------------------------------------------ which unit
    // when the clusters do not all fit at once they go out longest prefix first (ties by sequence index); every warp finds
    // out by itself
    const int len_hi = (int)p.len_cap;
    static_assert(!PACK || NT == 1, "the packed form runs one query tile per CTA");
    int b = order / p.Hkv;
    const int h = order % p.Hkv;
    if (!PACK && ranked) b = rank_by_length(p, b, len_hi, lane);
    int P;
    int bt_lo = 0, n_blk = 1;               // first tile of block keys on the block axis, how many
    if constexpr (PACK) {
        // blocks j_lo..j_hi have rows in this query tile: stream up to their largest anchor
        const int i0 = tile_i0(0), i1 = min(p.K, i0 + kb_rows) - 1;
        const int j_lo = i0 / p.kb_width, j_hi = i1 / p.kb_width;
        bt_lo = j_lo * p.kb_width / TN;
        n_blk = ((j_hi + 1) * p.kb_width - 1) / TN - bt_lo + 1;
        P = 0;
        bool bad = false;
#pragma unroll 1
        for (int j = j_lo; j <= j_hi; ++j) {
            const int a = __ldg(p.cache_len + (long long)b * p.nb + j);
            bad |= a < 0 || a > len_hi;
            P = max(P, min(max(a, 0), len_hi));
        }
        if (bad && tid == 0 && rank == 0 && p.status) atomicOr(p.status, ORTHRUS_DEV_BAD_CACHE_LEN);
    } else {
        P = p.cache_len[b];
        if (P < 0 || P > len_hi) {
            if (tid == 0 && rank == 0 && p.status) atomicOr(p.status, ORTHRUS_DEV_BAD_CACHE_LEN);
            P = P < 0 ? 0 : len_hi;
        }
    }
    // the unit's tiles: n_pre prefix tiles followed by the tile(s) of block keys, shared out evenly
    const uint32_t n_pre = (uint32_t)(P + TN - 1) / TN;
    const uint32_t t0 = (uint32_t)rank * (n_pre + n_blk) / (uint32_t)S;
    const uint32_t t1 = (uint32_t)(rank + 1) * (n_pre + n_blk) / (uint32_t)S;
    const int n_tiles = (int)(t1 - t0);
    // prefix tiles of this CTA; the tiles behind them are block tiles (one, in the last CTA of the
    // cluster, unless the form is packed)
    const int n_mine = max(0, min(n_tiles, (int)n_pre - (int)t0));
    const bool active = n_tiles > 0 && aligned;

    // The ring holds K and V tiles in the order the MMAs consume them: K0, K1, V0, K2, V1, ...,
    // K(n-1), V(n-2), V(n-1) (the product P.V of a tile is issued after the scores of the next
    // one), so that slots are freed in the order they were filled and a V tile does not sit
    // in the ring while its softmax is still to come.  Item j lives in slot j % NSLOT.
    auto item_of_k = [&](int t) { return t == 0 ? 0 : 2 * t - 1; };
    auto item_of_v = [&](int t) { return min(2 * t + 2, 2 * n_tiles - 1); };
    auto slot_of = [&](int j) { return j % NSLOT; };
    auto use_of = [&](int j) { return j / NSLOT; };

    if (warp < 4 * NT) {
        const int ti = warp >> 2, wq = warp & 3;              // query tile, quarter of its TMEM lanes
        const int r = tid - ti * MROWS;
        const int rows_here = tile_rows(ti);
        const bool valid = r < rows_here;
        const bool warp_active = wq * 32 < rows_here;
        const int i_row = tile_i0(ti) + r / p.G;
        const long long row_at = (((long long)b * p.K + i_row) * p.Hq + h * p.G + r % p.G) * HD;   // this row in q and out
        if (quiescent) {
            // (a line that the preceding kernel is writing may be asked into L2: that is where it is written)
            if (valid) {
                const __nv_bfloat16 *q_row = static_cast<const __nv_bfloat16 *>(p.q) + row_at;
                prefetch_l2(q_row); prefetch_l2(q_row + 64);
            }
            griddep_wait();
        }
        griddep_launch();
        bar_start_wait(NTHREADS);
        tc_fence_after();
        const uint32_t lane_base = *tmem_slot + ((uint32_t)(wq * 32) << 16);
        const uint32_t TM_O = C::tm_o(ti);
        float m_run = 0.f, l_run = 0.f;
        bool fresh = true;                  // the row has seen no key yet, or only such with scores of -inf
        bool have_o = false;
        int a_row = 0, k0_row = 0;          // packed form: this row's anchor, first key of its block
        if constexpr (PACK) {
            if (valid) {
                const int j_row = i_row / p.kb_width;
                a_row = min(max(__ldg(p.cache_len + (long long)b * p.nb + j_row), 0), len_hi);
                k0_row = j_row * p.kb_width;
            }
        }
        if (active && warp_active) {
            // -------------------------------------------------------------- softmax
            const float sc = p.scale_log2;
            const float2 sc2 = make_float2(sc, sc);
            bool ok = true;
#pragma unroll 1
            for (int t = 0; t < n_tiles; ++t) {
                const int sb = t & 1;
                // visible columns of this row in this tile: [lo, lim)
                int lim, lo = 0;
                if constexpr (PACK) {
                    if (t < n_mine) {
                        lim = min(TN, a_row - ((int)t0 + t) * TN);
                    } else {
                        const int c0 = k0_row - (bt_lo + (int)t0 + t - (int)n_pre) * TN;
                        lo = max(c0, 0);
                        lim = min(TN, c0 + p.kb_width);
                    }
                    if (lim <= lo) { lim = 0; lo = 0; }
                } else {
                    if (t < n_mine) lim = min(TN, P - ((int)t0 + t) * TN);
                    else lim = p.causal ? min(p.K, i_row + 1) : p.K;
                }
                lim = valid ? lim : 0;
                // (rows that see all of the tile or nothing, as most do in the packed form, need no masks: their probabilities are
                //  struck out)
                const bool masks = __any_sync(0xffffffffu, lim > lo && (lim < W || lo > 0));
                const bool strike = __any_sync(0xffffffffu, lim <= lo);
                ok = mbar_wait_warp_inline(bar(C::BAR_SFULL + ti * 2 + sb), (t >> 1) & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                const uint32_t TM_S = C::tm_s(ti, sb);
                // Probabilities with the reference as it is: 0 to begin with.  That will do as long as none is out of all
                // proportion and, in the first tile that shows the row a key, they are not all tiny: floating-point numbers
                // keep their relative precision whatever the reference, so that no tile pays for its row maxima.
                // (References are integers, as in attend_keys.cu: another reference scales a probability by a power of two, so
                // that its rounding to bf16 does not depend on the cut or the kernel.  The sums do depend on the kernel:
                // here of the probabilities before rounding, there of the rounded ones.  Summed after rounding
                // here too, a call of 8 units of 64 rows took 2.3 % longer, and fp32 sums in another order still differ.)
                uint32_t pk[W / 2];                            // this thread's probabilities, packed bf16
                float2 acc0 = make_float2(0.f, 0.f), acc1 = acc0;
                bool exact = false;
                const bool any = !PACK || __any_sync(0xffffffffu, lim > lo);
                if (!any)                                      // (packed form: a tile that none of the warp's rows sees)
#pragma unroll
                    for (int j = 0; j < W / 2; ++j) pk[j] = 0u;
#pragma unroll 1
                while (any) {
                    uint32_t s[W];
                    tmem_ld<W>(lane_base + TM_S, s);
                    tmem_ld_wait();
                    if (masks) {
#pragma unroll
                        for (int j = 0; j < W; ++j) if (j >= lim || j < lo) s[j] = 0xff800000u;
                    }
                    const float2 nm2 = make_float2(-m_run, -m_run);
                    uint32_t top = 0;                          // the largest, as bit patterns
                    acc0 = make_float2(0.f, 0.f); acc1 = acc0;
#pragma unroll
                    for (int j = 0; j < W; j += 4) {
                        float2 a = __ffma2_rn(make_float2(__uint_as_float(s[j]), __uint_as_float(s[j + 1])), sc2, nm2);
                        float2 c = __ffma2_rn(make_float2(__uint_as_float(s[j + 2]), __uint_as_float(s[j + 3])), sc2, nm2);
                        a.x = ex2(a.x); a.y = ex2(a.y); c.x = ex2(c.x); c.y = ex2(c.y);
                        acc0 = __fadd2_rn(acc0, a);
                        acc1 = __fadd2_rn(acc1, c);
                        pk[j >> 1] = pack_bf16(a.x, a.y);
                        pk[(j >> 1) + 1] = pack_bf16(c.x, c.y);
                        top = __vimax3_u16x2(top, pk[j >> 1], pk[(j >> 1) + 1]);
                    }
                    const uint32_t most = max(top & 0xffffu, top >> 16);
                    if (strike) {
                        const bool sees = lim > lo;
                        if (!sees) { acc0 = make_float2(0.f, 0.f); acc1 = acc0; }
#pragma unroll
                        for (int j = 0; j < W / 2; ++j) pk[j] = sees ? pk[j] : 0u;
                    }
                    const bool off = lim > lo && (most > P_HIGH || (fresh && most < P_LOW));
                    if (exact || !__any_sync(0xffffffffu, off)) break;
                    // the references of these rows are set to the maximum of the tile, or, behind the first, raised to it
                    exact = true;
                    float mx = -INFINITY;
#pragma unroll 1
                    for (int c = 0; c < W; c += 16) {
                        uint32_t x[16];
                        tmem_ld<16>(lane_base + TM_S + c, x);
                        tmem_ld_wait();
#pragma unroll
                        for (int j = 0; j < 16; ++j) if (c + j < lim && c + j >= lo) mx = fmaxf(mx, __uint_as_float(x[j]));
                    }
                    mx = ceilf(mx * sc);
                    float alpha = 1.f;
                    if (off && mx > -INFINITY && (fresh || mx > m_run)) {
                        if (!fresh) { alpha = ex2(m_run - mx); l_run *= alpha; }
                        m_run = mx;
                    }
                    if (t > 0 && __any_sync(0xffffffffu, alpha != 1.f)) {
                        // O holds the products of tiles 0..t-1 and nothing is adding to it now
                        ok = mbar_wait_warp_inline(bar(C::BAR_PVDONE + ti), (t - 1) & 1, abort_flag);
                        if (!ok) break;
                        tc_fence_after();
#pragma unroll 1
                        for (int c4 = 0; c4 < HD / 16; ++c4) {
                            uint32_t o[16];
                            tmem_ld<16>(lane_base + TM_O + c4 * 16, o);
                            tmem_ld_wait();
#pragma unroll
                            for (int j = 0; j < 16; ++j) o[j] = __float_as_uint(__uint_as_float(o[j]) * alpha);
                            tmem_st16(lane_base + TM_O + c4 * 16, o);
                        }
                    }
                }
                if (!ok) break;
                l_run += (acc0.x + acc0.y) + (acc1.x + acc1.y);
                fresh = fresh && !(l_run > 0.f);               // (nothing but scores of -inf tells of no reference)
                // P over the scores, 2 bf16 per 32-bit column
                tmem_st32(lane_base + TM_S, pk);
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(C::BAR_PFULL + ti * 2 + sb));
            }
            // BAR_PVDONE cannot be used here: a parity wait cannot tell phase k from phase k-2, and
            // by now the barrier may be one or two phases ahead of what this thread last observed
            if (ok) ok = mbar_wait_warp_inline(bar(C::BAR_ALLDONE + ti), 0, abort_flag);
            if (ok) tc_fence_after();
            have_o = ok;
        }
        const uint32_t tm_row = lane_base + TM_O;
        __nv_bfloat16 *row = static_cast<__nv_bfloat16 *>(p.out) + row_at;
        if (S == 1) {
            // ---------------------------------------------------------- direct output
            // the whole unit was here: normalise and write the final rows
            if (have_o) {
                const float inv = 1.f / l_run;
#pragma unroll 1
                for (int c = 0; c < HD; c += 32) {
                    uint32_t o[32];
                    tmem_ld32(tm_row + c, o);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 32; i += 8)
                        st_global_if(valid, row + c + i, make_uint4(
                            pack_bf16(__uint_as_float(o[i]) * inv, __uint_as_float(o[i + 1]) * inv),
                            pack_bf16(__uint_as_float(o[i + 2]) * inv, __uint_as_float(o[i + 3]) * inv),
                            pack_bf16(__uint_as_float(o[i + 4]) * inv, __uint_as_float(o[i + 5]) * inv),
                            pack_bf16(__uint_as_float(o[i + 6]) * inv, __uint_as_float(o[i + 7]) * inv)));
                }
            }
        } else {
            // ---------------------------------------------------------- merge
            cluster_arrive_relaxed();                         // (every CTA's query tile and ring are to be idle)
            if (!have_o) l_run = 0.f;                         // a CTA without keys takes part with zeros
            const uint32_t buf = (uint32_t)(ti * EXCHANGE_BYTES);
            __syncwarp();
            cluster_wait();
            if (warp_active) {
                if constexpr (SC > 1) merge_fixed<SC>(tm_row, smem, buf, bar(C::BAR_X + ti), rank, r, valid, have_o, m_run, l_run, row, p.status);
                else merge(tm_row, smem, buf, bar(C::BAR_X + ti), S, rank, r, valid, have_o, m_run, l_run, row, p.status);
            }
        }
        tc_fence_before();
        __syncwarp();
        bar_tmem_arrive(NSOFT + 32);
    } else if (warp == C::PRODUCER_WARP) {
        // ------------------------------------------------------------------ producer
        if (active && lane == 0) {
            const uint64_t stream_policy = policy_evict_first();
            const int row_base = (int)(((long long)(PACK ? b : b / p.nb) * p.Hkv + h) * p.capacity);   // row of position 0
            const int n_items = 2 * n_tiles;
            // with a promise that the cache rows below cache_len are not being written by the preceding kernel the first
            // prefix tiles are asked for before the wait for it (up to the block tile's first item)
            int early = quiescent ? min(n_mine < n_tiles ? item_of_k(n_mine) : n_items, NSLOT) : 0;
            bool ok = true;
            int j = 0;
#pragma unroll 1
            for (; j < n_items; ++j) {
                if (j == early) { if (quiescent) griddep_wait(); early = -1; }
                const int slot = slot_of(j), use = use_of(j);
                if (use > 0) ok = mbar_wait_call(bar(BAR_EMPTY + slot), (use - 1) & 1, abort_flag);
                if (!ok) break;
                const bool is_v = j == n_items - 1 || (j > 0 && (j & 1) == 0);
                const int t = is_v ? (j == n_items - 1 ? n_tiles - 1 : j / 2 - 1) : (j + 1) / 2;
                const uint32_t dst = sbase + OFF_RING + slot * SLOT_BYTES, fb = bar(BAR_FULL + slot);
                mbar_expect_tx(fb, SLOT_BYTES);
                if (t < n_mine || (!PACK && p.blk_in_cache)) {
                    // (block tile in the cache = the 64 cache rows from P on: rows >= K hold whatever follows the block, masked
                    // out of the scores, cleared in the V tile before its product)
                    const CUtensorMap *m = is_v ? &tm.v : &tm.k;
                    const int at = row_base + (t < n_mine ? ((int)t0 + t) * TN : P);
                    tma_load_2d(dst, m, 0, at, fb, stream_policy);
                    tma_load_2d(dst + SUB_BYTES, m, 64, at, fb, stream_policy);
                } else {
                    // a tile of the block axis: rows past its end are out of bounds and arrive as zeros
                    const CUtensorMap *m = is_v ? &tm.vb : &tm.kb;
                    const int at = PACK ? (bt_lo + (int)t0 + t - (int)n_pre) * TN : 0;
                    tma_load_4d(dst, m, 0, h, at, b, fb);
                    tma_load_4d(dst + SUB_BYTES, m, 64, h, at, b, fb);
                }
            }
            if (*abort_flag) {
                // give the copies that were armed a bounded time to land before smem is released
                uint32_t seen = 0;
#pragma unroll 1
                for (int i = j - 1; i >= 0 && seen != (1u << NSLOT) - 1; --i) {   // latest use of each slot
                    int dummy = 0;
                    if (!(seen >> slot_of(i) & 1)) mbar_wait_call(bar(BAR_FULL + slot_of(i)), use_of(i) & 1, &dummy);
                    seen |= 1u << slot_of(i);
                }
            }
        }
        __syncwarp();
        if (S > 1) { cluster_arrive_relaxed(); cluster_wait(); }
    } else {
        // ------------------------------------------------------------------ MMA issue, query tile ti
        const int ti = warp - C::MMA_WARP;
        tc_fence_before();
        bar_start_wait(NTHREADS);
        tc_fence_after();
        const uint32_t tmem = *tmem_slot;
        if (ti == 0) {
            if (quiescent) griddep_wait();
            if (active && elect_one()) {
                // the query rows of every tile: box = 64 columns x G heads x kb_rows positions
                int n_q = 0;
                for (int x = 0; x < NT; ++x) n_q += tile_rows(x) > 0;
                mbar_expect_tx(bar(BAR_QFULL), (uint32_t)(n_q * 2 * 128 * p.G * kb_rows));
                for (int x = 0; x < NT; ++x)
                    if (tile_rows(x) > 0) {
                        const uint32_t q_dst = sbase + OFF_Q + x * 2 * QSUB_BYTES;
                        tma_load_4d(q_dst, &tm.q, 0, h * p.G, tile_i0(x), b, bar(BAR_QFULL));
                        tma_load_4d(q_dst + QSUB_BYTES, &tm.q, 64, h * p.G, tile_i0(x), b, bar(BAR_QFULL));
                    }
            }
            __syncwarp();
        }
        bool ok = active && tile_rows(ti) > 0;
        if (ok) {
            constexpr uint32_t IDESC_QK = make_idesc(TN, 0);  // A = Q, B = K tile, both K-major
            constexpr uint32_t IDESC_PV = make_idesc(HD, 1);  // A = P (TMEM), B = V tile (MN-major)
            const uint64_t q_desc = make_desc(sbase + OFF_Q + ti * 2 * QSUB_BYTES, 16, 1024);
            ok = mbar_wait_warp_call(bar(BAR_QFULL), 0, abort_flag);
            // step t: the scores of tile t, then, while its softmax runs, the product of tile t - 1
#pragma unroll 1
            for (int t = 0; t <= n_tiles && ok; ++t) {
                if (t < n_tiles) {
                    const int j = item_of_k(t), slot = slot_of(j);
                    ok = mbar_wait_warp_inline(bar(BAR_FULL + slot), use_of(j) & 1, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
                        const uint64_t kd = make_desc(sbase + OFF_RING + slot * SLOT_BYTES, 16, 1024);
                        const uint32_t d = tmem + C::tm_s(ti, t & 1);
#pragma unroll
                        for (int kk = 0; kk < HD / 16; ++kk)          // 16 head-dim columns per MMA
                            umma_ss(d, q_desc + (((kk >> 2) * QSUB_BYTES + (kk & 3) * 32) >> 4),
                                    kd + (((kk >> 2) * SUB_BYTES + (kk & 3) * 32) >> 4), IDESC_QK, kk > 0);
                        umma_commit(bar(BAR_EMPTY + slot));
                        umma_commit(bar(C::BAR_SFULL + ti * 2 + (t & 1)));
                    }
                    __syncwarp();
                }
                if (t > 0) {
                    const int pt = t - 1, j = item_of_v(pt), slot = slot_of(j);
                    ok = mbar_wait_warp_inline(bar(BAR_FULL + slot), use_of(j) & 1, abort_flag);
                    if (!ok) break;
                    // Only the 16-key groups that hold keys are multiplied (an instruction costs its issuing
                    // thread the same whatever its size): the block's own tile is K keys wide, a ragged
                    // prefix tile ends at the prefix.  In the last group, V rows past the keys may hold
                    // anything where they come from the cache, and 0 * NaN would poison the product, so
                    // they are cleared before the MMA reads them (by every MMA warp: the same zeros, and
                    // no warp has to wait for another); rows of the block's own tensor past K arrive as zeros.
                    const bool from_cache = pt < n_mine || p.blk_in_cache;
                    const int nv = pt < n_mine ? min(TN, P - ((int)t0 + pt) * TN) : (PACK ? TN : p.K);
                    const int n_kk = (nv + 15) >> 4;
                    if (from_cache && nv < n_kk * 16) {
                        unsigned char *vt = smem + OFF_RING + slot * SLOT_BYTES;
#pragma unroll 1
                        for (int e = lane; e < (n_kk * 16 - nv) * 16; e += 32) {
                            const int rr = nv + (e >> 4), c = e & 15;
                            *reinterpret_cast<uint4 *>(vt + sw_off(rr, c, SUB_BYTES)) = make_uint4(0, 0, 0, 0);
                        }
                        fence_proxy_async();
                        __syncwarp();
                    }
                    ok = mbar_wait_warp_inline(bar(C::BAR_PFULL + ti * 2 + (pt & 1)), (pt >> 1) & 1, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
                        const uint64_t vd = make_desc(sbase + OFF_RING + slot * SLOT_BYTES, SUB_BYTES, 1024);
                        const uint32_t a = tmem + C::tm_s(ti, pt & 1);
#pragma unroll
                        for (int kk = 0; kk < TN / 16; ++kk)          // 16 key positions per MMA
                            if (kk < n_kk)
                                umma_ts(tmem + C::tm_o(ti), a + kk * 8, vd + (kk * 2048 >> 4), IDESC_PV, (pt > 0) || (kk > 0));
                        umma_commit(bar(BAR_EMPTY + slot));
                        umma_commit(bar(C::BAR_PVDONE + ti));
                        if (pt == n_tiles - 1) umma_commit(bar(C::BAR_ALLDONE + ti));
                    }
                    __syncwarp();
                }
            }
            // every MMA of this warp must have retired before TMEM is freed
            if (ok) ok = mbar_wait_warp_call(bar(C::BAR_ALLDONE + ti), 0, abort_flag);
            if (!ok) {
                // a wait gave up: this warp's MMAs in flight still read shared memory and write TMEM, and the query rows may
                // still be on their way
                const int drain = C::BAR_DRAIN + ti;
                if (elect_one()) umma_commit(bar(drain));     // (a commit tells of its own thread's MMAs)
                __syncwarp();
                int dummy = 0;
                mbar_wait_warp_call(bar(drain), 0, &dummy);
                if (ti == 0) mbar_wait_warp_call(bar(BAR_QFULL), 0, &dummy);
            }
        }
        tc_fence_before();
        __syncwarp();
        if (S > 1) cluster_arrive_relaxed();
        if (ti == 0) {
            bar_tmem_wait(NSOFT + 32);                        // the softmax warps have read their TMEM
            tc_fence_after();
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::TM_COLS) : "memory");
            if (lane == 0 && *abort_flag && p.status) atomicOr(p.status, ORTHRUS_DEV_WAIT_TIMEOUT);
        }
        if (S > 1) cluster_wait();
    }
}

#include "attend_tc_stream.cuh"

// ---------------------------------------------------------------------------- host side

}  // namespace

EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) ==
                cudaSuccess && qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(ptr);
    });
    return fn;
}

namespace {

// Tensor maps over bf16 tensors whose innermost dimension is the head (hd = 64 or 128 wide): up to
// four dimensions, boxes of 64 columns with the 128-byte swizzle.  Cached by (pointer, shape).
struct MapKey {
    const void *ptr; unsigned long long d1, d2, d3; unsigned b1, b2, hd;
    bool operator==(const MapKey &o) const {
        return ptr == o.ptr && hd == o.hd && d1 == o.d1 && d2 == o.d2 && d3 == o.d3 && b1 == o.b1 && b2 == o.b2;
    }
};
struct MapKeyHash {
    size_t operator()(const MapKey &k) const {
        size_t x = std::hash<const void *>()(k.ptr);
        for (unsigned long long v : {k.d1, k.d2, k.d3, (unsigned long long)k.b1 << 32 | k.b2, (unsigned long long)k.hd})
            x = (x ^ v) * 0x9E3779B97F4A7C15ull;
        return x;
    }
};

}  // namespace

// dims: (hd, d1, d2, d3) row-major with d3 outermost; box (64, b1, b2, 1).  rank = 2 when
// d2 == 0 (then the box is (64, b1)).
bool tensor_map(const void *ptr, unsigned hd, unsigned long long d1, unsigned long long d2, unsigned long long d3,
             unsigned b1, unsigned b2, CUtensorMap *out)
{
    static std::mutex mu;
    static std::unordered_map<MapKey, CUtensorMap, MapKeyHash> cache;
    std::lock_guard<std::mutex> lock(mu);
    const MapKey key{ptr, d1, d2, d3, b1, b2, hd};
    auto it = cache.find(key);
    if (it != cache.end()) { *out = it->second; return true; }
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const int rank = d2 == 0 ? 2 : 4;
    const cuuint64_t dims[4] = {(cuuint64_t)hd, (cuuint64_t)d1, (cuuint64_t)d2, (cuuint64_t)d3};
    const cuuint64_t strides[3] = {(cuuint64_t)hd * 2, (cuuint64_t)hd * 2 * d1, (cuuint64_t)hd * 2 * d1 * d2};
    const cuuint32_t box[4] = {64, b1, b2, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    CUtensorMap tm;
    const CUresult r = fn(&tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void *>(ptr), dims,
                          strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                          CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return false;
    if (cache.size() > 4096) cache.clear();
    cache.emplace(key, tm);
    *out = tm;
    return true;
}

// block positions per query tile of 128 rows
int tc_kb_rows(int G, int K) { return K < MROWS / G ? K : MROWS / G; }

int tc_row_tiles(int G, int K)
{
    if (G < 1 || G > MROWS) return 0;
    const int kb = tc_kb_rows(G, K);
    return (K + kb - 1) / kb;
}

// Query tiles per CTA.  Units wider than one 128-row tile run one CTA per query tile by default:
// the CTAs of a unit walk the cache in step, so the second read of every K/V tile is an L2 hit
// (measured DRAM read 545 MB for 539 MB of cache at 256 rows) and two CTAs per SM overlap better
// than one wide CTA.  ORTHRUS_TC_ROW_TILES_PER_CTA=2 selects the shape whose two query tiles share
// one K/V ring (measured 8 % slower at 256 rows; kept for measurements).
int tc_tiles_per_cta(int G, int K)
{
    static const int forced = [] { const char *e = getenv("ORTHRUS_TC_ROW_TILES_PER_CTA"); return e ? atoi(e) : 0; }();
    return (forced == 2 && tc_row_tiles(G, K) >= 2) ? 2 : 1;
}

// CTAs along the query-tile axis of the grid
int tc_cta_groups(int G, int K)
{
    const int nt = tc_tiles_per_cta(G, K);
    return (tc_row_tiles(G, K) + nt - 1) / nt;
}

bool tc_driver_ok() { return encode_fn() != nullptr; }

// CTAs of the shape with nt query tiles one SM of the current device keeps resident: what its
// shared memory holds (each CTA also costs the 1 KB the system reserves per block), at most what
// the 512 TMEM columns allow.  2 and 1 on a B200.  Asked once per device; those values are assumed
// where there is no device.
int tc_ctas_per_sm(int nt)
{
    constexpr int kMaxDevices = 64;
    static std::mutex mu;
    static int smem_cached[kMaxDevices] = {};
    const int smem_bytes = nt == 2 ? Shape<2>::SMEM_BYTES : Shape<1>::SMEM_BYTES;
    const int by_tmem = nt == 2 ? 1 : 2;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) { (void)cudaGetLastError(); return by_tmem; }
    std::lock_guard<std::mutex> lock(mu);
    if (!smem_cached[dev]) {
        int smem_per_sm = 0;
        if (cudaDeviceGetAttribute(&smem_per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess) {
            (void)cudaGetLastError();
            return by_tmem;
        }
        smem_cached[dev] = smem_per_sm;
    }
    const int n = smem_cached[dev] / (smem_bytes + 1024);
    return n < 1 ? 1 : (n > by_tmem ? by_tmem : n);
}

namespace {

template <int NT, bool PACK = false, int SC = 0>
cudaError_t configure_kernel()
{   // function attributes belong to a device: set them once on each device that launches
    constexpr int kMaxDevices = 64;
    static std::mutex mu;
    static bool configured[kMaxDevices] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (!configured[dev]) {
        e = cudaFuncSetAttribute(attend_tc_kernel<NT, PACK, SC>, cudaFuncAttributeMaxDynamicSharedMemorySize, Shape<NT>::SMEM_BYTES);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(attend_tc_kernel<NT, PACK, SC>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        configured[dev] = true;
    }
    return cudaSuccess;
}

template <int NT>
int max_cluster_of_shape()
{
    constexpr int kMaxDevices = 64;
    static std::mutex mu;
    static int cached[kMaxDevices] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 16;
    std::lock_guard<std::mutex> lock(mu);
    if (cached[dev]) return cached[dev];
    int best = 16;
    if (configure_kernel<NT>() == cudaSuccess) {
        for (int s = 16; s >= 2; s >>= 1) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(s, 1, 1);
            cfg.blockDim = dim3(Shape<NT>::NTHREADS);
            cfg.dynamicSmemBytes = Shape<NT>::SMEM_BYTES;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = s; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr; cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, attend_tc_kernel<NT, false, 0>, &cfg) == cudaSuccess && n > 0) { best = s; break; }
            best = s >> 1;
        }
        if (best < 1) best = 1;
    } else {
        (void)cudaGetLastError();
    }
    cached[dev] = best;
    return best;
}

}  // namespace

// Largest cluster size (a power of two up to 16) the current device can co-schedule for the shape
// with nt query tiles; 16 on a full B200.  Without a device (or if the query fails) 16 is assumed
// and a launch that cannot be scheduled reports its error.
int tc_max_cluster(int nt) { return nt == 2 ? max_cluster_of_shape<2>() : max_cluster_of_shape<1>(); }
int tc_tile_positions() { return TN; }

template <int NT, bool PACK = false, int SC = 0>
static cudaError_t launch_tc(const AttnParams &p, const TcMaps &tm, int kb, int flags, cudaStream_t st)
{
    const int S = p.n_splits;
    if constexpr (NT == 1 && SC == 0) {                       // the instance of this cluster size, where there is one
        switch (S) {
        case 1: return launch_tc<NT, PACK, 1>(p, tm, kb, flags, st);
        case 2: return launch_tc<NT, PACK, 2>(p, tm, kb, flags, st);
        case 4: return launch_tc<NT, PACK, 4>(p, tm, kb, flags, st);
        case 8: return launch_tc<NT, PACK, 8>(p, tm, kb, flags, st);
        case 10: return launch_tc<NT, PACK, 10>(p, tm, kb, flags, st);
        case 12: return launch_tc<NT, PACK, 12>(p, tm, kb, flags, st);
        case 16: return launch_tc<NT, PACK, 16>(p, tm, kb, flags, st);
        }
    }
    cudaError_t e = configure_kernel<NT, PACK, SC>();
    if (e != cudaSuccess) return e;
    const int row_tiles = (p.K + kb - 1) / kb;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(S, p.B * p.Hkv, (row_tiles + NT - 1) / NT);
    cfg.blockDim = dim3(Shape<NT>::NTHREADS);
    cfg.dynamicSmemBytes = Shape<NT>::SMEM_BYTES;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int n_attr = 0;
    if (S > 1) {
        attr[n_attr].id = cudaLaunchAttributeClusterDimension;
        attr[n_attr].val.clusterDim.x = S;
        attr[n_attr].val.clusterDim.y = 1;
        attr[n_attr].val.clusterDim.z = 1;
        ++n_attr;
    }
    if (!(flags & ORTHRUS_LAYER_NO_EARLY_LAUNCH)) {
        attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n_attr].val.programmaticStreamSerializationAllowed = 1;
        ++n_attr;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n_attr;
    const long long ctas = (long long)S * p.B * p.Hkv * cfg.gridDim.z;
    const int ranked = !PACK && p.B > 1 && p.B <= 128 && ctas > (long long)tc_ctas_per_sm(NT) * num_sms();
    e = cudaLaunchKernelEx(&cfg, attend_tc_kernel<NT, PACK, SC>, p, tm, S, kb, (flags & ORTHRUS_LAYER_CACHE_QUIESCENT) ? 1 : 0, ranked);
    count_launch();
    return e;
}

// The persistent kernel serves one query tile per unit and ranks at most 128 batch entries.
bool tc_stream_shape(int B, int G, int K) { return B <= STREAM_MAX_B && G >= 1 && G * K <= MROWS && K <= TN; }

// Workspace of the persistent kernel behind the header: two partial tiles and their (max, sum)
// rows per CTA, then one arrival counter per unit (zero between calls).
size_t tc_stream_workspace_bytes(int B, int Hkv, int n_ctas)
{
    return (size_t)n_ctas * 2 * (MROWS * HD * sizeof(float) + MROWS * 2 * sizeof(float)) +
           (((size_t)B * Hkv * sizeof(int32_t) + 255) / 256) * 256;
}

cudaError_t launch_attend_tc_stream(const AttnParams &p, int n_ctas, void *ws_body, int flags, cudaStream_t st)
{
    TcMaps tm;
    const unsigned long long rows = (unsigned long long)(p.B / p.nb) * p.Hkv * p.capacity;
    if (!tensor_map(p.k_cache, HD, rows, 0, 0, TN, 0, &tm.k) || !tensor_map(p.v_cache, HD, rows, 0, 0, TN, 0, &tm.v) ||
        !tensor_map(p.q, HD, p.Hq, p.K, p.B, p.G, p.K, &tm.q))
        return cudaErrorInvalidValue;
    if (p.blk_in_cache) {
        tm.kb = tm.k; tm.vb = tm.v;
    } else if (!tensor_map(p.k_blk, HD, p.Hkv, p.K, p.B, 1, TN, &tm.kb) || !tensor_map(p.v_blk, HD, p.Hkv, p.K, p.B, 1, TN, &tm.vb)) {
        return cudaErrorInvalidValue;
    }
    {   // function attributes belong to a device: set them once on each device that launches
        constexpr int kMaxDevices = 64;
        static std::mutex mu;
        static bool configured[kMaxDevices] = {};
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
        std::lock_guard<std::mutex> lock(mu);
        if (!configured[dev]) {
            e = cudaFuncSetAttribute(attend_tc_stream_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, STREAM_SMEM_BYTES);
            if (e != cudaSuccess) return e;
            configured[dev] = true;
        }
    }
    StreamArgs sa;
    unsigned char *base = static_cast<unsigned char *>(ws_body);
    sa.part_o = reinterpret_cast<float4 *>(base);
    sa.part_ml = reinterpret_cast<float2 *>(base + (size_t)n_ctas * 2 * MROWS * HD * sizeof(float));
    sa.counters = reinterpret_cast<int32_t *>(base + (size_t)n_ctas * 2 * (MROWS * HD + MROWS * 2) * sizeof(float));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n_ctas, 1, 1);
    cfg.blockDim = dim3(Shape<1>::NTHREADS);
    cfg.dynamicSmemBytes = STREAM_SMEM_BYTES;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    int n_attr = 0;
    if (!(flags & ORTHRUS_LAYER_NO_EARLY_LAUNCH)) {
        attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n_attr].val.programmaticStreamSerializationAllowed = 1;
        ++n_attr;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n_attr;
    cudaError_t e = cudaLaunchKernelEx(&cfg, attend_tc_stream_kernel, p, tm, sa);
    count_launch();
    return e;
}

cudaError_t launch_attend_tc(const AttnParams &p, int flags, cudaStream_t st)
{
    const int kb = tc_kb_rows(p.G, p.K);
    TcMaps tm;
    const unsigned long long rows = (unsigned long long)(p.B / p.nb) * p.Hkv * p.capacity;
    if (!tensor_map(p.k_cache, HD, rows, 0, 0, TN, 0, &tm.k) || !tensor_map(p.v_cache, HD, rows, 0, 0, TN, 0, &tm.v) ||
        !tensor_map(p.q, HD, p.Hq, p.K, p.B, p.G, kb, &tm.q))
        return cudaErrorInvalidValue;
    if (p.blk_in_cache) {
        tm.kb = tm.k; tm.vb = tm.v;           // unused: the block tile comes through the cache maps
    } else if (!tensor_map(p.k_blk, HD, p.Hkv, p.K, p.B, 1, TN, &tm.kb) || !tensor_map(p.v_blk, HD, p.Hkv, p.K, p.B, 1, TN, &tm.vb)) {
        return cudaErrorInvalidValue;
    }
    if (tc_tiles_per_cta(p.G, p.K) == 2) return launch_tc<2>(p, tm, kb, flags, st);
    return launch_tc<1>(p, tm, kb, flags, st);
}

// Packed multi-block form: p.B sequences, p.nb blocks of p.kb_width positions each on one position
// axis of p.K = nb * kb_width, anchors in p.cache_len[B][nb].
cudaError_t launch_attend_tc_packed(const AttnParams &p, int flags, cudaStream_t st)
{
    const int kb = tc_kb_rows(p.G, p.K);
    TcMaps tm;
    const unsigned long long rows = (unsigned long long)p.B * p.Hkv * p.capacity;
    if (!tensor_map(p.k_cache, HD, rows, 0, 0, TN, 0, &tm.k) || !tensor_map(p.v_cache, HD, rows, 0, 0, TN, 0, &tm.v) ||
        !tensor_map(p.q, HD, p.Hq, p.K, p.B, p.G, kb, &tm.q) ||
        !tensor_map(p.k_blk, HD, p.Hkv, p.K, p.B, 1, TN, &tm.kb) || !tensor_map(p.v_blk, HD, p.Hkv, p.K, p.B, 1, TN, &tm.vb))
        return cudaErrorInvalidValue;
    return launch_tc<1, true>(p, tm, kb, flags, st);
}

}  // namespace orthrus
