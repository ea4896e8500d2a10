// C-ABI entry points: argument validation, split-KV planning, kernel-path dispatch.
#include <atomic>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <unistd.h>
#include "common.cuh"

namespace orthrus {

static std::atomic<long long> g_launches{0};
void count_launch(int n) { g_launches.fetch_add(n, std::memory_order_relaxed); }

enum Path { PATH_AUTO = 0, PATH_SIMT, PATH_MMA, PATH_TCGEN05 };
static std::atomic<int> g_path{-1};
static thread_local const char *t_last_path = "none";

static int parse_path(const char *s)
{
    if (!s || !*s || !strcmp(s, "auto")) return PATH_AUTO;
    if (!strcmp(s, "simt")) return PATH_SIMT;
    if (!strcmp(s, "mma")) return PATH_MMA;
    if (!strcmp(s, "tcgen05")) return PATH_TCGEN05;
    return -1;
}

static int current_path()
{
    int v = g_path.load();
    if (v < 0) {
        v = parse_path(getenv("ORTHRUS_FORCE_PATH"));
        if (v < 0) v = PATH_AUTO;
        g_path.store(v);
    }
    return v;
}

// The tuning variables of the environment, read at every call that plans (a test changes them
// between calls).  One walk over the environment, which hardly ever holds any of them, instead of a
// search per variable: half a dozen searches were a tenth of a call's host time.
struct Knobs {
    int splits = 0, min_chunk_tiles = 2, target_ctas = 0;     // 0: not forced / the default
    int small_rows = -1;                                      // -1: by the rule of keys_usable
    bool no_early_launch = false, stream = false, pack = true;
};
static Knobs read_knobs()
{
    Knobs k;
    for (char **e = environ; e && *e; ++e) {
        const char *s = *e;
        if (s[0] != 'O' || strncmp(s, "ORTHRUS_", 8) != 0) continue;
        s += 8;
        const char *eq = strchr(s, '=');
        if (!eq || !eq[1]) continue;
        const size_t n = (size_t)(eq - s);
        const char *val = eq + 1;
        auto is = [&](const char *name) { return strlen(name) == n && !strncmp(s, name, n); };
        auto positive = [&](int &x) { const int v = atoi(val); if (v > 0) x = v; };
        int on = 0;
        if (is("SPLITS")) positive(k.splits);
        else if (is("MIN_CHUNK_TILES")) positive(k.min_chunk_tiles);
        else if (is("TARGET_CTAS")) positive(k.target_ctas);
        else if (is("NO_EARLY_LAUNCH")) { positive(on); k.no_early_launch = on > 0; }
        else if (is("TC_SCHEDULE")) k.stream = !strcmp(val, "stream");
        else if (is("TC_SMALL_ROWS")) k.small_rows = val[0] != '0' ? 1 : 0;
        else if (is("MULTI_BLOCK_PACK")) k.pack = val[0] != '0';
    }
    return k;
}
bool early_launch_allowed() { return !read_knobs().no_early_launch; }

}  // namespace orthrus

int orthrus::num_sms()
{
    constexpr int kMaxDevices = 64;
    static std::atomic<int> cached[kMaxDevices];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        (void)cudaGetLastError();
        return kDefaultSMs;
    }
    int n = cached[dev].load(std::memory_order_relaxed);
    if (n > 0) return n;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) {
        (void)cudaGetLastError();
        return kDefaultSMs;
    }
    cached[dev].store(n, std::memory_order_relaxed);
    return n;
}

// What the query below asks for: the occupancy of an attention kernel's cluster without its tensor memory, for which the runtime
// counts one CTA per SM whatever it allocates.  (Clusters of 5, 6, 8, 10, 11, 12, 13 and 14 with two CTAs per SM: 56, 45, 33,
// 26, 21, 21, 17 and 14 by this query, and measured to run in one wave up to there; half-sized clusters with an SM each,
// asked before, say 52, 45, 33, 26, 22, 22, 15 and 15.)
__global__ void __launch_bounds__(320) cluster_probe_kernel() {}

int orthrus::clusters_resident(int S, int per_sm)
{
    constexpr int kMaxDevices = 64, kMaxCluster = 16, kBytes[2] = {200 * 1024, 113 * 1024};
    static std::atomic<int> cached[2][kMaxDevices][kMaxCluster + 1];      // 0: not asked; else the number plus one
    int dev = 0;
    if (S < 1 || S > kMaxCluster || per_sm < 1 || per_sm > 2) return 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        (void)cudaGetLastError();
        return per_sm * kDefaultSMs / S;
    }
    std::atomic<int> &known = cached[per_sm - 1][dev][S];
    int n = known.load(std::memory_order_relaxed);
    if (n > 0) return n - 1;
    n = per_sm * num_sms();
    if (S > 1) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(S);
        cfg.blockDim = dim3(320);
        cfg.dynamicSmemBytes = kBytes[per_sm - 1];
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = S; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (cudaFuncSetAttribute(cluster_probe_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBytes[0]) != cudaSuccess ||
            cudaFuncSetAttribute(cluster_probe_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&n, cluster_probe_kernel, &cfg) != cudaSuccess || n < 1) {
            (void)cudaGetLastError();
            n = S <= 8 ? num_sms() / S : 0;           // a size the device cannot schedule is not chosen
        }
    }
    known.store(n + 1, std::memory_order_relaxed);
    return n;
}

namespace orthrus {

static bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

static orthrus_status_t check_layer(const orthrus_layer_t *L)
{
    if (!L) return ORTHRUS_ERR_INVALID_ARG;
    if (L->batch < 1 || L->n_q_heads < 1 || L->n_kv_heads < 1 || L->block < 1 || L->capacity < 1)
        return ORTHRUS_ERR_INVALID_ARG;
    if (L->n_q_heads % L->n_kv_heads != 0) return ORTHRUS_ERR_INVALID_ARG;
    if (L->dtype != ORTHRUS_BF16 && L->dtype != ORTHRUS_FP32) return ORTHRUS_ERR_UNSUPPORTED;
    if (L->head_dim != 32 && L->head_dim != 64 && L->head_dim != 128 && L->head_dim != 256)
        return ORTHRUS_ERR_UNSUPPORTED;
    if (L->block > 64) return ORTHRUS_ERR_UNSUPPORTED;
    if (L->max_len_hint < 0 || !(L->softmax_scale >= 0.f) || std::isinf(L->softmax_scale))
        return ORTHRUS_ERR_INVALID_ARG;
    if (L->block > L->capacity) return ORTHRUS_ERR_CAPACITY;
    if (L->capacity > 0x7fffffffLL) return ORTHRUS_ERR_UNSUPPORTED;
    if ((long long)L->max_len_hint + L->block > L->capacity) return ORTHRUS_ERR_CAPACITY;
    if (L->flags & ~(uint32_t)(ORTHRUS_LAYER_CACHE_QUIESCENT | ORTHRUS_LAYER_NO_EARLY_LAUNCH |
                               ORTHRUS_LAYER_BLOCK_IN_CACHE))
        return ORTHRUS_ERR_INVALID_ARG;
    return ORTHRUS_OK;
}

static int max_len_of(const orthrus_layer_t *L)
{
    return L->max_len_hint > 0 ? L->max_len_hint : (int)(L->capacity - L->block);
}

// Split-KV plan: a pure function of the descriptor, the kernel path and a few tuning
// variables read from the environment, so that the workspace query and the launch agree.
struct Plan { int chunk, n_splits, tile; };

static bool tc_shape(const orthrus_layer_t *L)
{
    return L->dtype == ORTHRUS_BF16 && L->head_dim == 128 && L->block <= 64 &&
           tc_row_tiles(L->n_q_heads / L->n_kv_heads, L->block) > 0;
}

// The tcgen05 path as a whole: the shape, the row count a 2-D tensor map can index and a
// driver that offers the tensor-map encoder.  Anything else plans and launches on mma / SIMT.
static bool tc_usable(const orthrus_layer_t *L)
{
    if (!tc_shape(L)) return false;
    const unsigned long long rows = (unsigned long long)L->batch * L->n_kv_heads * (unsigned long long)L->capacity;
    return rows < 0x7fffffffull && tc_driver_ok();
}

// ORTHRUS_TC_SCHEDULE=stream (read at every call) selects the persistent kernel, which cuts the
// work by tiles instead of by units, for the shapes it serves; it was measured slower than the
// cluster kernel and is a measurement knob.  A forced split count keeps the cluster kernel.
static bool tc_use_stream(const orthrus_layer_t *L, const Knobs &kn)
{
    return kn.stream && kn.splits == 0 && tc_usable(L) &&
           tc_stream_shape(L->batch, L->n_q_heads / L->n_kv_heads, L->block);
}
static int tc_stream_ctas() { return tc_ctas_per_sm(1) * num_sms(); }

static Plan make_plan(const orthrus_layer_t *L, bool tc, const Knobs &kn)
{
    const int max_len = max_len_of(L);
    const int forced = kn.splits;
    Plan pl;
    if (tc) {
        // The splits of a unit are the CTAs of one thread-block cluster (<= 16).  Few units:
        // as many splits as still fit on the GPU in one wave.  Many units: just enough CTAs
        // to fill every slot once; sequences of unequal length are handed out longest first.
        const int tn = tc_tile_positions();
        const int G = L->n_q_heads / L->n_kv_heads, nt = tc_tiles_per_cta(G, L->block);
        const int units = L->batch * L->n_kv_heads * tc_cta_groups(G, L->block);
        const int slots = tc_ctas_per_sm(nt) * num_sms();
        const int tiles = max_len > 0 ? (max_len + tn - 1) / tn : 1;
        int S = 1;
        if (forced > 0) {
            S = forced;
        } else if (units * 2 <= slots) {
            // Up to four CTAs for a tile each where they leave most SMs idle (8 units of 300 keys 7.6 us
            // a call at 4, 8.1 at 2).  Sixteen only with an SM for each CTA: clusters of that size do not
            // fill the second places (16 units of 4000 keys 16.2 us at 8, 23.2 at 16; of 16000 keys
            // 40 and 45).
            while (S < 16 && units * S * 2 <= (S == 8 ? num_sms() : slots) &&
                   tiles / (S * 2) >= (S < 4 && units * 8 <= num_sms() ? 1 : kn.min_chunk_tiles)) S *= 2;
        } else {
            // (a lone CTA streams slower than an SM's share of HBM, so the longest unit is
            //  still split; many small CTAs would spend their time starting and merging)
            while (S < 16 && units * S < slots && tiles / (S * 2) >= 8) S *= 2;
        }
        // Sixteen only where every cluster finds SMs of its own (up to 7 units on a B200; a cluster stays within a GPC): on shared ones
        // the CTAs of a cluster share the way to the others, which the merge fills.  Else the largest size that does and has a
        // merge of its own (128 rows, 8 units of 2000, 4000, 8000 and 16000 keys 11.6, 12.9, 16.9 and 25.7 us at 16, 8.9, 11.1, 15.4 and
        // 25.3 at 10; 6 units of 8000 13.1 at 16, 15.8 at 10), until streaming the keys is nearly all there is (24000 keys 34.5 and 34.9; 64
        // rows, 2000 and 4000 keys 8.3 and 9.9 at 16, 7.8 and 10.1 at 10).  Behind a rotary write, whose CTAs are in between, 128 rows
        // and clusters of 10 do not go together (4000, 8000 and 16000 keys 14.1, 20.0 and 32.0 at 8, 16.5, 22.8 and 35.3 at 10, 15.6, 19.1
        // and 27.5 at 16).
        const int rows = G * L->block;
        const bool behind_write = (L->flags & ORTHRUS_LAYER_BLOCK_IN_CACHE) && rows > 96;
        if (forced <= 0 && S == 16 && units > clusters_resident(16, 1) &&
            tiles < (behind_write ? 112 : rows > 96 ? 320 : rows > 64 ? 64 : 48))
            S = units <= clusters_resident(10, 1) && !behind_write ? 10 : 8;
        const int max_cluster = tc_max_cluster(nt);
        if (S > max_cluster) S = max_cluster;
        if (S > tiles) S = tiles;
        if (S > 12 && S < 16) S = 12;             // (the merge shares 128 columns out by eights; its buffer)
        if (S < 1) S = 1;
        pl.n_splits = S;
        pl.chunk = ((tiles + S - 1) / S) * tn;
        pl.tile = tn;
        return pl;
    }
    const int granule = 128;
    const int units = L->batch * L->n_kv_heads;
    const int tiles = max_len > 0 ? (max_len + granule - 1) / granule : 1;
    const int target = kn.target_ctas > 0 ? kn.target_ctas : 2 * num_sms();
    const int min_chunk_tiles = kn.min_chunk_tiles;
    int splits = (target + units - 1) / units;
    if (forced > 0) splits = forced;
    int max_splits = forced > 0 ? tiles : tiles / min_chunk_tiles;
    if (max_splits < 1) max_splits = 1;
    if (max_splits > kMaxSplits) max_splits = kMaxSplits;
    if (splits > max_splits) splits = max_splits;
    if (splits < 1) splits = 1;
    const int chunk_tiles = (tiles + splits - 1) / splits;
    pl.chunk = chunk_tiles * granule;
    pl.n_splits = max_len > 0 ? (max_len + pl.chunk - 1) / pl.chunk : 1;
    pl.tile = granule;
    return pl;
}

// 33 to 64 query rows at head_dim 128 can run on either tcgen05 kernel: with the keys on the MMA's rows
// (attend_keys.cu) or with the query rows there, padded to 128 (attend_tc.cu, the wide kernel).  (Us a call, keys against wide, 64 rows.)
//  - Prefixes of one tile of 64 keys at most: the wide kernel, which needs no merge for them (8 units of 64 keys 5.3 and 4.4).
//  - Where the caller promises a quiescent cache, the keys kernel has its first three tiles in shared memory by the time the
//    query rows come, and is the rule while three CTAs a unit have an SM each (8 units of 500, 1000, 2000, 4000 and 8000 keys 5.4 and
//    6.2, 5.5 and 6.6, 6.3 and 7.7, 8.7 and 9.9, 13.5 and 13.5; 16 of 2000 8.8 and 9.6; 40 of 4000 18.7 and 21.2; 48 of 2000 14.2 and 14.2;
//    but 28 to 33, whom the wide kernel's clusters of 8 suit, 32 of 2000 11.8 and 11.0, kept for the reason at the end).  With more
//    units the SMs are full in any case, and the wide kernel takes less per key (56 of 1000 11.6 and 10.0, 64 of 2000 16.4 and 15.1).  A
//    few tiles a unit do not pay for its merge from 9 units on (12 of 300 keys 5.8 and 5.4; 8 level), unless the rows do not fill warps
//    of 32, which costs the wide kernel a second way through its softmax (12 of 300 keys, 48 rows, 5.3 and 5.4).  From 24 units on
//    only with bounds of 1024 keys and more: below, the two are level where the lengths reach the bound, and the wide one is the faster
//    where they do not.
//  - Without the promise every load waits for the preceding kernel.  Up to 9 units the keys kernel is the faster one from 512 keys on while
//    sixteen CTAs have two tiles each or fewer (8 units of 700 keys 6.4 and 6.7, of 2000 8.0 and 8.5, of 3500 10.3 and 10.4; of 300 6.2
//    and 5.8, of 4096 11.8 and 10.8).  Else the wide kernel is the rule where its plan, whose clusters are mostly powers of two, suits
//    the number of units: not where its clusters are not all resident (36 units of 1500 keys cut in 8 11.8 and 16.9), nor where clusters
//    of 4 or 8 leave more than two fifths of the places empty (10 to 22 and 38 to 44 units) and the prefix is long (12 units of
//    8000 keys 15.4 and 17.7, 44 of 6000 26.5 and 30.8); rows that do not fill warps of 32 draw that line lower.
//    Where clusters of 8 fill the grid (23 to 33 units), bounds of 1537 to 3072 keys go to the keys kernel, on which a width-1 step
//    (M <= 32) runs too: it rounds the same probabilities and sums the same rounded ones (32 units of 2000 13.0 and 11.9).
// So the promise decides which kernel serves some calls, and with it their rounding: see the flag in orthrus.h.
static bool wide_better(const orthrus_layer_t *L, const Knobs &kn)
{
    if (!tc_usable(L)) return false;
    const int units = L->batch * L->n_kv_heads, M = L->n_q_heads / L->n_kv_heads * L->block, max_len = max_len_of(L);
    if (max_len <= tc_tile_positions()) return true;
    if ((L->flags & ORTHRUS_LAYER_CACHE_QUIESCENT) && 3 * units <= num_sms()) {
        if (25 * units <= 4 * num_sms()) return M == 64 && max_len <= 384 && 17 * units > num_sms();      // to 23 units, from 9 on
        if (max_len >= 1024) return false;
    }
    constexpr int kTwoTiles = 16 * 2 * 128 - 64;              // two tiles for each of sixteen CTAs, but for the block's half
    if (16 * units <= num_sms() && max_len > 512 && max_len + L->block <= kTwoTiles) return false;
    const int S = make_plan(L, true, kn).n_splits;
    if (S > 1 && units > clusters_resident(S, 2)) return false;   // (the two kernels' CTAs fit an SM alike)
    const bool roomy = 5 * units * S < 3 * tc_ctas_per_sm(1) * num_sms();
    if (S == 8 && !roomy) return max_len <= 1536 || max_len > 3072;
    return !((S == 4 || S == 8) && roomy && max_len > (M == 64 ? 4096 : 2048));
}

static int keys_tiles(const orthrus_layer_t *L)
{
    const int kb = keys_kb_rows(L->head_dim, L->n_q_heads / L->n_kv_heads, L->block);
    return (L->block + kb - 1) / kb;
}

// Units of at most 32 query rows (4 rows, 8 units of 4000 keys 5.7 against 9.7 us on the wide kernel, 32 rows 6.9), of 33
// to 64 by the rule above, and of any number at head_dim 64 run with the keys on the MMA's
// rows.  ORTHRUS_TC_SMALL_ROWS=0 keeps them on the other kernels, =1 puts there whatever fits but 65 to 128 rows at
// head_dim 128, which then stay on the wide kernel (measurement knobs).
// 65 to 128 rows at head_dim 128 are two tiles there, which read the same keys: the faster way where latency counts, that is, with
// the promise of a quiescent cache, while nine CTAs a tile have SMs (up to 16 tiles), and up to 8192 keys (keys against wide, 128 rows: 4 units of 700, 2000 and 8000 keys 5.4
// and 7.2 us, 6.3 and 8.7, 13.1 and 13.0; 8 units 6.3 and 7.2, 8.9 and 8.8, 15.5 and 15.4; of 64 keys 5.3 and 5.2).
// Wide units at head_dim 64 with short prefixes stay on mma.sync: a CTA of 128 rows has an SM to itself
// and takes about 9 us before its first key (128 units of 128 rows, bound 150, 9.3 against 12.1 us;
// from 400 on it is the better one: 29 against 16 us, bound 2000 60 against 38 us).
static bool keys_usable(const orthrus_layer_t *L, const Knobs &kn)
{
    if (L->dtype != ORTHRUS_BF16 || (L->head_dim != 64 && L->head_dim != 128) || kn.small_rows == 0) return false;
    const int rows = keys_rows(L->head_dim, L->n_q_heads / L->n_kv_heads, L->block);
    const unsigned long long cache = (unsigned long long)L->batch * L->n_kv_heads * (unsigned long long)L->capacity;
    if (!rows || cache >= 0x7fffffffull || L->batch > 65535 || (long long)L->n_kv_heads * keys_tiles(L) > 65535 || !tc_driver_ok()) return false;
    const int M = L->n_q_heads / L->n_kv_heads * L->block, units = L->batch * L->n_kv_heads;
    if (L->head_dim == 128 && M > 64)
        return kn.small_rows < 0 && (L->flags & ORTHRUS_LAYER_CACHE_QUIESCENT) && 9 * units * keys_tiles(L) <= num_sms() &&
               max_len_of(L) > tc_tile_positions() && max_len_of(L) <= 8192;
    if (kn.small_rows > 0) return true;
    if (rows > 64) return max_len_of(L) > 320;
    return rows < 64 || L->head_dim == 64 || !wide_better(L, kn);
}
static int keys_plan(const orthrus_layer_t *L, const Knobs &kn, bool *apart)
{
    *apart = false;
    if (kn.splits > 0) return kn.splits < 16 ? kn.splits : 16;
    return keys_splits(L->head_dim, L->n_q_heads / L->n_kv_heads, L->block, L->batch * L->n_kv_heads * keys_tiles(L),
                       max_len_of(L), apart);
}
// Split partials of the mma and SIMT paths (the tcgen05 kernels merge through shared memory)
static size_t partial_bytes(const orthrus_layer_t *L, const Plan &pl, size_t *ml_off)
{
    if (ml_off) *ml_off = 0;
    if (pl.n_splits == 1) return 0;
    const size_t units = (size_t)L->batch * L->n_kv_heads, M = (size_t)(L->n_q_heads / L->n_kv_heads) * L->block;
    const size_t o_bytes = units * pl.n_splits * M * L->head_dim * sizeof(float);
    const size_t ml_bytes = units * pl.n_splits * M * 2 * sizeof(float);
    if (ml_off) *ml_off = o_bytes;
    return o_bytes + ml_bytes;
}

// nb: blocks per sequence (the batch of *L then counts blocks, and batch entry b reads the cache
// of sequence b / nb)
static orthrus_status_t attend(const orthrus_layer_t *L, int causal, const void *q,
                               const void *k_blk, const void *v_blk, void *out, void *ws,
                               size_t ws_bytes, void *stream, int nb = 1)
{
    orthrus_status_t st = check_layer(L);
    if (st != ORTHRUS_OK) return st;
    const bool in_cache = (L->flags & ORTHRUS_LAYER_BLOCK_IN_CACHE) != 0;
    if (in_cache) k_blk = v_blk = nullptr;    // not read in this mode
    if (!q || (!in_cache && (!k_blk || !v_blk)) || !out || !ws || !L->k_cache || !L->v_cache || !L->cache_len)
        return ORTHRUS_ERR_INVALID_ARG;
    if (!aligned16(q) || !aligned16(k_blk) || !aligned16(v_blk) || !aligned16(out) ||
        !aligned16(ws) || !aligned16(L->k_cache) || !aligned16(L->v_cache) ||
        (reinterpret_cast<uintptr_t>(L->cache_len) & 3))
        return ORTHRUS_ERR_INVALID_ARG;
    const int want = current_path();
    const bool tc = (want == PATH_AUTO || want == PATH_TCGEN05) && tc_usable(L);
    const Knobs kn = read_knobs();
    const bool stream_k = tc && tc_use_stream(L, kn);
    Plan pl = make_plan(L, tc, kn);
    if (stream_k) pl.n_splits = 1;
    size_t ml_off = 0;
    const bool keys = !stream_k && (want == PATH_AUTO || (want == PATH_TCGEN05 && tc)) && keys_usable(L, kn);
    bool apart = false;
    if (keys) pl.n_splits = keys_plan(L, kn, &apart);
    const size_t need = kHeaderBytes + (stream_k ? tc_stream_workspace_bytes(L->batch, L->n_kv_heads, tc_stream_ctas())
                                        : keys || tc ? 0 : partial_bytes(L, pl, &ml_off));
    if (ws_bytes < need) return ORTHRUS_ERR_WORKSPACE;

    AttnParams p;
    p.q = q; p.k_blk = k_blk; p.v_blk = v_blk; p.k_cache = L->k_cache; p.v_cache = L->v_cache;
    p.cache_len = L->cache_len; p.out = out;
    unsigned char *base = static_cast<unsigned char *>(ws);
    p.status = reinterpret_cast<int32_t *>(base);
    p.part_o = reinterpret_cast<float *>(base + kHeaderBytes);
    p.part_ml = reinterpret_cast<float *>(base + kHeaderBytes + ml_off);
    p.B = L->batch; p.K = L->block; p.Hq = L->n_q_heads; p.Hkv = L->n_kv_heads;
    p.G = p.Hq / p.Hkv; p.M = p.G * p.K; p.d = L->head_dim; p.capacity = L->capacity;
    p.chunk = pl.chunk; p.n_splits = pl.n_splits; p.causal = causal;
    p.blk_in_cache = in_cache ? 1 : 0;
    p.nb = nb; p.kb_width = 0; p.len_cap = L->capacity - L->block;
    const float scale = L->softmax_scale > 0.f ? L->softmax_scale : 1.f / sqrtf((float)p.d);
    p.scale_log2 = scale * 1.4426950408889634f;

    int flags = (int)(L->flags & (ORTHRUS_LAYER_CACHE_QUIESCENT | ORTHRUS_LAYER_NO_EARLY_LAUNCH));
    if (kn.no_early_launch) flags |= ORTHRUS_LAYER_NO_EARLY_LAUNCH;
    p.apart = apart;
    p.early = !(flags & ORTHRUS_LAYER_NO_EARLY_LAUNCH);

    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    cudaError_t e;
    bool merge_kernel = pl.n_splits > 1;
    if (keys) {
        t_last_path = "tcgen05";
        e = launch_attend_keys(p, flags, cs);
        merge_kernel = false;
    } else if (tc) {
        t_last_path = "tcgen05";
        if (stream_k) e = launch_attend_tc_stream(p, tc_stream_ctas(), base + kHeaderBytes, flags, cs);
        else e = launch_attend_tc(p, flags, cs);
        merge_kernel = false;
    } else if (want != PATH_SIMT && mma_path_supports(p, L->dtype)) {
        t_last_path = "mma";
        e = launch_attend_mma(p, cs);
    } else {
        t_last_path = "simt";
        e = launch_attend_simt(p, L->dtype, cs);
    }
    if (e != cudaSuccess) return ORTHRUS_ERR_CUDA;
    if (merge_kernel) {
        e = launch_combine(p, L->dtype, cs);
        if (e != cudaSuccess) return ORTHRUS_ERR_CUDA;
    }
    return ORTHRUS_OK;
}

}  // namespace orthrus

using namespace orthrus;

extern "C" {

size_t orthrus_attend_workspace_bytes(const orthrus_layer_t *layer)
{
    if (check_layer(layer) != ORTHRUS_OK) return 0;
    // enough for whichever kernel path a later call resolves to
    const Knobs kn = read_knobs();
    size_t need = partial_bytes(layer, make_plan(layer, false, kn), nullptr);
    if (tc_usable(layer) && tc_use_stream(layer, kn)) {
        const size_t n3 = tc_stream_workspace_bytes(layer->batch, layer->n_kv_heads, tc_stream_ctas());
        if (n3 > need) need = n3;
    }
    return kHeaderBytes + need;
}

orthrus_status_t orthrus_workspace_init(void *workspace, size_t workspace_bytes, void *stream)
{
    if (!workspace || workspace_bytes < (size_t)kHeaderBytes) return ORTHRUS_ERR_INVALID_ARG;
    // all of it: besides the status word, the arrival counters some kernels keep there must start at zero
    return cudaMemsetAsync(workspace, 0, workspace_bytes, static_cast<cudaStream_t>(stream)) == cudaSuccess
               ? ORTHRUS_OK : ORTHRUS_ERR_CUDA;
}

orthrus_status_t orthrus_diffusion_block_attend(const orthrus_layer_t *layer, const void *q_diff,
        const void *k_diff_blk, const void *v_diff_blk, void *out, void *workspace,
        size_t workspace_bytes, void *stream)
{
    return attend(layer, 0, q_diff, k_diff_blk, v_diff_blk, out, workspace, workspace_bytes, stream);
}

orthrus_status_t orthrus_ar_verify_attend(const orthrus_layer_t *layer, const void *q_ar,
        const void *k_ar_blk, const void *v_ar_blk, void *out, void *workspace,
        size_t workspace_bytes, void *stream)
{
    return attend(layer, 1, q_ar, k_ar_blk, v_ar_blk, out, workspace, workspace_bytes, stream);
}

// Eq. 6 as a batch of blocks: the descriptor of S sequences becomes one of S * n_blocks batch
// entries whose prefix lengths are the anchors; entry b reads the cache of sequence b / n_blocks.
static bool multi_block_layer(const orthrus_layer_t *layer, int32_t n_blocks, const int32_t *anchors,
                              orthrus_layer_t *out)
{
    if (!layer || n_blocks < 1 || layer->batch < 1 || (long long)layer->batch * n_blocks > 0x7fffffffLL) return false;
    *out = *layer;
    out->batch = layer->batch * n_blocks;
    out->cache_len = const_cast<int32_t *>(anchors);
    out->flags = layer->flags & ~(uint32_t)ORTHRUS_LAYER_BLOCK_IN_CACHE;
    return true;
}

// The packed form of Eq. 6 (tcgen05 path): the blocks of a sequence share 128-row query tiles, so
// the prefix is streamed once per tile instead of once per block.  Taken when at least two blocks
// fit one tile; ORTHRUS_MULTI_BLOCK_PACK=0 keeps the one-unit-per-block form (a measurement knob).
static bool multi_block_packed(const orthrus_layer_t *layer, int32_t n_blocks, const Knobs &kn)
{
    if (n_blocks < 2 || check_layer(layer) != ORTHRUS_OK || !tc_usable(layer)) return false;
    const int want = current_path();
    if (want != PATH_AUTO && want != PATH_TCGEN05) return false;
    if (2 * (layer->n_q_heads / layer->n_kv_heads) * layer->block > 128) return false;
    if ((long long)n_blocks * layer->block > (1 << 20)) return false;
    return kn.pack;
}

// the descriptor the packed form plans with: one "block" of n_blocks * K positions per sequence
static orthrus_layer_t packed_layer(const orthrus_layer_t *layer, int32_t n_blocks)
{
    orthrus_layer_t L = *layer;
    L.max_len_hint = max_len_of(layer);
    L.block = n_blocks * layer->block;
    L.flags = layer->flags & ~(uint32_t)ORTHRUS_LAYER_BLOCK_IN_CACHE;
    return L;
}

static orthrus_status_t attend_packed(const orthrus_layer_t *layer, int32_t n_blocks, const int32_t *anchors,
                                      const void *q, const void *k_blk, const void *v_blk, void *out,
                                      void *ws, size_t ws_bytes, void *stream, const Knobs &kn)
{
    if (!q || !k_blk || !v_blk || !out || !ws || !layer->k_cache || !layer->v_cache) return ORTHRUS_ERR_INVALID_ARG;
    if (!aligned16(q) || !aligned16(k_blk) || !aligned16(v_blk) || !aligned16(out) || !aligned16(ws) ||
        !aligned16(layer->k_cache) || !aligned16(layer->v_cache) || (reinterpret_cast<uintptr_t>(anchors) & 3))
        return ORTHRUS_ERR_INVALID_ARG;
    const orthrus_layer_t L = packed_layer(layer, n_blocks);
    const Plan pl = make_plan(&L, true, kn);
    if (ws_bytes < (size_t)kHeaderBytes) return ORTHRUS_ERR_WORKSPACE;

    AttnParams p;
    p.q = q; p.k_blk = k_blk; p.v_blk = v_blk; p.k_cache = layer->k_cache; p.v_cache = layer->v_cache;
    p.cache_len = anchors; p.out = out;
    unsigned char *base = static_cast<unsigned char *>(ws);
    p.status = reinterpret_cast<int32_t *>(base);
    p.part_o = p.part_ml = nullptr;
    p.B = layer->batch; p.K = L.block; p.Hq = layer->n_q_heads; p.Hkv = layer->n_kv_heads;
    p.G = p.Hq / p.Hkv; p.M = p.G * p.K; p.d = layer->head_dim; p.capacity = layer->capacity;
    p.chunk = pl.chunk; p.n_splits = pl.n_splits; p.causal = 0; p.blk_in_cache = 0;
    p.nb = n_blocks; p.kb_width = layer->block; p.len_cap = layer->capacity - layer->block;
    const float scale = layer->softmax_scale > 0.f ? layer->softmax_scale : 1.f / sqrtf((float)p.d);
    p.scale_log2 = scale * 1.4426950408889634f;
    t_last_path = "tcgen05";
    int flags = (int)(layer->flags & (ORTHRUS_LAYER_CACHE_QUIESCENT | ORTHRUS_LAYER_NO_EARLY_LAUNCH));
    if (kn.no_early_launch) flags |= ORTHRUS_LAYER_NO_EARLY_LAUNCH;
    p.apart = 0;
    p.early = !(flags & ORTHRUS_LAYER_NO_EARLY_LAUNCH);
    return launch_attend_tc_packed(p, flags, static_cast<cudaStream_t>(stream)) == cudaSuccess
               ? ORTHRUS_OK : ORTHRUS_ERR_CUDA;
}

size_t orthrus_multi_block_workspace_bytes(const orthrus_layer_t *layer, int32_t n_blocks)
{
    orthrus_layer_t L;
    if (!multi_block_layer(layer, n_blocks, nullptr, &L)) return 0;
    // enough for either form (the packed one needs the header alone)
    return orthrus_attend_workspace_bytes(&L);
}

orthrus_status_t orthrus_multi_block_attend(const orthrus_layer_t *layer, int32_t n_blocks,
        const int32_t *anchors, const void *q_diff, const void *k_diff_blk, const void *v_diff_blk,
        void *out, void *workspace, size_t workspace_bytes, void *stream)
{
    orthrus_layer_t L;
    if (!anchors || !multi_block_layer(layer, n_blocks, anchors, &L)) return ORTHRUS_ERR_INVALID_ARG;
    if (layer->flags & ORTHRUS_LAYER_BLOCK_IN_CACHE) return ORTHRUS_ERR_INVALID_ARG;
    const Knobs kn = read_knobs();
    if (multi_block_packed(layer, n_blocks, kn))
        return attend_packed(layer, n_blocks, anchors, q_diff, k_diff_blk, v_diff_blk, out, workspace,
                             workspace_bytes, stream, kn);
    return attend(&L, 0, q_diff, k_diff_blk, v_diff_blk, out, workspace, workspace_bytes, stream, n_blocks);
}

size_t orthrus_consensus_workspace_bytes(int32_t batch, int32_t block, int32_t vocab)
{
    if (batch < 1 || block < 1 || vocab < 1) return 0;
    return kHeaderBytes + (size_t)batch * block * consensus_segments(batch, block, vocab) * 8;
}

orthrus_status_t orthrus_consensus_accept(const void *ar_logits, int32_t dtype, const int32_t *draft,
        int32_t batch, int32_t block, int32_t vocab, int32_t *n_commit, int32_t *committed,
        int32_t *ar_argmax, int32_t *next_anchor, void *workspace, size_t workspace_bytes,
        void *stream)
{
    if (batch < 1 || block < 1 || vocab < 1) return ORTHRUS_ERR_INVALID_ARG;
    if (dtype != ORTHRUS_BF16 && dtype != ORTHRUS_FP32) return ORTHRUS_ERR_UNSUPPORTED;
    if (block > 1024 || (long long)batch * block > 65535) return ORTHRUS_ERR_UNSUPPORTED;
    if (!ar_logits || !draft || !n_commit || !committed || !ar_argmax || !next_anchor || !workspace)
        return ORTHRUS_ERR_INVALID_ARG;
    const size_t es = dtype == ORTHRUS_FP32 ? 4 : 2;
    if ((reinterpret_cast<uintptr_t>(ar_logits) & (es - 1)) || !aligned16(workspace) ||
        ((reinterpret_cast<uintptr_t>(draft) | reinterpret_cast<uintptr_t>(n_commit) |
          reinterpret_cast<uintptr_t>(committed) | reinterpret_cast<uintptr_t>(ar_argmax) |
          reinterpret_cast<uintptr_t>(next_anchor)) & 3))
        return ORTHRUS_ERR_INVALID_ARG;
    if (workspace_bytes < orthrus_consensus_workspace_bytes(batch, block, vocab))
        return ORTHRUS_ERR_WORKSPACE;
    const int n_seg = consensus_segments(batch, block, vocab);
    cudaError_t e = launch_consensus(ar_logits, dtype, draft, batch, block, vocab, n_commit, committed,
                                     ar_argmax, next_anchor,
                                     static_cast<unsigned char *>(workspace) + kHeaderBytes, n_seg,
                                     static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? ORTHRUS_OK : ORTHRUS_ERR_CUDA;
}

size_t orthrus_consensus_sample_workspace_bytes(int32_t batch, int32_t block, int32_t vocab)
{
    if (batch < 1 || block < 1 || vocab < 1) return 0;
    return kHeaderBytes + sample_workspace_bytes(batch, block, vocab);
}

orthrus_status_t orthrus_consensus_sample(const void *ar_logits, const void *diff_logits, int32_t dtype,
        const int32_t *draft, const float *u_accept, const float *u_resample, float temperature,
        int32_t batch, int32_t block, int32_t vocab, int32_t *n_commit, int32_t *committed,
        int32_t *next_anchor, void *workspace, size_t workspace_bytes, void *stream)
{
    if (batch < 1 || block < 1 || vocab < 1 || !(temperature > 0.f) || std::isinf(temperature))
        return ORTHRUS_ERR_INVALID_ARG;
    if (dtype != ORTHRUS_BF16 && dtype != ORTHRUS_FP32) return ORTHRUS_ERR_UNSUPPORTED;
    if (block > 1024 || (long long)batch * block > 65535) return ORTHRUS_ERR_UNSUPPORTED;
    if (!ar_logits || !diff_logits || !draft || !u_accept || !u_resample || !n_commit || !committed ||
        !next_anchor || !workspace)
        return ORTHRUS_ERR_INVALID_ARG;
    const size_t es = dtype == ORTHRUS_FP32 ? 4 : 2;
    if (((reinterpret_cast<uintptr_t>(ar_logits) | reinterpret_cast<uintptr_t>(diff_logits)) & (es - 1)) ||
        !aligned16(workspace) ||
        ((reinterpret_cast<uintptr_t>(draft) | reinterpret_cast<uintptr_t>(u_accept) |
          reinterpret_cast<uintptr_t>(u_resample) | reinterpret_cast<uintptr_t>(n_commit) |
          reinterpret_cast<uintptr_t>(committed) | reinterpret_cast<uintptr_t>(next_anchor)) & 3))
        return ORTHRUS_ERR_INVALID_ARG;
    if (workspace_bytes < orthrus_consensus_sample_workspace_bytes(batch, block, vocab))
        return ORTHRUS_ERR_WORKSPACE;
    cudaError_t e = launch_consensus_sample(ar_logits, diff_logits, dtype, draft, u_accept, u_resample,
                                            temperature, batch, block, vocab, n_commit, committed, next_anchor,
                                            static_cast<unsigned char *>(workspace) + kHeaderBytes,
                                            static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? ORTHRUS_OK : ORTHRUS_ERR_CUDA;
}

orthrus_status_t orthrus_consensus_accept_static(const void *ar_logits, int32_t dtype,
        const int32_t *draft, int32_t batch, int32_t block, int32_t vocab, int32_t *n_commit,
        int32_t *committed, int32_t *ar_argmax, int32_t *next_anchor, void *stream)
{
    if (batch < 1 || block < 1 || vocab < 1) return ORTHRUS_ERR_INVALID_ARG;
    if (dtype != ORTHRUS_BF16 && dtype != ORTHRUS_FP32) return ORTHRUS_ERR_UNSUPPORTED;
    if (block > 1024 || (long long)batch * block > 65535) return ORTHRUS_ERR_UNSUPPORTED;
    if (!ar_logits || !draft || !n_commit || !committed || !ar_argmax || !next_anchor)
        return ORTHRUS_ERR_INVALID_ARG;
    const size_t es = dtype == ORTHRUS_FP32 ? 4 : 2;
    if ((reinterpret_cast<uintptr_t>(ar_logits) & (es - 1)) ||
        ((reinterpret_cast<uintptr_t>(draft) | reinterpret_cast<uintptr_t>(n_commit) |
          reinterpret_cast<uintptr_t>(committed) | reinterpret_cast<uintptr_t>(ar_argmax) |
          reinterpret_cast<uintptr_t>(next_anchor)) & 3))
        return ORTHRUS_ERR_INVALID_ARG;
    // the built-in scratch has a fixed size: larger problems need the workspace variant
    if (static_consensus_segments(batch, block, vocab) < 1) return ORTHRUS_ERR_WORKSPACE;
    cudaError_t e = launch_consensus_static(ar_logits, dtype, draft, batch, block, vocab, n_commit,
                                            committed, ar_argmax, next_anchor,
                                            static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? ORTHRUS_OK : ORTHRUS_ERR_CUDA;
}

size_t orthrus_lm_head_consensus_workspace_bytes(int32_t batch, int32_t block, int32_t vocab)
{
    if (batch < 1 || block < 1 || vocab < 1) return 0;
    return kHeaderBytes + (size_t)batch * block * lm_head_max_vocab_tiles(vocab) * sizeof(ArgPart);
}

orthrus_status_t orthrus_lm_head_consensus(const void *hidden, const void *lm_head, int32_t dtype,
        int32_t hidden_dim, const int32_t *draft, int32_t batch, int32_t block, int32_t vocab,
        int32_t *n_commit, int32_t *committed, int32_t *ar_argmax, int32_t *next_anchor,
        void *workspace, size_t workspace_bytes, void *stream)
{
    if (batch < 1 || block < 1 || vocab < 1 || hidden_dim < 1) return ORTHRUS_ERR_INVALID_ARG;
    if (dtype != ORTHRUS_BF16) return ORTHRUS_ERR_UNSUPPORTED;
    if (block > 1024 || (long long)batch * block > 65535 || vocab > (1 << 24) || (hidden_dim & 7))
        return ORTHRUS_ERR_UNSUPPORTED;
    if (!hidden || !lm_head || !draft || !n_commit || !committed || !ar_argmax || !next_anchor || !workspace)
        return ORTHRUS_ERR_INVALID_ARG;
    if (!aligned16(hidden) || !aligned16(lm_head) || !aligned16(workspace) ||
        ((reinterpret_cast<uintptr_t>(draft) | reinterpret_cast<uintptr_t>(n_commit) |
          reinterpret_cast<uintptr_t>(committed) | reinterpret_cast<uintptr_t>(ar_argmax) |
          reinterpret_cast<uintptr_t>(next_anchor)) & 3))
        return ORTHRUS_ERR_INVALID_ARG;
    if (workspace_bytes < orthrus_lm_head_consensus_workspace_bytes(batch, block, vocab))
        return ORTHRUS_ERR_WORKSPACE;
    if (!lm_head_supported()) return ORTHRUS_ERR_UNSUPPORTED;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    ArgPart *parts = reinterpret_cast<ArgPart *>(static_cast<unsigned char *>(workspace) + kHeaderBytes);
    cudaError_t e = launch_lm_head_argmax(hidden, lm_head, batch * block, vocab, hidden_dim, parts,
                                          static_cast<int32_t *>(workspace), st);
    if (e == cudaErrorNotSupported) return ORTHRUS_ERR_UNSUPPORTED;
    if (e == cudaSuccess)
        e = launch_consensus_finalize(parts, lm_head_vocab_tiles(batch * block, vocab), draft, batch, block, n_commit,
                                           committed, ar_argmax, next_anchor, st);
    return e == cudaSuccess ? ORTHRUS_OK : ORTHRUS_ERR_CUDA;
}

orthrus_status_t orthrus_kv_append(const orthrus_layer_t *layer, const void *k_ar_blk,
        const void *v_ar_blk, const int32_t *n_commit, int32_t update_len, void *workspace,
        size_t workspace_bytes, void *stream)
{
    orthrus_status_t st = check_layer(layer);
    if (st != ORTHRUS_OK) return st;
    if (!k_ar_blk || !v_ar_blk || !n_commit || !layer->k_cache || !layer->v_cache || !layer->cache_len)
        return ORTHRUS_ERR_INVALID_ARG;
    if (!aligned16(k_ar_blk) || !aligned16(v_ar_blk) || !aligned16(layer->k_cache) ||
        !aligned16(layer->v_cache) || (reinterpret_cast<uintptr_t>(n_commit) & 3) ||
        (reinterpret_cast<uintptr_t>(layer->cache_len) & 3))
        return ORTHRUS_ERR_INVALID_ARG;
    if (workspace && (workspace_bytes < (size_t)kHeaderBytes || !aligned16(workspace)))
        return ORTHRUS_ERR_WORKSPACE;
    cudaError_t e = launch_kv_append(*layer, k_ar_blk, v_ar_blk, n_commit, update_len,
                                     static_cast<int32_t *>(workspace),
                                     static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? ORTHRUS_OK : ORTHRUS_ERR_CUDA;
}

static orthrus_status_t check_block_call(const orthrus_layer_t *layer, void *workspace, size_t workspace_bytes)
{
    const orthrus_status_t st = check_layer(layer);
    if (st != ORTHRUS_OK) return st;
    if (!layer->k_cache || !layer->v_cache || !layer->cache_len) return ORTHRUS_ERR_INVALID_ARG;
    if (!aligned16(layer->k_cache) || !aligned16(layer->v_cache) ||
        (reinterpret_cast<uintptr_t>(layer->cache_len) & 3))
        return ORTHRUS_ERR_INVALID_ARG;
    if (workspace && (workspace_bytes < (size_t)kHeaderBytes || !aligned16(workspace)))
        return ORTHRUS_ERR_WORKSPACE;
    return ORTHRUS_OK;
}

orthrus_status_t orthrus_block_kv_write(const orthrus_layer_t *layer, const void *k_blk, const void *v_blk,
        void *workspace, size_t workspace_bytes, void *stream)
{
    const orthrus_status_t st = check_block_call(layer, workspace, workspace_bytes);
    if (st != ORTHRUS_OK) return st;
    if (!k_blk || !v_blk || !aligned16(k_blk) || !aligned16(v_blk)) return ORTHRUS_ERR_INVALID_ARG;
    cudaError_t e = launch_block_kv_write(*layer, k_blk, v_blk, static_cast<int32_t *>(workspace),
                                          static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? ORTHRUS_OK : ORTHRUS_ERR_CUDA;
}

orthrus_status_t orthrus_commit_len(const orthrus_layer_t *layer, const int32_t *n_commit,
        void *workspace, size_t workspace_bytes, void *stream)
{
    const orthrus_status_t st = check_block_call(layer, workspace, workspace_bytes);
    if (st != ORTHRUS_OK) return st;
    if (!n_commit || (reinterpret_cast<uintptr_t>(n_commit) & 3)) return ORTHRUS_ERR_INVALID_ARG;
    cudaError_t e = launch_commit_len(*layer, n_commit, static_cast<int32_t *>(workspace),
                                      static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? ORTHRUS_OK : ORTHRUS_ERR_CUDA;
}

orthrus_status_t orthrus_rope_block_kv_write(const orthrus_layer_t *layer, const void *q, const void *k_blk,
        const void *v_blk, float rope_theta, void *q_out, void *workspace, size_t workspace_bytes, void *stream)
{
    const orthrus_status_t st = check_block_call(layer, workspace, workspace_bytes);
    if (st != ORTHRUS_OK) return st;
    if (!q || !k_blk || !v_blk || !q_out || !aligned16(q) || !aligned16(k_blk) || !aligned16(v_blk) ||
        !aligned16(q_out) || !(rope_theta > 0.f) || std::isinf(rope_theta))
        return ORTHRUS_ERR_INVALID_ARG;
    cudaError_t e = launch_rope_block_kv_write(*layer, q, k_blk, v_blk, (double)rope_theta, q_out,
                                               static_cast<int32_t *>(workspace),
                                               static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? ORTHRUS_OK : ORTHRUS_ERR_CUDA;
}

orthrus_status_t orthrus_kv_append_layers(const orthrus_layer_t *layers, int32_t n_layers,
        const void *const *k_ar_blks, const void *const *v_ar_blks, const int32_t *n_commit,
        int32_t update_len, void *workspace, size_t workspace_bytes, void *stream)
{
    if (!layers || !k_ar_blks || !v_ar_blks || !n_commit || n_layers < 1 || n_layers > 128)
        return ORTHRUS_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(n_commit) & 3) return ORTHRUS_ERR_INVALID_ARG;
    if (workspace && (workspace_bytes < (size_t)kHeaderBytes || !aligned16(workspace)))
        return ORTHRUS_ERR_WORKSPACE;
    AppendLayer al[128];
    int32_t *lens[128];
    int n_lens = 0;
    const orthrus_layer_t &L0 = layers[0];
    for (int l = 0; l < n_layers; ++l) {
        const orthrus_layer_t &L = layers[l];
        const orthrus_status_t st = check_layer(&L);
        if (st != ORTHRUS_OK) return st;
        if (L.batch != L0.batch || L.n_kv_heads != L0.n_kv_heads || L.head_dim != L0.head_dim ||
            L.block != L0.block || L.dtype != L0.dtype || L.capacity != L0.capacity)
            return ORTHRUS_ERR_INVALID_ARG;
        if (!k_ar_blks[l] || !v_ar_blks[l] || !L.k_cache || !L.v_cache || !L.cache_len)
            return ORTHRUS_ERR_INVALID_ARG;
        if (!aligned16(k_ar_blks[l]) || !aligned16(v_ar_blks[l]) || !aligned16(L.k_cache) ||
            !aligned16(L.v_cache) || (reinterpret_cast<uintptr_t>(L.cache_len) & 3))
            return ORTHRUS_ERR_INVALID_ARG;
        al[l] = AppendLayer{L.k_cache, L.v_cache, k_ar_blks[l], v_ar_blks[l], L.cache_len};
        bool seen = false;
        for (int j = 0; j < n_lens; ++j) seen |= lens[j] == L.cache_len;
        if (!seen) lens[n_lens++] = L.cache_len;
    }
    cudaError_t e = launch_kv_append_layers(L0, al, n_layers, lens, update_len ? n_lens : 0, n_commit,
                                            static_cast<int32_t *>(workspace),
                                            static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? ORTHRUS_OK : ORTHRUS_ERR_CUDA;
}

orthrus_status_t orthrus_read_status(const void *workspace, void *stream, int32_t *host_status)
{
    if (!workspace || !host_status) return ORTHRUS_ERR_INVALID_ARG;
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    if (cudaMemcpyAsync(host_status, workspace, sizeof(int32_t), cudaMemcpyDeviceToHost, cs) != cudaSuccess)
        return ORTHRUS_ERR_CUDA;
    if (cudaStreamSynchronize(cs) != cudaSuccess) return ORTHRUS_ERR_CUDA;
    return (*host_status & ORTHRUS_DEV_WAIT_TIMEOUT) ? ORTHRUS_ERR_TIMEOUT : ORTHRUS_OK;
}

orthrus_status_t orthrus_set_path(const char *name)
{
    const int v = parse_path(name);
    if (v < 0) return ORTHRUS_ERR_INVALID_ARG;
    g_path.store(v);
    return ORTHRUS_OK;
}

const char *orthrus_last_path(void) { return t_last_path; }

int64_t orthrus_launch_count(void) { return g_launches.load(); }

const char *orthrus_status_string(orthrus_status_t status)
{
    switch (status) {
    case ORTHRUS_OK: return "ok";
    case ORTHRUS_ERR_INVALID_ARG: return "invalid argument";
    case ORTHRUS_ERR_UNSUPPORTED: return "unsupported shape or dtype";
    case ORTHRUS_ERR_CAPACITY: return "block does not fit in the cache capacity";
    case ORTHRUS_ERR_WORKSPACE: return "workspace too small";
    case ORTHRUS_ERR_CUDA: return "CUDA runtime error";
    case ORTHRUS_ERR_TIMEOUT: return "a bounded wait inside a kernel ran out";
    }
    return "unknown status";
}

int32_t orthrus_version(void) { return 200; }

}  // extern "C"
