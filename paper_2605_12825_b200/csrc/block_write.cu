// The write-then-truncate form of the KV commit and the step in front of it.
//   block_kv_write        every pass puts the K/V rows of its whole block behind the prefix of the
//                         shared cache (rows [P, P + K) of every KV head); the length is left alone,
//                         so those rows are dead until the consensus confirms some of them
//   commit_len            the consensus result only grows the length: len += n_commit
//   rope_block_kv_write   the same write fused with the rotary embedding of the block's queries and
//                         keys (row i of sequence b sits at position P_b + i), so that the projection
//                         outputs go straight to their places: rotated Q to the query tensor the
//                         attention reads, rotated K and V into the cache
// All are copies or a few flops per element: latency-bound launches of a few microseconds.
#include <type_traits>
#include "common.cuh"

namespace orthrus {
namespace {

// grid (B, Hkv): the K destination rows of one KV head are contiguous
__global__ void __launch_bounds__(128) block_kv_write_kernel(
    uint4 *k_cache, uint4 *v_cache, const int32_t *cache_len, const uint4 *k_blk, const uint4 *v_blk,
    int K, int Hkv, int row_vecs, long long capacity, int32_t *status)
{
    pdl_begin();
    const int b = blockIdx.x, h = blockIdx.y;
    const int P = cache_len[b];
    if (P < 0 || (long long)P + K > capacity) {
        if (status && threadIdx.x == 0 && h == 0) atomicOr(status, ORTHRUS_DEV_APPEND_OVERFLOW);
        return;
    }
    const long long dst0 = (((long long)b * Hkv + h) * capacity + P) * row_vecs;
    const int total = K * row_vecs;
    for (int e = threadIdx.x; e < total; e += blockDim.x) {
        const int i = e / row_vecs, c = e - i * row_vecs;
        const long long src = (((long long)b * K + i) * Hkv + h) * row_vecs + c;
        k_cache[dst0 + e] = k_blk[src];
        v_cache[dst0 + e] = v_blk[src];
    }
}

__global__ void commit_len_kernel(int32_t *cache_len, const int32_t *n_commit, int B, int K,
                                  long long capacity, int32_t *status)
{
    pdl_begin();
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < B; b += gridDim.x * blockDim.x) {
        const int P = cache_len[b], n = n_commit[b];
        if (n >= 0 && n <= K && P >= 0 && (long long)P + n <= capacity) cache_len[b] = P + n;
        else if (status) atomicOr(status, ORTHRUS_DEV_APPEND_OVERFLOW);
    }
}

// four consecutive elements
template <typename T> struct Quad;
template <> struct Quad<float> {
    using V = float4;
    __device__ static void unpack(const V &v, double (&x)[4]) { x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w; }
    __device__ static V pack(const double (&x)[4]) { return make_float4((float)x[0], (float)x[1], (float)x[2], (float)x[3]); }
};
template <> struct Quad<__nv_bfloat16> {
    using V = uint2;
    __device__ static void unpack(const V &v, double (&x)[4]) {
        x[0] = __uint_as_float(v.x << 16); x[1] = __uint_as_float(v.x & 0xffff0000u);
        x[2] = __uint_as_float(v.y << 16); x[3] = __uint_as_float(v.y & 0xffff0000u);
    }
    __device__ static V pack(const double (&x)[4]) {
        V v;
        reinterpret_cast<__nv_bfloat162 &>(v.x) = __floats2bfloat162_rn((float)x[0], (float)x[1]);
        reinterpret_cast<__nv_bfloat162 &>(v.y) = __floats2bfloat162_rn((float)x[2], (float)x[3]);
        return v;
    }
};

// grid (K, B): one CTA per block row.  The d/2 angles of the row are taken once, in double
// (pos * theta^(-2c/d) reaches tens of thousands of radians at long contexts, where a float
// angle would be off by more than the output's rounding), then every head is rotated with them.
// Latency is all there is to this kernel: a dependent load of the length, the sine and cosine, a
// barrier, the stores.  The frequencies are formed before the wait for the preceding kernel, and
// the row's elements (four per load) are requested before the angles are taken.
template <typename T>
__global__ void __launch_bounds__(256) rope_block_kv_write_kernel(
    const T *q, const T *k_blk, const T *v_blk, T *q_out, T *k_cache, T *v_cache, const int32_t *cache_len,
    int K, int Hq, int Hkv, int d, long long capacity, double log2_theta, int32_t *status)
{
    using V = typename Quad<T>::V;
    constexpr int U = 4;                       // items a thread requests at once
    extern __shared__ double cs[];             // [d/2] cosines, [d/2] sines
    const int i = blockIdx.x, b = blockIdx.y;
    const int half = d >> 1;
    double freq = 0.0;                         // of column threadIdx.x (half <= 128 <= blockDim.x)
    if ((int)threadIdx.x < half) freq = exp2(-2.0 * (double)threadIdx.x / (double)d * log2_theta);
    pdl_begin();
    const int P = cache_len[b];
    const long long row = (long long)b * K + i;
    // item: four column pairs of one head, the query heads first, then the KV heads
    const int per_head = half >> 2, n_q = Hq * per_head, n_items = n_q + Hkv * per_head;
    auto place = [&](int e, int &head, int &c) { head = e / per_head; c = (e - head * per_head) << 2; };
    for (int e0 = threadIdx.x; e0 < n_items || e0 == (int)threadIdx.x; e0 += U * 256) {
        V lo[U], hi[U], vl[U], vh[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int e = e0 + u * 256;
            int head, c;
            place(e, head, c);
            if (e < n_q) {
                const T *src = q + (row * Hq + head) * d + c;
                lo[u] = *reinterpret_cast<const V *>(src); hi[u] = *reinterpret_cast<const V *>(src + half);
            } else if (e < n_items) {
                const long long off = (row * Hkv + head - Hq) * d + c;
                lo[u] = *reinterpret_cast<const V *>(k_blk + off); hi[u] = *reinterpret_cast<const V *>(k_blk + off + half);
                vl[u] = *reinterpret_cast<const V *>(v_blk + off); vh[u] = *reinterpret_cast<const V *>(v_blk + off + half);
            }
        }
        const bool room = P >= 0 && (long long)P + K <= capacity;
        if (e0 == (int)threadIdx.x) {
            if (!room && status && threadIdx.x == 0 && i == 0) atomicOr(status, ORTHRUS_DEV_APPEND_OVERFLOW);
            const int pos = (P < 0 ? 0 : P) + i;       // (a sequence without room is not written; its
                                                       //  queries are still rotated, for a defined output)
            if ((int)threadIdx.x < half) {
                double s, co;
                sincos((double)pos * freq, &s, &co);
                cs[threadIdx.x] = co; cs[half + threadIdx.x] = s;
            }
            __syncthreads();
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int e = e0 + u * 256;
            if (e >= n_items) break;
            int head, c;
            place(e, head, c);
            double x0[4], x1[4], y0[4], y1[4];
            Quad<T>::unpack(lo[u], x0);
            Quad<T>::unpack(hi[u], x1);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                y0[j] = x0[j] * cs[c + j] - x1[j] * cs[half + c + j];
                y1[j] = x1[j] * cs[c + j] + x0[j] * cs[half + c + j];
            }
            if (e < n_q) {
                T *dst = q_out + (row * Hq + head) * d + c;
                *reinterpret_cast<V *>(dst) = Quad<T>::pack(y0);
                *reinterpret_cast<V *>(dst + half) = Quad<T>::pack(y1);
            } else if (room) {
                // keys (rotated) and values (copied) go to the cache row P + i of their head
                const long long dst = (((long long)b * Hkv + head - Hq) * capacity + P + i) * d + c;
                *reinterpret_cast<V *>(k_cache + dst) = Quad<T>::pack(y0);
                *reinterpret_cast<V *>(k_cache + dst + half) = Quad<T>::pack(y1);
                *reinterpret_cast<V *>(v_cache + dst) = vl[u];
                *reinterpret_cast<V *>(v_cache + dst + half) = vh[u];
            }
        }
    }
}

}  // namespace

cudaError_t launch_block_kv_write(const orthrus_layer_t &L, const void *k_blk, const void *v_blk,
                                  int32_t *status, cudaStream_t st)
{
    const int es = L.dtype == ORTHRUS_FP32 ? 4 : 2;
    const int row_vecs = L.head_dim * es / 16;
    return launch_kernel(early_launch(L), block_kv_write_kernel, dim3(L.batch, L.n_kv_heads), 128, 0, st,
                         static_cast<uint4 *>(L.k_cache), static_cast<uint4 *>(L.v_cache), L.cache_len,
                         static_cast<const uint4 *>(k_blk), static_cast<const uint4 *>(v_blk), L.block, L.n_kv_heads,
                         row_vecs, L.capacity, status);
}

cudaError_t launch_commit_len(const orthrus_layer_t &L, const int32_t *n_commit, int32_t *status,
                              cudaStream_t st)
{
    const int blocks = (L.batch + 255) / 256 < 64 ? (L.batch + 255) / 256 : 64;
    return launch_kernel(early_launch(L), commit_len_kernel, dim3(blocks), 256, 0, st, L.cache_len, n_commit, L.batch,
                         L.block, L.capacity, status);
}

cudaError_t launch_rope_block_kv_write(const orthrus_layer_t &L, const void *q, const void *k_blk,
                                       const void *v_blk, double theta, void *q_out, int32_t *status,
                                       cudaStream_t st)
{
    const dim3 grid(L.block, L.batch);
    const size_t smem = (size_t)L.head_dim * sizeof(double);
    const double log2_theta = log2(theta);
    auto run = [&](auto *zero) {
        using T = std::remove_pointer_t<decltype(zero)>;
        return launch_kernel(early_launch(L), rope_block_kv_write_kernel<T>, grid, 256, smem, st,
                             static_cast<const T *>(q), static_cast<const T *>(k_blk), static_cast<const T *>(v_blk),
                             static_cast<T *>(q_out), static_cast<T *>(L.k_cache), static_cast<T *>(L.v_cache),
                             L.cache_len, L.block, L.n_q_heads, L.n_kv_heads, L.head_dim, L.capacity, log2_theta, status);
    };
    return L.dtype == ORTHRUS_FP32 ? run(static_cast<float *>(nullptr)) : run(static_cast<__nv_bfloat16 *>(nullptr));
}

}  // namespace orthrus
