// Sampled consensus for temperature T > 0: the rejection-sampling rule of Section 3.3.
//
// With p = softmax(ar_logits / T) and q = softmax(diff_logits / T) per block position, the
// drafts are visited left to right; draft y_k is kept iff u_accept * q_k(y_k) <= p_k(y_k);
// the first position that fails gets a correction token drawn from max(0, p_k - q_k) by
// inverting its running sum with u_resample.  Two kernels (three for large problems):
//   sample_stats   a warp per (row, stretch of the vocabulary): one online pass over BOTH logit rows
//                  giving an integer reference at or above the maximum and the sum of exponentials
//                  relative to it (16-byte loads, eight in flight per lane; 1/T and log2(e) folded into
//                  one multiply).  Bound by the loads and, close behind, by the exponentials.
//   sample_finish  a cluster of CTAs per sequence: folds the stretches, takes the accept tests, sums
//                  the residual of the first rejected row (a share of the vocabulary per CTA, exchanged
//                  through distributed shared memory), and the CTA whose share holds the drawn point
//                  finds the token by block scans.
// Verification halts at the first rejected draft, so rows behind it are not needed.  When the logits
// are many times what the GPU holds in flight, the statistics pass takes the rows of all sequences in
// the order of their block position; whoever completes a row takes its accept test and lowers the
// sequence's first failure, and stretches behind a known failure are skipped.  Nobody waits: a row
// that is read in vain costs time only, and the result is the smallest failing row either way.  (With
// one statistics pass over a quarter of the block, a second one over the rest for the sequences still
// open, and serial folds, the two configurations named in the benchmark took 124 and 41 us.)
// Exponentials are fp32; every sum is carried in double and taken in a fixed order, and
// references are integers so that rescaling is exact: the result is reproducible run to run
// and departs from an exact evaluation only by the rounding of the individual exponentials.
#include "common.cuh"
#include "tc_ptx.cuh"

namespace orthrus {
namespace {

constexpr int kThreads = 256, kWarps = kThreads / 32;
constexpr int kStretch = 4096;          // logits of a row a warp takes at a time (about), where there are plenty

template <typename T> struct Elem;
template <> struct Elem<__nv_bfloat16> {
    static constexpr int N = 8;
    __device__ static void unpack(const uint4 &u, float (&x)[8]) {
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            x[2 * k] = __uint_as_float(w[k] << 16);
            x[2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u);
        }
    }
    __device__ static float load(const __nv_bfloat16 *p) { return __bfloat162float(*p); }
};
template <> struct Elem<float> {
    static constexpr int N = 4;
    __device__ static void unpack(const uint4 &u, float (&x)[4]) {
        x[0] = __uint_as_float(u.x); x[1] = __uint_as_float(u.y);
        x[2] = __uint_as_float(u.z); x[3] = __uint_as_float(u.w);
    }
    __device__ static float load(const float *p) { return *p; }
};

// Running (reference, sum of 2^(x - reference)).  The reference is an INTEGER at or above the
// largest value seen (in the log2 domain), so that moving it rescales the sum by an exact
// power of two: partial results of different threads and segments then combine without any
// rounding beyond that of the additions, which are carried in double.
struct RefSum { float m; double s; };
__device__ inline float pow2i(float k) {                 // 2^k for integer-valued k <= 0 (0 below the normal range)
    const int e = (int)k + 127;
    return e > 0 ? __int_as_float(e << 23) : 0.f;
}
// R x N raw logits; c > 0 scales them into the log2 domain.  The instruction count matters (the loop
// is bound by the exponentials only while the rest stays below them): the maximum is taken over the
// raw values, once for all R vectors (some lane of a warp raises its reference at nearly every check),
// scaling and reference are one fused multiply-add, and the sum of a vector enters in double.
template <int R, int N>
__device__ inline void absorb(RefSum &a, const float (&x)[R][N], float c) {
    float mx[R];
#pragma unroll
    for (int q = 0; q < R; ++q) {
        mx[q] = fmaxf(x[q][0], x[q][1]);
#pragma unroll
        for (int e = 2; e < N; e += 2) mx[q] = max3(mx[q], x[q][e], x[q][e + 1]);
    }
#pragma unroll
    for (int q = 1; q < R; ++q) mx[0] = fmaxf(mx[0], mx[q]);
    mx[0] *= c;
    if (mx[0] > a.m) {
        const float m_new = ceilf(mx[0]);
        if (a.m > -INFINITY) a.s *= (double)pow2i(a.m - m_new);
        a.m = m_new;
    }
    if (a.m == -INFINITY) return;
    const float2 c2 = make_float2(c, c), m2 = make_float2(-a.m, -a.m);
    float sum[R];
#pragma unroll
    for (int q = 0; q < R; ++q) {
        float2 s0 = make_float2(0.f, 0.f);
#pragma unroll
        for (int e = 0; e < N; e += 2) {
            const float2 y = __ffma2_rn(make_float2(x[q][e], x[q][e + 1]), c2, m2);
            s0 = __fadd2_rn(s0, make_float2(ex2(y.x), ex2(y.y)));
        }
        sum[q] = s0.x + s0.y;
    }
#pragma unroll
    for (int q = 0; q < R; ++q) a.s += (double)sum[q];
}
__device__ inline double warp_sum(double x) {
#pragma unroll
    for (int off = 16; off; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    return x;
}
__device__ inline float warp_max(float x) {
    float y;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(y) : "f"(x));
    return y;
}
// fold over a warp in a fixed order, known to every lane: the reference first, then each lane's sum is
// scaled to it once (scaling at each of the five steps is a chain of three dependent double operations)
__device__ inline RefSum warp_fold(const RefSum &v) {
    const float M = warp_max(v.m);
    return RefSum{M, warp_sum(v.m > -INFINITY ? v.s * (double)pow2i(v.m - M) : 0.0)};
}

struct alignas(8) StatPart { float ma, md; double sa, sd; };       // per (row, stretch)

// The logits of one row as vectors of N elements on 16-byte boundaries: vector v holds elements
// [v * N - a, v * N - a + N), of which those outside [0, V) do not exist.  Only the first and the last
// can be incomplete.  `vec` false (the two tensors' rows are not aligned alike): no 16-byte loads.
struct RowShape { int V, a, n_vec; bool vec; };
template <typename T> __device__ inline RowShape row_shape(const T *ra, const T *rd, int V) {
    const uintptr_t x = reinterpret_cast<uintptr_t>(ra) & 15, y = reinterpret_cast<uintptr_t>(rd) & 15;
    RowShape s;
    s.V = V;
    s.vec = x == y;
    s.a = s.vec ? (int)(x / sizeof(T)) : 0;
    s.n_vec = (V + s.a + Elem<T>::N - 1) / Elem<T>::N;
    return s;
}
template <typename T> __device__ inline bool whole(const RowShape &s, int v) {
    return s.vec && v * Elem<T>::N >= s.a && v * Elem<T>::N - s.a + Elem<T>::N <= s.V;
}
// one vector of a row; elements that do not exist are -inf (their exponential is 0)
template <typename T> struct VecOf { float x[Elem<T>::N]; };
template <typename T> __device__ __noinline__ VecOf<T> load_part(const T *row, int i0, int V) {
    VecOf<T> r;
#pragma unroll
    for (int e = 0; e < Elem<T>::N; ++e) r.x[e] = i0 + e >= 0 && i0 + e < V ? Elem<T>::load(row + i0 + e) : -INFINITY;
    return r;
}
template <typename T> __device__ inline void load_vec(const T *row, const RowShape &s, int v, float (&x)[Elem<T>::N]) {
    const int i0 = v * Elem<T>::N - s.a;
    if (whole<T>(s, v)) {
        Elem<T>::unpack(__ldg(reinterpret_cast<const uint4 *>(row + i0)), x);
    } else {
        const VecOf<T> r = load_part<T>(row, i0, s.V);
#pragma unroll
        for (int e = 0; e < Elem<T>::N; ++e) x[e] = r.x[e];
    }
}

// the accept test of one row, from its folded statistics
template <typename T>
__device__ inline bool keeps(const T *ra, const T *rd, const RefSum &a, const RefSum &d, int draft, float u, int V, float c)
{
    const int y = min(max(draft, 0), V - 1);            // an out-of-range draft id is clamped, not dereferenced
    // u * q(y) <= p(y), both sides times the two sums
    return (double)u * (double)ex2(Elem<T>::load(rd + y) * c - d.m) * a.s <= (double)ex2(Elem<T>::load(ra + y) * c - a.m) * d.s;
}
// a warp folds the stretches of a row (four per lane requested together)
__device__ inline void fold_row(const StatPart *parts, int n_seg, int lane, RefSum &a, RefSum &d) {
    a = d = RefSum{-INFINITY, 0.0};
    for (int s0 = lane; s0 < n_seg; s0 += 128) {
        StatPart t[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            t[q] = StatPart{-INFINITY, -INFINITY, 0.0, 0.0};
            if (s0 + q * 32 < n_seg) {                  // (written by other SMs: past L1)
                const StatPart *x = parts + s0 + q * 32;
                const float2 m = __ldcg(reinterpret_cast<const float2 *>(x));
                t[q].ma = m.x; t[q].md = m.y;
                t[q].sa = __ldcg(&x->sa); t[q].sd = __ldcg(&x->sd);
            }
        }
        auto add = [](RefSum &v, float m0, double s0, float m1, double s1, float m2, double s2, float m3, double s3) {
            const float M = fmaxf(fmaxf(fmaxf(m0, m1), fmaxf(m2, m3)), v.m);
            if (M == -INFINITY) return;
            auto at = [M](float m, double x) { return m > -INFINITY ? x * (double)pow2i(m - M) : 0.0; };
            v = RefSum{M, at(v.m, v.s) + ((at(m0, s0) + at(m1, s1)) + (at(m2, s2) + at(m3, s3)))};
        };
        add(a, t[0].ma, t[0].sa, t[1].ma, t[1].sa, t[2].ma, t[2].sa, t[3].ma, t[3].sa);
        add(d, t[0].md, t[0].sd, t[1].md, t[1].sd, t[2].md, t[2].sd, t[3].md, t[3].sd);
    }
    a = warp_fold(a);
    d = warp_fold(d);
}

// the same out of line, for the finish kernel, where it stands twice and its code counts
struct RowFold { RefSum a, d; };
__device__ __noinline__ RowFold fold_row_call(const StatPart *parts, int n_seg, int lane) {
    RowFold f;
    fold_row(parts, n_seg, lane, f.a, f.d);
    return f;
}

// per sequence: first row known to fail; per row: stretches done.  Only the skipping form reads them.
__global__ void sample_init_kernel(int *fail, int *done, int B, int K)
{
    pdl_begin();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < B * K; i += gridDim.x * blockDim.x) {
        done[i] = 0;
        if (i < B) fail[i] = K;
    }
}

// A warp takes items (block position k, sequence b, stretch) in that order, k outermost.
template <typename T, bool SKIP>
__global__ void __launch_bounds__(kThreads) sample_stats_kernel(const T *la, const T *ld, int B, int K, int V, int n_seg,
                                                                float c, const int32_t *draft, const float *u_accept,
                                                                StatPart *parts, int *fail, int *done)
{
    constexpr int N = Elem<T>::N;
    pdl_begin();
    const int lane = threadIdx.x & 31;
    const long long n_items = (long long)K * B * n_seg, stride = (long long)gridDim.x * kWarps;
    for (long long it = (long long)blockIdx.x * kWarps + (threadIdx.x >> 5); it < n_items; it += stride) {
        const int seg = (int)(it % n_seg), kb = (int)(it / n_seg), b = kb % B, k = kb / B;
        const long long row = (long long)b * K + k;
        bool needed = true;
        if (SKIP) needed = *reinterpret_cast<volatile int *>(fail + b) >= k;
        if (SKIP) needed = __all_sync(0xffffffffu, needed);
        if (needed) {
            const T *ra = la + row * V, *rd = ld + row * V;
            const RowShape sh = row_shape(ra, rd, V);
            const int per = (sh.n_vec + n_seg - 1) / n_seg, v0 = seg * per, v1 = min(sh.n_vec, v0 + per);
            RefSum a{-INFINITY, 0.0}, d{-INFINITY, 0.0};
            // whole vectors, four of each row at a time; the ends of the row by a lane an element
            const int w0 = max(v0, sh.vec ? (sh.a + N - 1) / N : v1), w1 = min(v1, (V + sh.a) / N);
            const uint4 *va = reinterpret_cast<const uint4 *>(ra - sh.a), *vd = reinterpret_cast<const uint4 *>(rd - sh.a);
            int v = w0 + lane;
            for (; v + 96 < w1; v += 128) {
                uint4 x[4], y[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) { x[q] = __ldg(va + v + q * 32); y[q] = __ldg(vd + v + q * 32); }
                float f[4][N];
#pragma unroll
                for (int q = 0; q < 4; ++q) Elem<T>::unpack(x[q], f[q]);
                absorb<4, N>(a, f, c);
#pragma unroll
                for (int q = 0; q < 4; ++q) Elem<T>::unpack(y[q], f[q]);
                absorb<4, N>(d, f, c);
            }
            for (; v < w1; v += 32) {
                const uint4 x = __ldg(va + v), y = __ldg(vd + v);
                float f[1][N];
                Elem<T>::unpack(x, f[0]); absorb<1, N>(a, f, c);
                Elem<T>::unpack(y, f[0]); absorb<1, N>(d, f, c);
            }
            if (sh.vec) {
                // the elements in front of the first whole vector, then those behind the last one
                const int lo = max(v0 * N - sh.a, 0), hi = min(v1 * N - sh.a, V);
                const int h = min(w0 * N - sh.a, hi), t = max(w1 * N - sh.a, h);
                if (lo < h || t < hi) {
                    const int e = lane < 8 ? lo + lane : t + lane - 8;
                    const bool mine = lane < 8 ? e < h : lane < 16 && e < hi;
                    float f[1][2];
                    f[0][1] = -INFINITY;
                    f[0][0] = mine ? Elem<T>::load(ra + e) : -INFINITY; absorb<1, 2>(a, f, c);
                    f[0][0] = mine ? Elem<T>::load(rd + e) : -INFINITY; absorb<1, 2>(d, f, c);
                }
            }
            else for (int e = v0 + lane; e < v1; e += 32) {
                float f[1][N];
                load_vec<T>(ra, sh, e, f[0]); absorb<1, N>(a, f, c);
                load_vec<T>(rd, sh, e, f[0]); absorb<1, N>(d, f, c);
            }
            a = warp_fold(a);
            d = warp_fold(d);
            if (lane == 0) parts[row * n_seg + seg] = StatPart{a.m, d.m, a.s, d.s};
        }
        // (a stretch that was skipped is not counted: its row is behind a failure, and nobody asks for it)
        if (SKIP && needed) {
            int before = 0;
            if (lane == 0) {
                __threadfence();                        // the statistics before the count
                before = atomicAdd(done + row, 1);
            }
            before = __shfl_sync(0xffffffffu, before, 0);
            // the row is complete
            if (before == n_seg - 1 && *reinterpret_cast<volatile int *>(fail + b) >= k) {
                __threadfence();
                RefSum a, d;
                fold_row(parts + row * n_seg, n_seg, lane, a, d);
                if (lane == 0 && !keeps(la + row * V, ld + row * V, a, d, draft[row], u_accept[row], V, c)) atomicMin(fail + b, k);
            }
        }
    }
}

struct RowStat { float ma, md; double inv_za, inv_zd; };  // of the first rejected row (1 / sums)

// an element's share of the residual max(0, p - q), or (use_p) of p; 0 for one that does not exist
__device__ inline double mass_of(float xa, float xd, float c, const RowStat &st, bool use_p) {
    const double p = (double)ex2(xa * c - st.ma) * st.inv_za;
    const double r = use_p ? p : fma(-(double)ex2(xd * c - st.md), st.inv_zd, p);
    return r > 0.0 ? r : 0.0;
}
__device__ inline double peer_double(const double *mine, int rank) {
    double x;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(x) : "r"(map_to_rank(smem_u32(mine), rank)) : "memory");
    return x;
}

// Grid (C, B) in clusters of C: one sequence.  The residual's running sum is taken over CTAs, then a
// CTA's warps, then a warp's groups of rounds (a round is 32 vectors, a lane each), in index order, and
// each level keeps its sums, so that the drawn point is found level by level.  Bound by latencies (dependent
// double operations, loads from L2), hence 16 warps a CTA, the mass of p only where the residual turns out to be
// empty, and sums in several chains.  With 8 warps and both masses in one chain each the residual of a row of
// 128256 took 13 us in clusters of 8; whole passes 102 -> 93 us (batch 32) and 23.8 -> 18.8 us (batch 1).
// An SM's instruction cache holds 32 KB, and every warp runs through this code once: one round per turn of the loop, the next
// one's vectors asked for ahead, incomplete vectors and the fold of a row out of line (66 -> 49 KB), in the statistics
// the ends of a row by a lane an element: 93.6 -> 85.9 us (batch 32), 19.2 -> 18.0 us (batch 1).  The fold out of line in the
// statistics as well, where it writes to the stack: 118 us.
constexpr int kFinishThreads = 512, kFinishWarps = kFinishThreads / 32, kGroups = 64;
template <typename T>
__global__ void __launch_bounds__(kFinishThreads, 2) sample_finish_kernel(const T *la, const T *ld, int K, int V, int n_seg, float c,
                                                                 const int32_t *draft, const float *u_accept,
                                                                 const float *u_resample, const StatPart *parts,
                                                                 const int *fail, int32_t *n_commit, int32_t *committed,
                                                                 int32_t *next_anchor)
{
    constexpr int N = Elem<T>::N;
    __shared__ double grp[kFinishWarps][kGroups], wsum[kFinishWarps], csum[2];
    __shared__ double s_before, s_target;
    __shared__ int s_first, s_owner, s_use_p, s_empty;
    __shared__ RowStat s_stat;
    extern __shared__ RefSum folded[];                  // [K][2], unless the failures are known already
    const int b = blockIdx.y, rank = blockIdx.x, C = gridDim.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    pdl_begin();
    if (tid == 0) s_first = fail ? fail[b] : K;
    __syncthreads();
    if (!fail) {
        for (int i = warp; i < K; i += kFinishWarps) {
            const long long row = (long long)b * K + i;
            const RowFold f = fold_row_call(parts + row * n_seg, n_seg, lane);
            if (lane == 0) {
                folded[2 * i] = f.a; folded[2 * i + 1] = f.d;
                if (!keeps(la + row * V, ld + row * V, f.a, f.d, draft[row], u_accept[row], V, c)) atomicMin(&s_first, i);
            }
        }
        __syncthreads();
    }
    const int j = s_first;                              // K: every draft is kept
    if (rank == 0) {
        for (int i = tid; i < K; i += kFinishThreads)
            if (i != j) committed[(long long)b * K + i] = i < j ? draft[(long long)b * K + i] : -1;
        if (tid == 0) {
            n_commit[b] = j < K ? j + 1 : K;
            if (j >= K) next_anchor[b] = draft[(long long)b * K + K - 1];
        }
    }
    if (j >= K) return;                                 // (the whole cluster)
    const long long row = (long long)b * K + j;
    const T *ra = la + row * V, *rd = ld + row * V;
    if (warp == 0) {
        RowFold f;
        if (fail) f = fold_row_call(parts + row * n_seg, n_seg, lane);
        else f = RowFold{folded[2 * j], folded[2 * j + 1]};
        if (lane == 0) s_stat = RowStat{f.a.m, f.d.m, 1.0 / f.a.s, 1.0 / f.d.s};
    }
    __syncthreads();
    const RowStat st = s_stat;
    const RowShape sh = row_shape(ra, rd, V);
    const int per = (sh.n_vec + C - 1) / C, v0 = rank * per, v1 = min(sh.n_vec, v0 + per);
    const int per_w = (per + kFinishWarps - 1) / kFinishWarps, w0 = min(v1, v0 + warp * per_w), w1 = min(v1, w0 + per_w);
    // (a group costs two warp sums, a round in the end two loads: two rounds and up to a group)
    const int rounds = (per_w + 31) / 32, gsz = max(2, (rounds + kGroups - 1) / kGroups), n_grp = (rounds + gsz - 1) / gsz;
    // the residual; if it is empty (p and q agree to the last bit), the mass of p
#pragma unroll 1
    for (int use_p = 0; use_p < 2; ++use_p) {
        double total = 0.0, sum = 0.0;
        // (whole vectors are asked for one round ahead, as they come)
        uint4 nx = make_uint4(0, 0, 0, 0), ny = nx;
        auto ask = [&](int r) {
            const int v = w0 + r * 32 + lane;
            if (r < rounds && v < w1 && whole<T>(sh, v)) {
                nx = __ldg(reinterpret_cast<const uint4 *>(ra + v * N - sh.a));
                ny = __ldg(reinterpret_cast<const uint4 *>(rd + v * N - sh.a));
            }
        };
        ask(0);
        int left = gsz, g = 0;                          // rounds left in this group
#pragma unroll 1
        for (int r = 0; r < rounds; ++r) {
            const uint4 cx = nx, cy = ny;
            ask(r + 1);
            const int v = w0 + r * 32 + lane;
            if (v < w1) {
                float x[N], y[N];
                if (whole<T>(sh, v)) { Elem<T>::unpack(cx, x); Elem<T>::unpack(cy, y); }
                else { load_vec<T>(ra, sh, v, x); load_vec<T>(rd, sh, v, y); }
                double m[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
                for (int e = 0; e < N; ++e) m[e & 3] += mass_of(x[e], y[e], c, st, use_p);
                sum += (m[0] + m[1]) + (m[2] + m[3]);
            }
            if (--left == 0 || r == rounds - 1) {
                sum = warp_sum(sum);
                if (lane == 0) grp[warp][g] = sum;
                total += sum;
                sum = 0.0;
                left = gsz;
                ++g;
            }
        }
        if (lane == 0) wsum[warp] = total;
        __syncthreads();
        if (warp == 0) {
            const double s = warp_sum(lane < kFinishWarps ? wsum[lane] : 0.0);
            if (lane == 0) csum[use_p] = s;
        }
        cluster_sync_all();
        // every CTA finds the share that holds the drawn point: the first whose running sum exceeds the target,
        // the last that is not empty if rounding leaves the target at or past the total
        if (warp == 0) {
            const double x = lane < C ? peer_double(&csum[use_p], lane) : 0.0;
            double incl = x;                            // running sum over the CTAs
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const double o = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += o;
            }
            const double tot = __shfl_sync(0xffffffffu, incl, 31), target = (double)u_resample[row] * tot;
            const unsigned hit = __ballot_sync(0xffffffffu, x > 0.0 && incl > target), some = __ballot_sync(0xffffffffu, x > 0.0);
            const int pick = hit ? __ffs(hit) - 1 : some ? 31 - __clz(some) : 0;
            const double upto = __shfl_sync(0xffffffffu, incl - x, pick);
            if (lane == 0) { s_owner = pick; s_use_p = use_p; s_before = hit ? upto : tot; s_target = target; s_empty = !(tot > 0.0); }
        }
        __syncthreads();
        if (!s_empty) break;
    }
    if (rank == s_owner && warp == 0) {
        // the warp and the group of rounds, by the same rule (a lane's warp total, then a lane's two groups)
        const int use_p = s_use_p;
        const double target = s_target;
        double run = s_before, at = run;
        int last = 0;
        auto pick = [&](const double *sums, int n, bool none) {   // -1: past the end
            int z = -1;
#pragma unroll 4
            for (int i = 0; i < n; ++i) {
                const double v = sums[i];
                if (v > 0.0) {
                    last = i;
                    if (z < 0 && !none && run + v > target) { z = i; at = run; }
                    run += v;
                }
            }
            if (z < 0) at = run;
            return z;
        };
        int pw = pick(wsum, kFinishWarps, false);
        const bool past = pw < 0;                       // rounding: take the last element that is positive
        if (past) pw = last;
        run = at;
        last = 0;
        int pg = pick(grp[pw], n_grp, past);
        if (pg < 0) pg = last;
        // the vector and the element
        const int q0 = min(v1, v0 + pw * per_w), q1 = min(v1, q0 + per_w);
        int z = -1, z_last = -1;
        run = at;
#pragma unroll 1
        for (int r = pg * gsz; r < min(rounds, (pg + 1) * gsz) && z < 0; ++r) {
            const int v = q0 + r * 32 + lane;
            float x[N], y[N];
            double mine[N], sum = 0.0;
            if (v < q1) { load_vec<T>(ra, sh, v, x); load_vec<T>(rd, sh, v, y); }
#pragma unroll
            for (int e = 0; e < N; ++e) {
                mine[e] = v < q1 ? mass_of(x[e], y[e], c, st, use_p) : 0.0;
                sum += mine[e];
            }
            double incl = sum;                          // running sum over the lanes
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const double o = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += o;
            }
            const unsigned hit = __ballot_sync(0xffffffffu, !past && sum > 0.0 && run + incl > target);
            int my_last = -1, my_z = -1;
            double acc = run + (incl - sum);
#pragma unroll
            for (int e = 0; e < N; ++e)
                if (mine[e] > 0.0) {
                    my_last = v * N - sh.a + e;
                    acc += mine[e];
                    if (my_z < 0 && acc > target) my_z = my_last;
                }
            if (hit) {
                const int l = __ffs(hit) - 1;
                z = __shfl_sync(0xffffffffu, my_z >= 0 ? my_z : my_last, l);
            }
            const unsigned some = __ballot_sync(0xffffffffu, my_last >= 0);
            if (some) z_last = __shfl_sync(0xffffffffu, my_last, 31 - __clz(some));
            run += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (z < 0) z = z_last >= 0 ? z_last : 0;
        if (lane == 0) {
            committed[(long long)b * K + j] = z;
            next_anchor[b] = z;
        }
    }
    cluster_sync_all();                                 // the peers have read this CTA's sums
}

}  // namespace

// Stretches per row: about kStretch logits each, shorter ones (down to 512) where the rows are too few
// to give every SM 16 warps.
static int sample_stat_segments(int B, int K, int V)
{
    const long long want = (16LL * num_sms() + (long long)B * K - 1) / ((long long)B * K);
    const int lo = (V + kStretch - 1) / kStretch, hi = (V + 511) / 512;
    return want < lo ? lo : want > hi ? hi : (int)want;
}

size_t sample_workspace_bytes(int B, int K, int V)
{
    return (size_t)B * K * sample_stat_segments(B, K, V) * sizeof(StatPart) + (size_t)B * K * sizeof(int) + (size_t)B * sizeof(int);
}

template <typename T>
static cudaError_t launch_sample_t(const void *ar_logits, const void *diff_logits, const int32_t *draft,
                                   const float *u_accept, const float *u_resample, float temperature, int B, int K,
                                   int V, int32_t *n_commit, int32_t *committed, int32_t *next_anchor,
                                   unsigned char *ws, cudaStream_t st)
{
    const T *la = static_cast<const T *>(ar_logits), *ld = static_cast<const T *>(diff_logits);
    const float c = 1.4426950408889634f / temperature;
    const int n_seg = sample_stat_segments(B, K, V);
    StatPart *parts = reinterpret_cast<StatPart *>(ws);
    int *done = reinterpret_cast<int *>(ws + (size_t)B * K * n_seg * sizeof(StatPart)), *fail = done + (size_t)B * K;
    // The skipping form pays for its counters and its extra launch once the logits are several waves
    // of the grid below: then whole rows behind the first rejection are left out.
    const long long n_items = (long long)B * K * n_seg;
    // (every resident warp more is a stretch more that may be read in vain)
    const bool skip = K > 1 && n_items > 64LL * num_sms();
    const int ctas_per_sm = skip ? 3 : 4;
    const int grid = (int)((n_items + kWarps - 1) / kWarps < (long long)ctas_per_sm * num_sms()
                               ? (n_items + kWarps - 1) / kWarps : (long long)ctas_per_sm * num_sms());
    cudaError_t e;
    if (skip) {
        const int n = (B * K + 255) / 256;
        e = launch_kernel(true, sample_init_kernel, dim3(n < 64 ? n : 64), 256, 0, st, fail, done, B, K);
        if (e == cudaSuccess)
            e = launch_kernel(true, sample_stats_kernel<T, true>, dim3(grid), kThreads, 0, st, la, ld, B, K, V, n_seg, c, draft,
                              u_accept, parts, fail, done);
    } else {
        e = launch_kernel(true, sample_stats_kernel<T, false>, dim3(grid), kThreads, 0, st, la, ld, B, K, V, n_seg, c, draft,
                          u_accept, parts, fail, done);
    }
    if (e != cudaSuccess) return e;
    // CTAs per sequence: 16 for the first few, 8 (the portable cluster size) while that does not crowd the GPU
    int C = B <= 4 ? 16 : 8;
    while (C > 1 && (long long)B * C > 4LL * num_sms()) C /= 2;
    if (C > 8) {
        e = cudaFuncSetAttribute(sample_finish_kernel<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C, B);
    cfg.blockDim = dim3(kFinishThreads);
    cfg.dynamicSmemBytes = skip ? 0 : (size_t)K * 2 * sizeof(RefSum);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = early_launch_allowed() ? 2 : 1;
    count_launch();
    return cudaLaunchKernelEx(&cfg, sample_finish_kernel<T>, la, ld, K, V, n_seg, c, draft, u_accept, u_resample,
                              static_cast<const StatPart *>(parts), static_cast<const int *>(skip ? fail : nullptr), n_commit,
                              committed, next_anchor);
}

cudaError_t launch_consensus_sample(const void *ar_logits, const void *diff_logits, int dtype, const int32_t *draft,
                                    const float *u_accept, const float *u_resample, float temperature, int B, int K,
                                    int V, int32_t *n_commit, int32_t *committed, int32_t *next_anchor, void *ws,
                                    cudaStream_t st)
{
    unsigned char *w = static_cast<unsigned char *>(ws);
    if (dtype == ORTHRUS_FP32)
        return launch_sample_t<float>(ar_logits, diff_logits, draft, u_accept, u_resample, temperature, B, K, V,
                                      n_commit, committed, next_anchor, w, st);
    return launch_sample_t<__nv_bfloat16>(ar_logits, diff_logits, draft, u_accept, u_resample, temperature, B, K, V,
                                          n_commit, committed, next_anchor, w, st);
}

}  // namespace orthrus
