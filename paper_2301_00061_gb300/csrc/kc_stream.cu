// kc_stream.cu -- the float bound of few nodes (kc_lb.cu's streaming path).
#include <cuda_runtime.h>

#include "kc_device.cuh"
#include "kc_internal.cuh"
#include "kc_prune.cuh"

namespace kc {

namespace {

// ---- few nodes: one streaming pass, every term evaluated
// At one or two nodes a sample's bytes cost as much as its arithmetic, and the
// sort of the batch kernel would cost more than it saves.  Four consecutive
// samples of a row are one 16-byte load, used as it comes as two packed pairs
// (no register moves, which cost 40 us of 124 at N = 1e7, D = 8, K = 5 when
// pairs were of attributes); even and odd attributes accumulate in two chains
// that meet in one sum, so each lane's value is box_dist_f32's.  The upper
// difference is taken of the swapped pair, so that the 3-input maximum reads
// one even and one odd register (220 against 235 us at four nodes).
__device__ __forceinline__ float min3f(float a, float b, float c)
{
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Row values of samples s0 .. s0 + 3 as two pairs (past n - 1: sample n - 1).
__device__ __forceinline__ void load_quad(const float *__restrict__ row, int64_t n, bool vec, int64_t s0, uint64_t (&x)[2])
{
    if (vec && s0 + 4 <= n) {
        const ulonglong2 q = __ldg(reinterpret_cast<const ulonglong2 *>(row + s0));
        x[0] = q.x;
        x[1] = q.y;
    } else {
        float v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = __ldg(row + (s0 + j < n ? s0 + j : n - 1));
        x[0] = pk(v[0], v[1]);
        x[1] = pk(v[2], v[3]);
    }
}

__device__ __forceinline__ uint64_t swap2(uint64_t x)
{
    const float2 t = upk(x);
    return pk(t.y, t.x);
}

// max(lo - x, x - hi, 0) of a pair (xs: the pair swapped)
__device__ __forceinline__ uint64_t clamp2(uint64_t x, uint64_t xs, const ulonglong2 q)
{
    const float2 t0 = upk(sub2(q.x, x)), t1 = upk(sub2(xs, q.y));
    return pk(max3f(t0.x, t1.y, 0.f), max3f(t0.y, t1.x, 0.f));
}

// q = ((lo, lo), (hi, hi)) of one attribute: one more square into acc.
__device__ __forceinline__ void clamp_acc(const uint64_t (&x)[2], const uint64_t (&xs)[2], const ulonglong2 q,
                                          uint64_t (&acc)[2])
{
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint64_t m = clamp2(x[h], xs[h], q);
        acc[h] = fma2(m, m, acc[h]);
    }
}

// A thread's best value and its position; the samples come in increasing
// order, so an equal later value does not replace an earlier one.
struct StreamBest {
    float v = -1.f;
    uint32_t pos = 0u;
    template <int Q>
    __device__ void take(const float (&d)[4 * Q], int64_t s0, int64_t n)
    {
        float m = fmaxf(d[0], d[1]);
#pragma unroll
        for (int j = 2; j < 4 * Q; j += 2) m = max3f(m, d[j], d[j + 1]);
        if (m > v) {
            v = m;
            int jm = 4 * Q - 1;
#pragma unroll
            for (int j = 4 * Q - 2; j >= 0; --j)
                if (d[j] == m) jm = j;
            pos = (uint32_t)(s0 + jm < n ? s0 + jm : n - 1);
        }
    }
    __device__ unsigned long long key() const { return v >= 0.f ? key_max(v, pos) : 0ull; }
};

__device__ __forceinline__ void stream_boxes(const PruneArgs &A, ulonglong2 *box)
{
    const float *lo = static_cast<const float *>(A.lo), *hi = static_cast<const float *>(A.hi);
    for (int i = threadIdx.x; i < A.B * A.K * A.D; i += kThreads)
        box[i] = make_ulonglong2(pk(lo[i], lo[i]), pk(hi[i], hi[i]));
}

// The arguments of node range blockIdx.y.
__device__ __forceinline__ PruneArgs node_range(PruneArgs A)
{
    const int b0 = blockIdx.y * A.per;
    const size_t o = (size_t)b0 * A.K * A.D;
    A.lo = static_cast<const float *>(A.lo) + o;
    A.hi = static_cast<const float *>(A.hi) + o;
    A.B = min(A.per, A.B - b0);
    A.keys += b0;
    if (A.tmax) A.tmax += b0 * A.rows;
    return A;
}

__device__ __forceinline__ void stream_finish(const PruneArgs &A, int b, unsigned long long k, unsigned long long *red)
{
    k = warp_max_u64(k);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = k;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kThreads / 32; ++w) k = red[w] > k ? red[w] : k;
        if (k > peek(&A.keys[b])) atomicMax(&A.keys[b], k);
    }
}

// D = DC <= 8 attributes: 4 Q samples in registers, two clusters at a time (KC:
// K fixed, the loop over the clusters unrolled; 0: any K, about 8 % slower).  K = 3, 4
// and 5 are the cluster counts of the package's workloads; another one would be 24
// kernels more to compile, and a gather's latency hides the loop (no fixed K there).
// MANY (more than two nodes): each warp keeps its nodes' keys in shared memory
// and reduces over its lanes only when one of them may beat the key.
// A CTA takes a range of the nodes (blockIdx.y) where there may be more than two.
template <int DC, int KC, int Q, int CTAS, bool MANY, bool TM, bool GATHER = false>
__global__ void __launch_bounds__(kThreads, CTAS)
stream_max_small(const PruneArgs all)
{
    const PruneArgs A = MANY || TM ? node_range(all) : all;
    if (MANY && !GATHER && A.left && A.left[A.gx] == 0) return;
    constexpr int ST = 4 * Q, NWP = kThreads / 32;
    extern __shared__ __align__(16) unsigned char smem[];
    ulonglong2 *box = reinterpret_cast<ulonglong2 *>(smem);   // [B * K][DC]
    unsigned long long *wkey = reinterpret_cast<unsigned long long *>(box + A.B * A.K * DC);   // MANY: [warps][B]
    unsigned long long *mine = wkey + (threadIdx.x >> 5) * A.B;
    __shared__ unsigned long long red[NWP];
    stream_boxes(A, box);
    if (MANY || TM)
        for (int i = threadIdx.x; i < NWP * A.B; i += kThreads) wkey[i] = 0ull;
    __syncthreads();
    const float *X = static_cast<const float *>(A.X);
    const int K = KC ? KC : A.K;
    StreamBest best0, best1;
    for (int64_t base = (int64_t)blockIdx.x * (kThreads * ST); base < A.n; base += (int64_t)gridDim.x * (kThreads * ST)) {
        if (MANY && !GATHER && A.left) {
            // only what the pruning kernel left: its tiles of A.T, dealt to A.gx CTAs
            bool some = false;
            for (int64_t t = base / A.T; t <= (base + kThreads * ST - 1) / A.T; ++t) some |= A.left[t % A.gx] != 0;
            if (!some) continue;
        }
        // quad q of a thread: samples base + (q kThreads + tid) 4 ..
        const int64_t s0 = base + (int64_t)threadIdx.x * 4;
        uint64_t x[Q][DC][2];
        uint32_t id[GATHER ? ST : 1];
        if constexpr (GATHER) {
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int64_t t0 = s0 + q * kThreads * 4;
                if (A.vec && t0 + 4 <= A.n) {
                    const uint4 v = __ldg(reinterpret_cast<const uint4 *>(A.ids + t0));
                    id[4 * q] = v.x; id[4 * q + 1] = v.y; id[4 * q + 2] = v.z; id[4 * q + 3] = v.w;
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) id[4 * q + j] = __ldg(A.ids + (t0 + j < A.n ? t0 + j : A.n - 1));
                }
            }
#pragma unroll
            for (int q = 0; q < Q; ++q)
#pragma unroll
                for (int a = 0; a < DC; ++a)
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        x[q][a][h] = pk(__ldg(X + (size_t)a * A.ld + id[4 * q + 2 * h]),
                                        __ldg(X + (size_t)a * A.ld + id[4 * q + 2 * h + 1]));
        } else {
#pragma unroll
            for (int q = 0; q < Q; ++q)
#pragma unroll
                for (int a = 0; a < DC; ++a)
                    load_quad(X + (size_t)a * A.ld, A.n, A.vec != 0, s0 + q * kThreads * 4, x[q][a]);
        }
        uint64_t xs[Q][DC][2];
#pragma unroll
        for (int q = 0; q < Q; ++q)
#pragma unroll
            for (int a = 0; a < DC; ++a)
#pragma unroll
                for (int h = 0; h < 2; ++h) xs[q][a][h] = swap2(x[q][a][h]);
        auto dists = [&](const ulonglong2 *bx, float (&d)[ST]) {
            uint64_t e[Q][2], o[Q][2];
#pragma unroll
            for (int a = 0; a < DC; ++a) {
                const ulonglong2 c = bx[a];
#pragma unroll
                for (int q = 0; q < Q; ++q)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const uint64_t m = clamp2(x[q][a][h], xs[q][a][h], c);
                        uint64_t &acc = (a & 1) ? o[q][h] : e[q][h];
                        acc = fma2(m, m, a < 2 ? 0ull : acc);
                    }
            }
#pragma unroll
            for (int q = 0; q < Q; ++q)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float2 r = upk(DC > 1 ? add2(e[q][h], o[q][h]) : e[q][h]);
                    d[4 * q + 2 * h] = r.x;
                    d[4 * q + 2 * h + 1] = r.y;
                }
        };
        for (int b = 0; b < A.B; ++b) {
            const ulonglong2 *bb = box + b * K * DC;
            float m[ST];
            if (K & 1) {
                dists(bb, m);
            } else {
#pragma unroll
                for (int j = 0; j < ST; ++j) m[j] = __int_as_float(0x7f800000);
            }
#pragma unroll(KC ? KC : 1)
            for (int k = K & 1; k < K; k += 2) {
                float d0[ST], d1[ST];
                dists(bb + k * DC, d0);
                dists(bb + (k + 1) * DC, d1);
#pragma unroll
                for (int j = 0; j < ST; ++j) m[j] = min3f(m[j], d0[j], d1[j]);
            }
            if constexpr (TM) {
                const unsigned w = __reduce_max_sync(0xffffffffu, __float_as_uint(max_of<ST>(m)));
                if ((threadIdx.x & 31) == 0) {
                    const int64_t row = (base >> 7) + (threadIdx.x >> 5);
                    if (row * kStreamTile < A.n) A.tmax[b * A.rows + row] = __uint_as_float(w);
                    const unsigned long long key = ((unsigned long long)w << 32) | 1ull;
                    if (key > mine[b]) mine[b] = key;
                }
            } else if constexpr (MANY) {
                const unsigned long long cur = mine[b];
                const bool may = max_of<ST>(m) >= key_val(cur);
                if (__any_sync(0xffffffffu, may)) {
                    unsigned long long key = 0ull;
#pragma unroll
                    for (int j = 0; j < ST; ++j) {
                        const int64_t s = s0 + (j / 4) * kThreads * 4 + j % 4;
                        const uint32_t pos = GATHER ? id[GATHER ? j : 0] : (uint32_t)(s < A.n ? s : A.n - 1);
                        const unsigned long long c = may ? key_max(m[j], pos) : 0ull;
                        key = c > key ? c : key;
                    }
                    key = warp_max_u64(key);
                    if ((threadIdx.x & 31) == 0 && key > cur) mine[b] = key;
                    __syncwarp();
                }
            } else {
                // each quad's samples lie before the next one's
                StreamBest &best = b == 0 ? best0 : best1;
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    const float d[4] = {m[4 * q], m[4 * q + 1], m[4 * q + 2], m[4 * q + 3]};
                    best.take<1>(d, s0 + q * kThreads * 4, A.n);
                }
            }
        }
    }
    if constexpr (MANY || TM) {
        __syncthreads();
        for (int b = threadIdx.x; b < A.B; b += kThreads) {
            unsigned long long k = 0ull;
            for (int w = 0; w < NWP; ++w) k = wkey[w * A.B + b] > k ? wkey[w * A.B + b] : k;
            if (k > peek(&A.keys[b])) atomicMax(&A.keys[b], k);
        }
    } else {
        stream_finish(A, 0, best0.key(), red);
        if (A.B > 1) stream_finish(A, 1, best1.key(), red);
    }
}

// Any D: the attributes stream through, KC >= nodes x clusters accumulators in
// registers.
template <int KC, bool TM>
__global__ void __launch_bounds__(kThreads, KC <= 4 ? 4 : (KC <= 8 ? 2 : 1))
stream_max_wide(const PruneArgs A)
{
    extern __shared__ __align__(16) unsigned char smem[];
    ulonglong2 *box = reinterpret_cast<ulonglong2 *>(smem);   // [B * K][D]
    __shared__ unsigned long long red[kThreads / 32];
    stream_boxes(A, box);
    __syncthreads();
    const float *X = static_cast<const float *>(A.X);
    const int K = A.K, D = A.D, C = A.B * K;
    StreamBest best0, best1;
    for (int64_t base = (int64_t)blockIdx.x * (kThreads * 4); base < A.n; base += (int64_t)gridDim.x * (kThreads * 4)) {
        const int64_t s0 = base + (int64_t)threadIdx.x * 4;
        uint64_t e[KC][2], o[KC][2];
#pragma unroll
        for (int c = 0; c < KC; ++c) e[c][0] = e[c][1] = o[c][0] = o[c][1] = 0;
        int a = 0;
#pragma unroll 2
        for (; a + 1 < D; a += 2) {
            uint64_t x0[2], x1[2];
            load_quad(X + (size_t)a * A.ld, A.n, A.vec != 0, s0, x0);
            load_quad(X + (size_t)(a + 1) * A.ld, A.n, A.vec != 0, s0, x1);
            const uint64_t y0[2] = {swap2(x0[0]), swap2(x0[1])}, y1[2] = {swap2(x1[0]), swap2(x1[1])};
#pragma unroll
            for (int c = 0; c < KC; ++c)
                if (c < C) {
                    clamp_acc(x0, y0, box[c * D + a], e[c]);
                    clamp_acc(x1, y1, box[c * D + a + 1], o[c]);
                }
        }
        if (a < D) {
            uint64_t x0[2];
            load_quad(X + (size_t)a * A.ld, A.n, A.vec != 0, s0, x0);
            const uint64_t y0[2] = {swap2(x0[0]), swap2(x0[1])};
#pragma unroll
            for (int c = 0; c < KC; ++c)
                if (c < C) clamp_acc(x0, y0, box[c * D + a], e[c]);
        }
        float2 m0 = make_float2(0.f, 0.f), m1 = m0;
#pragma unroll
        for (int c = 0; c < KC; ++c)
            if (c < C) {
                const float2 d0 = upk(add2(e[c][0], o[c][0])), d1 = upk(add2(e[c][1], o[c][1]));
                const bool fresh = c == 0 || c == K;
                m0 = fresh ? d0 : make_float2(fminf(m0.x, d0.x), fminf(m0.y, d0.y));
                m1 = fresh ? d1 : make_float2(fminf(m1.x, d1.x), fminf(m1.y, d1.y));
                const float d[4] = {m0.x, m0.y, m1.x, m1.y};
                if (c != K - 1 && c != C - 1) continue;
                StreamBest &best = c == K - 1 ? best0 : best1;
                if constexpr (TM) {
                    const unsigned w = __reduce_max_sync(0xffffffffu, __float_as_uint(max_of<4>(d)));
                    const int64_t row = (base >> 7) + (threadIdx.x >> 5);
                    if ((threadIdx.x & 31) == 0 && row * kStreamTile < A.n)
                        A.tmax[(c == K - 1 ? 0 : A.rows) + row] = __uint_as_float(w);
                    best.v = fmaxf(best.v, __uint_as_float(w));
                } else {
                    best.take<1>(d, s0, A.n);
                }
            }
    }
    stream_finish(A, 0, best0.key(), red);
    if (A.B > 1) stream_finish(A, 1, best1.key(), red);
}

using StreamKernel = void (*)(const PruneArgs);

// Registers: a sample takes 4 D with its swapped copy, so D <= 4 keeps two
// quads a thread (half the box reads per sample) at 3 or 4 CTAs an SM.
template <int DC, int KC>
constexpr StreamKernel small_kernel(bool many, bool tm)
{
    constexpr int Q = DC <= 4 ? 2 : 1, CT = DC <= 2 ? 4 : 3;
    return tm ? stream_max_small<DC, KC, 1, CT, false, true>
              : (many ? stream_max_small<DC, KC, Q, CT, true, false> : stream_max_small<DC, KC, Q, CT, false, false>);
}
template <int DC>
StreamKernel small_kernel_k(int K, bool many, bool tm)
{
    return K == 3 ? small_kernel<DC, 3>(many, tm) : K == 4 ? small_kernel<DC, 4>(many, tm)
         : K == 5 ? small_kernel<DC, 5>(many, tm) : small_kernel<DC, 0>(many, tm);
}
StreamKernel small_kernel_of(int D, int K, bool many, bool tm)
{
    switch (D) {
    case 1: return small_kernel_k<1>(K, many, tm);
    case 2: return small_kernel_k<2>(K, many, tm);
    case 3: return small_kernel_k<3>(K, many, tm);
    case 4: return small_kernel_k<4>(K, many, tm);
    case 5: return small_kernel_k<5>(K, many, tm);
    case 6: return small_kernel_k<6>(K, many, tm);
    case 7: return small_kernel_k<7>(K, many, tm);
    default: return small_kernel_k<8>(K, many, tm);
    }
}
StreamKernel gather_kernel_of(int D)
{
    switch (D) {
    case 1: return stream_max_small<1, 0, 2, 4, true, false, true>;
    case 2: return stream_max_small<2, 0, 2, 4, true, false, true>;
    case 3: return stream_max_small<3, 0, 1, 4, true, false, true>;
    case 4: return stream_max_small<4, 0, 1, 4, true, false, true>;
    case 5: return stream_max_small<5, 0, 1, 3, true, false, true>;
    case 6: return stream_max_small<6, 0, 1, 3, true, false, true>;
    case 7: return stream_max_small<7, 0, 1, 3, true, false, true>;
    default: return stream_max_small<8, 0, 1, 3, true, false, true>;
    }
}
template <bool TM>
StreamKernel wide_kernel_of(int cols)
{
    return cols <= 4 ? stream_max_wide<4, TM> : (cols <= 8 ? stream_max_wide<8, TM> : stream_max_wide<16, TM>);
}

}  // namespace

cudaError_t launch_stream_f32(PruneArgs A, int sms, cudaStream_t stream)
{
    const bool tm = A.tmax != nullptr;
    const int Q = A.D <= 4 && !tm ? 2 : 1;
    const int64_t tiles = (A.n + kThreads * 4 * Q - 1) / (kThreads * 4 * Q);
    const size_t node = (size_t)A.K * A.D * 16 + (A.D <= 8 ? kThreads / 32 * 8 : 0);
    // node ranges so that the last round of CTAs leaves little idle (three CTAs an SM
    // are resident; loading a tile again costs about two nodes' evaluation)
    int per = A.B;
    if (A.D <= 8 && A.B > 2) {
        const int64_t slots = 3 * (int64_t)sms;
        int64_t best = INT64_MAX;
        for (int64_t r = 1; r <= A.B && (r - 1) * tiles < 8 * slots; ++r) {
            const int64_t nodes = (A.B + r - 1) / r, cost = (tiles * r + slots - 1) / slots * (2 + nodes);
            if (cost < best) { best = cost; per = (int)nodes; }
        }
    }
    per = (int)std::min<int64_t>(per, 46 * 1024 / node);   // (a launch's limit without opting in)
    A.per = per;
    const size_t smem = per * node;
    const StreamKernel fn = A.D <= 8 ? small_kernel_of(A.D, A.K, A.B > 2, tm)
                          : tm ? wide_kernel_of<true>(A.B * A.K) : wide_kernel_of<false>(A.B * A.K);
    int per_sm = 0;
    const cudaError_t r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kThreads, smem);
    if (r != cudaSuccess) return r;
    const dim3 grid((unsigned)std::max<int64_t>(1, std::min<int64_t>(tiles, (int64_t)std::max(1, per_sm) * sms)),
                    (unsigned)((A.B + per - 1) / per));
    fn<<<grid, kThreads, smem, stream>>>(A);
    return cudaGetLastError();
}

cudaError_t launch_stream_gather_f32(PruneArgs A, int sms, cudaStream_t stream)
{
    A.per = A.B;
    const int Q = A.D <= 2 ? 2 : 1;
    const size_t smem = (size_t)A.B * A.K * A.D * 16 + (size_t)kThreads / 32 * A.B * 8;
    const StreamKernel fn = gather_kernel_of(A.D);
    int per_sm = 0;
    const cudaError_t r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kThreads, smem);
    if (r != cudaSuccess) return r;
    const int64_t tiles = (A.n + kThreads * 4 * Q - 1) / (kThreads * 4 * Q);
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(tiles, (int64_t)std::max(1, per_sm) * sms));
    fn<<<grid, kThreads, smem, stream>>>(A);
    return cudaGetLastError();
}

}  // namespace kc
