// kc_data.cu -- dataset ingest (attribute-major padded copy), the root region
// M0 of Section 2.1 (per-attribute min / max) with the non-finite check, and
// stream compaction of the surviving samples after sample reduction.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "kc_device.cuh"
#include "kc_internal.cuh"

namespace kc {

namespace {

// Rows s0 .. s0 + n of a row-major dataset, at src as [n][D] -> attribute-major
// dst[a * ld + s0 + i]; positions n_pad > n are zeroed.  A CTA takes tiles of rows
// as one contiguous read into shared memory (row stride D | 1, against bank
// conflicts) and writes each attribute's run, so every byte of src crosses the bus
// once: src may be pinned host memory, where the link (about 230 GB/s) bounds it.
// (From HBM an attribute at a time took the same 22 us for 32 MB at D = 8: the L2
// served the re-reads.)
constexpr int kRowTile = 24 * 1024;   // bytes of rows per tile

template <typename T>
__global__ void __launch_bounds__(256)
transpose_rows(const T *__restrict__ src, int64_t s0, int64_t n, int64_t n_pad, int D, int64_t ld, int rows, bool vec,
               T *__restrict__ dst)
{
    extern __shared__ __align__(16) unsigned char smem[];
    T *tile = reinterpret_cast<T *>(smem);
    constexpr int V = 16 / sizeof(T);
    const int st = D | 1;
    for (int64_t r0 = (int64_t)blockIdx.x * rows; r0 < n_pad; r0 += (int64_t)gridDim.x * rows) {
        const int m = (int)(n - r0 < rows ? (n - r0 > 0 ? n - r0 : 0) : rows), total = m * D;
        const int mp = (int)(n_pad - r0 < rows ? n_pad - r0 : rows);
        const T *from = src + r0 * D;
        __syncthreads();
        const int quads = vec ? total / V : 0;   // 16-byte reads (rows * D * sizeof(T) is a multiple of 16)
#pragma unroll 4
        for (int q = threadIdx.x; q < quads; q += 256) {
            union {
                uint4 u;
                T v[V];
            } w;
            w.u = *reinterpret_cast<const uint4 *>(from + (size_t)q * V);
            int i = q * V / D, a = q * V - i * D;
#pragma unroll
            for (int e = 0; e < V; ++e) {
                tile[i * st + a] = w.v[e];
                if (++a == D) { a = 0; ++i; }
            }
        }
        for (int e = quads * V + threadIdx.x; e < total; e += 256) tile[e / D * st + e % D] = from[e];
        __syncthreads();
        // lanes over the rows of one attribute
        for (int e = threadIdx.x; e < D * rows; e += 256) {
            const int a = e / rows, i = e - a * rows;
            if (i < mp) dst[(size_t)a * ld + s0 + r0 + i] = i < m ? tile[i * st + a] : T(0);
        }
    }
}

// Per-attribute min / max with order-preserving integer atomics (exact), and
// a flag for NaN / Inf.  Block y takes attribute y; 16-byte loads, four in flight
// a thread (bound by HBM: 320 MB in 49 us, 107 with 4-byte loads, one in flight).
template <typename T>
__global__ void __launch_bounds__(256)
root_box_kernel(const T *__restrict__ X, int64_t ld, int64_t N, unsigned long long *__restrict__ omin,
                unsigned long long *__restrict__ omax, int *__restrict__ nonfinite)
{
    constexpr int V = 16 / sizeof(T), U = 4;
    __shared__ unsigned long long red[2][8];
    const int a = blockIdx.y;
    const T *row = X + (size_t)a * ld;   // (rows are 256-byte aligned)
    using Key = typename std::conditional<sizeof(T) == 4, uint32_t, uint64_t>::type;
    Key mn = ~Key(0), mx = 0;
    bool bad = false;
    auto take = [&](T v) {
        bad |= !isfinite(v);
        Key o;
        if constexpr (sizeof(T) == 4) o = ord_f32(v);
        else o = ord_f64(v);
        mn = o < mn ? o : mn;
        mx = o > mx ? o : mx;
    };
    const int64_t quads = N / V, step = (int64_t)gridDim.x * 256 * U;
    for (int64_t q0 = (int64_t)blockIdx.x * 256 * U + threadIdx.x; q0 < quads; q0 += step) {
        union {
            uint4 u;
            T v[V];
        } w[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t q = q0 + u * 256;
            w[u].u = *reinterpret_cast<const uint4 *>(row + (q < quads ? q : q0) * V);
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int e = 0; e < V; ++e) take(w[u].v[e]);
    }
    if (blockIdx.x == 0 && threadIdx.x < N - quads * V) take(row[quads * V + threadIdx.x]);
    unsigned long long kn = mn, kx = mx;
    if (sizeof(T) == 4 && mn == ~Key(0)) kn = ~0ull;   // a thread without samples
    kn = ~warp_max_u64(~kn);
    kx = warp_max_u64(kx);
    bad = __any_sync(0xffffffffu, bad);
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        red[0][w] = kn;
        red[1][w] = kx;
        if (bad) atomicOr(nonfinite, 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < 8; ++i) {
            kn = red[0][i] < kn ? red[0][i] : kn;
            kx = red[1][i] > kx ? red[1][i] : kx;
        }
        atomicMin(&omin[a], kn);
        atomicMax(&omax[a], kx);
    }
}

__global__ void init_minmax(unsigned long long *omin, unsigned long long *omax, int D, int *flag)
{
    for (int a = threadIdx.x; a < D; a += blockDim.x) { omin[a] = ~0ull; omax[a] = 0ull; }
    if (threadIdx.x == 0 && flag) *flag = 0;
}

template <typename T>
__global__ void decode_minmax(const unsigned long long *omin, const unsigned long long *omax, int D, T *lo, T *hi)
{
    for (int a = threadIdx.x; a < D; a += blockDim.x) {
        if constexpr (sizeof(T) == 4) {
            lo[a] = unord_f32((uint32_t)omin[a]);
            hi[a] = unord_f32((uint32_t)omax[a]);
        } else {
            lo[a] = unord_f64(omin[a]);
            hi[a] = unord_f64(omax[a]);
        }
    }
}

}  // namespace

kc_status launch_ingest(kc_ctx *c, const void *src_dev, kc_layout layout, int64_t N, int D)
{
    // src_dev is device memory holding the caller's layout.
    if (layout == KC_COL_MAJOR) {
        KC_CUDA(c, cudaMemcpy2DAsync(c->X, c->ldx * c->esize, src_dev, N * c->esize, N * c->esize, D,
                                     cudaMemcpyDeviceToDevice, c->stream));
        if (c->ldx > N)
            KC_CUDA(c, cudaMemset2DAsync(static_cast<char *>(c->X) + N * c->esize, c->ldx * c->esize, 0,
                                         (c->ldx - N) * c->esize, D, c->stream));
        return KC_OK;
    }
    return launch_ingest_rows(c, src_dev, 0, N, true);
}

kc_status launch_ingest_rows(kc_ctx *c, const void *rows_dev, int64_t s0, int64_t n, bool pad)
{
    if (n <= 0) return KC_OK;
    const int64_t n_pad = pad ? c->ldx - s0 : n;
    // whole 16-byte groups to a tile, whatever D
    const int rows = std::max(16, kRowTile / (int)(c->esize * c->D) / 16 * 16);
    const size_t smem = (size_t)rows * (c->D | 1) * c->esize;
    const bool vec = (uintptr_t)rows_dev % 16 == 0;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((n_pad + rows - 1) / rows, (int64_t)c->num_sms * 8));
    if (c->dt == KC_F32)
        transpose_rows<float><<<grid, 256, smem, c->stream>>>(static_cast<const float *>(rows_dev), s0, n, n_pad, c->D,
                                                              c->ldx, rows, vec, static_cast<float *>(c->X));
    else
        transpose_rows<double><<<grid, 256, smem, c->stream>>>(static_cast<const double *>(rows_dev), s0, n, n_pad, c->D,
                                                               c->ldx, rows, vec, static_cast<double *>(c->X));
    return after_launch(c, "ingest transpose");
}

kc_status launch_root_box(kc_ctx *c, void *lo, void *hi, int *nonfinite_dev)
{
    const int D = c->D;
    KC_TRY(ensure(c, c->part, (size_t)2 * kMaxD * 8 + 16));
    unsigned long long *omin = static_cast<unsigned long long *>(c->part.p);
    unsigned long long *omax = omin + kMaxD;
    init_minmax<<<1, 64, 0, c->stream>>>(omin, omax, D, nonfinite_dev);
    KC_TRY(after_launch(c, "root box init"));
    const int64_t tiles = (c->N * (int64_t)c->esize + 16 * 1024 - 1) / (16 * 1024);
    const dim3 grid((unsigned)std::max<int64_t>(1, std::min<int64_t>(tiles, (8 * c->num_sms + D - 1) / D)), (unsigned)D);
    if (c->dt == KC_F32)
        root_box_kernel<float><<<grid, 256, 0, c->stream>>>(static_cast<const float *>(c->X), c->ldx, c->N, omin, omax,
                                                            nonfinite_dev);
    else
        root_box_kernel<double><<<grid, 256, 0, c->stream>>>(static_cast<const double *>(c->X), c->ldx, c->N, omin, omax,
                                                             nonfinite_dev);
    KC_TRY(after_launch(c, "root box"));
    if (c->dt == KC_F32)
        decode_minmax<float><<<1, 64, 0, c->stream>>>(omin, omax, D, static_cast<float *>(lo),
                                                      static_cast<float *>(hi));
    else
        decode_minmax<double><<<1, 64, 0, c->stream>>>(omin, omax, D, static_cast<double *>(lo),
                                                       static_cast<double *>(hi));
    return after_launch(c, "root box decode");
}

// ------------------------------------------------------------ compaction
// Stable stream compaction of the samples a mask keeps: per-block counts,
// one exclusive scan, then a scatter that preserves sample order (so
// positions stay ordered like sample indices).

namespace {

constexpr int kCompPer = 16;                       // samples per thread
constexpr int kCompBlock = 256 * kCompPer;         // samples per block

__global__ void comp_count(const uint8_t *__restrict__ mask, int64_t n, unsigned *__restrict__ counts)
{
    const int64_t b0 = (int64_t)blockIdx.x * kCompBlock;
    unsigned c = 0;
    for (int i = threadIdx.x; i < kCompBlock; i += 256) {
        const int64_t s = b0 + i;
        if (s < n && mask[s]) ++c;
    }
    __shared__ unsigned red[8];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned t = 0;
        for (int w = 0; w < 8; ++w) t += red[w];
        counts[blockIdx.x] = t;
    }
}

// Exclusive scan of nb counts by one block of 1024 threads; total -> *total.
__global__ void comp_scan(unsigned *__restrict__ counts, int64_t nb, unsigned long long *__restrict__ total)
{
    __shared__ unsigned long long part[1024];
    const int64_t per = (nb + 1023) / 1024;
    const int64_t s0 = threadIdx.x * per, s1 = (s0 + per < nb) ? s0 + per : nb;
    unsigned long long acc = 0;
    for (int64_t i = s0; i < s1; ++i) acc += counts[i];
    part[threadIdx.x] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long run = 0;
        for (int i = 0; i < 1024; ++i) {
            const unsigned long long v = part[i];
            part[i] = run;
            run += v;
        }
        *total = run;
    }
    __syncthreads();
    unsigned long long run = part[threadIdx.x];
    for (int64_t i = s0; i < s1; ++i) {
        const unsigned v = counts[i];
        counts[i] = (unsigned)run;
        run += v;
    }
}

template <typename T>
__global__ void comp_scatter(const T *__restrict__ X, int64_t ld, int64_t n, int D, const uint32_t *__restrict__ ids,
                             const uint8_t *__restrict__ mask, const unsigned *__restrict__ offs, T *__restrict__ Xo,
                             int64_t ldo, uint32_t *__restrict__ ido)
{
    __shared__ unsigned wsum[8];
    const int64_t b0 = (int64_t)blockIdx.x * kCompBlock;
    unsigned base = offs[blockIdx.x];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int r = 0; r < kCompPer; ++r) {
        const int64_t s = b0 + (int64_t)r * 256 + threadIdx.x;
        const bool keep = s < n && mask[s];
        const unsigned bal = __ballot_sync(0xffffffffu, keep);
        if (lane == 0) wsum[w] = __popc(bal);
        __syncthreads();
        unsigned before = 0, tot = 0;
        for (int q = 0; q < 8; ++q) {
            if (q < w) before += wsum[q];
            tot += wsum[q];
        }
        if (keep) {
            const unsigned p = base + before + __popc(bal & ((1u << lane) - 1u));
            for (int a = 0; a < D; ++a) Xo[(size_t)a * ldo + p] = X[(size_t)a * ld + s];
            ido[p] = ids ? ids[s] : (uint32_t)s;
        }
        base += tot;
        __syncthreads();
    }
}

}  // namespace

kc_status launch_compact(kc_ctx *c, const View &v, const uint8_t *mask, void *Xo, int64_t ldo, uint32_t *ido,
                         unsigned *scratch_counts, unsigned long long *total_dev)
{
    const int64_t nb = (v.n + kCompBlock - 1) / kCompBlock;
    if (nb == 0) {
        KC_CUDA(c, cudaMemsetAsync(total_dev, 0, 8, c->stream));
        return KC_OK;
    }
    comp_count<<<(unsigned)nb, 256, 0, c->stream>>>(mask, v.n, scratch_counts);
    KC_TRY(after_launch(c, "compaction count"));
    comp_scan<<<1, 1024, 0, c->stream>>>(scratch_counts, nb, total_dev);
    KC_TRY(after_launch(c, "compaction scan"));
    if (c->dt == KC_F32)
        comp_scatter<float><<<(unsigned)nb, 256, 0, c->stream>>>(static_cast<const float *>(v.X), v.ld, v.n, c->D, v.ids,
                                                                 mask, scratch_counts, static_cast<float *>(Xo), ldo, ido);
    else
        comp_scatter<double><<<(unsigned)nb, 256, 0, c->stream>>>(static_cast<const double *>(v.X), v.ld, v.n, c->D,
                                                                  v.ids, mask, scratch_counts, static_cast<double *>(Xo),
                                                                  ldo, ido);
    return after_launch(c, "compaction scatter");
}

int64_t compact_blocks(int64_t n) { return (n + kCompBlock - 1) / kCompBlock; }

}  // namespace kc
