// kc_exact.cu -- exact (double) maxima over samples of min_k ||x - box_k||^2:
// the objective of Eq. 1 at center sets (a set is K boxes lo = hi) for float
// and double data, and the node lower bound of Section 3.1 for double data.
//
// GB300 runs double arithmetic at 1/64 of its float rate, so almost none is
// done.  A float screen finds each node's largest float value M and, per tile
// of samples, the largest float value of the samples that may attain the exact
// maximum; float and exact value differ by a proved margin, so only samples
// whose float value reaches screen_floor(M) can.  A second kernel looks the
// tile values over and evaluates just those samples in double, in attribute
// order without contraction (bit-identical to a serial double evaluation), and
// keeps the largest value and the smallest position attaining it.
//
// Margins.  g = gamma of the float evaluation, g64 of the double one.  Float
// data: float and double value differ by a relative g + 2 g64, so
// c1^2 = (1 - G) / (1 + G).  Double data: a sample less the middle off of the
// data's range, rounded to float, is off by at most 2^-24 R per attribute
// (R = half the range); a box rounded inwards by at most 2^-23 (t + R) where t is
// the distance along the attribute.  With |R| the 2-norm over the attributes,
//   sqrt(exact) <= sqrt(float / (1 - g)) + 2^-24 |R|,
//   sqrt(exact) >= (sqrt(float (1 - g)) - 3 2^-24 |R|) / (1 + 2^-23),
// so c1 = (1 - g) / (1 + 2^-23) and eps = 4 2^-24 |R| (both with room for their
// own roundings).
//
// Small double problems skip the screen: every sample in double, the nodes
// spread over the SMs.
#include <cuda_runtime.h>

#include <cmath>

#include "kc_device.cuh"
#include "kc_internal.cuh"
#include "kc_prune.cuh"

namespace kc {

namespace {

__device__ __forceinline__ void raise128(ulonglong2 *p, double v, uint32_t pos)
{
    raise_key128(p, ord_f64(v), 0xFFFFFFFFull - pos);
}

__device__ __forceinline__ void warp_raise128(ulonglong2 *p, double v, uint32_t pos)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double v2 = __shfl_xor_sync(0xffffffffu, v, o);
        const uint32_t p2 = __shfl_xor_sync(0xffffffffu, pos, o);
        if (v2 > v || (v2 == v && p2 < pos)) { v = v2; pos = p2; }
    }
    if ((threadIdx.x & 31) == 0 && v >= 0.0) raise128(p, v, pos);
}

// Exact value of sample s: min over clusters, attribute order.
template <typename T>
__device__ double exact_value(const T *__restrict__ X, int64_t ld, int64_t s, const T *__restrict__ lo,
                              const T *__restrict__ hi, int K, int D)
{
    double e = __longlong_as_double(0x7ff0000000000000ll);
    for (int k = 0; k < K; ++k) {
        double acc = 0.0;
        for (int a = 0; a < D; ++a) {
            const double x = (double)X[(size_t)a * ld + s];
            const double d = __dsub_rn(x, mid3d((double)lo[k * D + a], x, (double)hi[k * D + a]));
            acc = __dadd_rn(acc, __dmul_rn(d, d));
        }
        if (acc < e) e = acc;
    }
    return e;
}

struct HitArgs {
    PruneArgs A;
    int T;                 // samples of a tmax row
    double gam, cut;       // nodes whose float value proves an exact value >= cut are skipped
    ulonglong2 *best;      // [B] exact maxima, zero before the screen
};

// Float data (double data have no cut: gam < 0): the screen proves value >= cut.
__device__ __forceinline__ bool node_cut(float m, double gam, double cut)
{
    return gam >= 0.0 && screen_proves(m, gam, cut);
}

// A CTA looks over 256 (node, tile) entries at a time: does the tile hold a
// sample that may attain the node's maximum?  All its threads then go through
// each such tile, four samples a thread at a time: in float, and those that
// reach the floor in double.  (The tiles of one sample far from everything are
// hits of every node; entries are ordered by node, so they meet different CTAs:
// with one warp to a hit and 32 nodes to a warp this took 375 us of 450.)
template <typename T>
__global__ void __launch_bounds__(256)
exact_hits_kernel(const HitArgs H)
{
    constexpr bool F64 = sizeof(T) == 8;
    constexpr int U = 4;
    __shared__ int64_t hits[256];
    __shared__ float floors[256];
    __shared__ int count;
    const PruneArgs &A = H.A;
    const int tid = threadIdx.x, K = A.K, D = A.D;
    const T *X = static_cast<const T *>(A.X);
    const int64_t total = A.rows * A.B;
    for (int64_t i0 = (int64_t)blockIdx.x * 256; i0 < total; i0 += (int64_t)gridDim.x * 256) {
        if (tid == 0) count = 0;
        __syncthreads();
        const int64_t i = i0 + tid;
        if (i < total) {
            const float m = key_val(A.keys[i / A.rows]), t = screen_floor(m, A.c1, A.eps);
            if (A.tmax[i] >= t && !node_cut(m, H.gam, H.cut)) {
                const int o = atomicAdd(&count, 1);
                hits[o] = i;
                floors[o] = t;
            }
        }
        __syncthreads();
        for (int o = 0; o < count; ++o) {
            const int64_t q = hits[o];
            const float tq = floors[o];
            const int b = (int)(q / A.rows);
            const int64_t s0 = q % A.rows * H.T, s1 = s0 + H.T < A.n ? s0 + H.T : A.n;
            const T *lo = static_cast<const T *>(A.lo) + (size_t)b * K * D;
            const T *hi = static_cast<const T *>(A.hi) + (size_t)b * K * D;
            double v = -1.0;
            uint32_t pos = 0xFFFFFFFFu;
            for (int64_t s = s0 + tid; s < s1; s += 256 * U) {
                float near[U];
#pragma unroll
                for (int u = 0; u < U; ++u) near[u] = __int_as_float(0x7f800000);
                for (int k = 0; k < K; ++k) {
                    // two chains over even and odd attributes, as the screen's
                    float acc[2][U];
#pragma unroll
                    for (int u = 0; u < U; ++u) acc[0][u] = acc[1][u] = 0.f;
                    for (int a = 0; a < D; ++a) {
                        float l, h, c[U];
                        if constexpr (F64) {
                            const double f = A.off[a];
                            l = __double2float_ru(__dsub_ru(lo[k * D + a], f));
                            h = __double2float_rd(__dsub_rd(hi[k * D + a], f));
#pragma unroll
                            for (int u = 0; u < U; ++u) {
                                const int64_t w = s + u * 256;
                                c[u] = __double2float_rn(X[(size_t)a * A.ld + (w < s1 ? w : s1 - 1)] - f);
                            }
                        } else {
                            l = lo[k * D + a];
                            h = hi[k * D + a];
#pragma unroll
                            for (int u = 0; u < U; ++u) {
                                const int64_t w = s + u * 256;
                                c[u] = X[(size_t)a * A.ld + (w < s1 ? w : s1 - 1)];
                            }
                        }
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            const float m = max3f(l - c[u], c[u] - h, 0.f);
                            if (a & 1) acc[1][u] = fmaf(m, m, acc[1][u]);
                            else acc[0][u] = fmaf(m, m, acc[0][u]);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u) near[u] = fminf(near[u], acc[0][u] + acc[1][u]);
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int64_t w = s + u * 256;
                    if (w < s1 && near[u] >= tq) {
                        const double e = exact_value<T>(X, A.ld, w, lo, hi, K, D);
                        if (e > v) { v = e; pos = (uint32_t)w; }   // (w increases)
                    }
                }
            }
            if (__any_sync(0xffffffffu, v >= 0.0)) warp_raise128(&H.best[b], v, pos);
        }
        __syncthreads();
    }
}

// Every sample in double: a CTA takes 256 samples and per nodes (blockIdx.y).
template <int DM>
__global__ void __launch_bounds__(256)
exact_direct_kernel(const double *__restrict__ X, int64_t ld, int64_t n, const double *__restrict__ lo,
                    const double *__restrict__ hi, int B, int per, int K, int D, ulonglong2 *__restrict__ best)
{
    const int64_t s = (int64_t)blockIdx.x * 256 + threadIdx.x;
    double x[DM];
#pragma unroll
    for (int a = 0; a < DM; ++a) x[a] = a < D ? X[(size_t)a * ld + (s < n ? s : n - 1)] : 0.0;
    const int b1 = min(B, (int)(blockIdx.y + 1) * per);
    for (int b = blockIdx.y * per; b < b1; ++b) {
        double e = __longlong_as_double(0x7ff0000000000000ll);
        for (int k = 0; k < K; ++k) {
            const double *l = lo + ((size_t)b * K + k) * D, *h = hi + ((size_t)b * K + k) * D;
            double acc = 0.0;
#pragma unroll
            for (int a = 0; a < DM; ++a)
                if (a < D) {
                    const double d = __dsub_rn(x[a], mid3d(__ldg(l + a), x[a], __ldg(h + a)));
                    acc = __dadd_rn(acc, __dmul_rn(d, d));
                }
            if (acc < e) e = acc;
        }
        // (the best value so far may be torn or old: only a filter)
        const unsigned long long cur = peek(&best[b].x);
        const bool may = ord_f64(e) >= cur;
        if (__any_sync(0xffffffffu, may)) warp_raise128(&best[b], may ? e : -1.0, (uint32_t)(s < n ? s : n - 1));
    }
}

// Exact maxima -> outputs; the keys and maxima go back to zero, as the next
// call wants them.  Bounds: val = raw value, lb deflated.  Sets proved >= cut
// by the screen: val = +inf, arg = -1.
__global__ void exact_finalize_kernel(unsigned long long *__restrict__ keys, ulonglong2 *__restrict__ best, int B,
                                      const uint32_t *__restrict__ ids, double gam, double cut, double defl, double slack,
                                      double *__restrict__ lb, double *__restrict__ val, int64_t *__restrict__ arg)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    const ulonglong2 k = best[b];
    const float m = key_val(keys[b]);
    best[b] = make_ulonglong2(0ull, 0ull);
    keys[b] = 0ull;
    if (node_cut(m, gam, cut)) {
        if (val) val[b] = __longlong_as_double(0x7ff0000000000000ll);
        if (arg) arg[b] = -1;
        return;
    }
    const bool none = k.x == 0ull;
    const double v = none ? 0.0 : unord_f64(k.x);
    if (val) val[b] = v;
    if (lb) lb[b] = certified_lb<double>(v, defl, slack);   // (only double data ask for it)
    if (arg) {
        const int64_t p = none ? -1 : (int64_t)(0xFFFFFFFFull - k.y);
        arg[b] = (p < 0 || !ids) ? p : (int64_t)ids[p];
    }
}

// Up to this many node x sample x cluster x attribute terms double data are
// evaluated directly.  Bounds, direct against screened, us: 0.1e6 terms 19 / 123,
// 1.9e6 43 / 358, 2.9e6 (D = 12) 61 / 173, 3.8e6 71 / 195, 19e6 305 / 74 (small sets
// leave much of the screen within its band, in one CTA's tile).
constexpr double kDirectTerms = 6e6;

using DirectFn = void (*)(const double *, int64_t, int64_t, const double *, const double *, int, int, int, int, ulonglong2 *);

}  // namespace

static double exact_screen_gamma(int D)
{
    return gamma_n(f32_roundings(D), kU32) + 2 * gamma_n(f64_roundings(D), kU64) + 1e-15;
}

namespace {

kc_status exact_max_chunk(kc_ctx *c, const View &v, const void *lo, const void *hi, int B, int K, double cut, double *lb,
                          double *val, int64_t *arg)
{
    const int D = c->D;
    const bool f64 = c->dt == KC_F64;
    const double g = gamma_n(f32_roundings(D), kU32), gam = exact_screen_gamma(D);
    const size_t kb = ((size_t)B * 8 + 255) & ~(size_t)255, need = kb + (size_t)B * 16;
    if (c->exact.bytes < need || c->exact_b < B) {
        // [keys][best]: zero between calls, laid out for the largest B so far
        KC_TRY(ensure(c, c->exact, need));
        c->exact_b = B;
        KC_CUDA(c, cudaMemsetAsync(c->exact.p, 0, c->exact.bytes, c->stream));
    }
    const size_t off = ((size_t)c->exact_b * 8 + 255) & ~(size_t)255;
    unsigned long long *keys = static_cast<unsigned long long *>(c->exact.p);
    ulonglong2 *best = reinterpret_cast<ulonglong2 *>(static_cast<char *>(c->exact.p) + off);
    bool screened = false;
    if (v.n > 0) {
        // beyond these ranges float distances could overflow
        const bool direct = f64 && ((double)v.n * B * K * D <= kDirectTerms || !(c->half_range < 1e15));
        if (direct) {
            const int64_t tiles = (v.n + 255) / 256;
            // nodes per CTA: about four CTAs an SM
            const int per = (int)std::max<int64_t>((B + 65534) / 65535,
                                                   std::max<int64_t>(1, tiles * B / (4 * c->num_sms)));
            const DirectFn fn = D <= 2 ? exact_direct_kernel<2> : D <= 4 ? exact_direct_kernel<4>
                              : D <= 8 ? exact_direct_kernel<8> : D <= 16 ? exact_direct_kernel<16>
                              : D <= 32 ? exact_direct_kernel<32> : D <= 64 ? exact_direct_kernel<64>
                                                                             : exact_direct_kernel<128>;
            const dim3 grid((unsigned)tiles, (unsigned)((B + per - 1) / per));
            fn<<<grid, 256, 0, c->stream>>>(static_cast<const double *>(v.X), v.ld, v.n, static_cast<const double *>(lo),
                                            static_cast<const double *>(hi), B, per, K, D, best);
            KC_TRY(after_launch(c, "exact maximum"));
        } else {
            screened = true;
            HitArgs H{};
            PruneArgs &A = H.A;
            A.X = v.X;
            A.ld = v.ld;
            A.n = v.n;
            A.lo = lo;
            A.hi = hi;
            A.B = B;
            A.K = K;
            A.D = D;
            A.keys = keys;
            const size_t es = f64 ? 8 : 4;
            A.vec = (uintptr_t)A.X % 16 == 0 && A.ld * es % 16 == 0;
            if (f64) {
                A.off = static_cast<const double *>(c->center.p);
                A.c1 = (float)((1.0 - g) / (1.0 + 1.2e-7) * (1.0 - 1e-6));
                A.eps = (float)(4 * kU32 * c->half_range * (1.0 + 1e-5));
            } else {
                A.c1 = (float)(std::sqrt((1.0 - gam) / (1.0 + gam)) * (1.0 - 1e-6));
            }
            const double cf = cut * (1.0 + gam) * (1.0 + 1e-6);   // a float value this large proves the cut
            A.cut = cf < 3e38 ? (float)cf : __builtin_huge_valf();
            const PruneEntry *e = f64 ? prune_pick(prune_table<true, true>(), D, v.n, c->num_sms, 0)
                                      : prune_pick(prune_table<false, true>(), D, v.n, c->num_sms, 0);
            const bool stream = !f64 && use_stream_f32(B, K, D);
            H.T = stream ? kStreamTile : e->T;
            const int64_t rows = (v.n + H.T - 1) / H.T;
            KC_TRY(ensure(c, c->tmax, (size_t)rows * B * 4));
            A.tmax = static_cast<float *>(c->tmax.p);
            A.rows = rows;
            if (stream) KC_CUDA(c, launch_stream_f32(A, c->num_sms, c->stream));
            else KC_CUDA(c, prune_run(e, A, true, c->num_sms, c->smem_optin > 0 ? c->smem_optin : 48 * 1024, 0, c->stream));
            ++c->launches;
            H.gam = f64 ? -1.0 : gam;
            H.cut = cut;
            H.best = best;
            const int grid = (int)std::min<int64_t>((rows * B + 255) / 256, (int64_t)c->num_sms * 8);
            if (f64) exact_hits_kernel<double><<<grid, 256, 0, c->stream>>>(H);
            else exact_hits_kernel<float><<<grid, 256, 0, c->stream>>>(H);
            KC_TRY(after_launch(c, "exact maximum of the screened samples"));
        }
    }
    exact_finalize_kernel<<<(B + 127) / 128, 128, 0, c->stream>>>(keys, best, B, v.ids, screened && !f64 ? gam : -1.0, cut,
                                                                  deflate_factor(c->dt, D), underflow_slack(c->dt, D), lb,
                                                                  val, arg);
    return after_launch(c, "exact maximum finalize");
}

}  // namespace

// lo, hi: [B][K][D] boxes in the data's type (device).  lb (with its deflation),
// val, arg: device, each may be NULL.  cut: see launch_objective.
kc_status launch_exact_max(kc_ctx *c, const View &v, const void *lo, const void *hi, int B, int K, double cut, double *lb,
                           double *val, int64_t *arg)
{
    // batches whose tile maxima (one float per node and 512 samples or so) stay
    // within 256 MiB
    const int64_t rows = v.n / 512 + 1;
    const int step = (int)std::max<int64_t>(16, std::min<int64_t>(B, ((int64_t)64 << 20) / rows / 8 * 8));
    const size_t box = (size_t)K * c->D * c->esize;
    for (int b0 = 0; b0 < B; b0 += step)
        KC_TRY(exact_max_chunk(c, v, static_cast<const char *>(lo) + b0 * box, static_cast<const char *>(hi) + b0 * box,
                               std::min(step, B - b0), K, cut, lb ? lb + b0 : nullptr, val ? val + b0 : nullptr,
                               arg ? arg + b0 : nullptr));
    return KC_OK;
}

}  // namespace kc
