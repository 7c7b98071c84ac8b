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

// Exact value of sample s: min over clusters, attribute order.  Few samples come here,
// so the loads of four attributes are in flight together.
template <typename T>
__device__ double exact_value(const T *__restrict__ X, int64_t ld, int64_t s, const T *__restrict__ lo,
                              const T *__restrict__ hi, int K, int D)
{
    constexpr int AH = 4;
    double e = __longlong_as_double(0x7ff0000000000000ll);
    for (int k = 0; k < K; ++k) {
        double acc = 0.0;
        for (int a0 = 0; a0 < D; a0 += AH) {
            T x[AH], l[AH], h[AH];
#pragma unroll
            for (int i = 0; i < AH; ++i) {
                const int a = a0 + i < D ? a0 + i : D - 1;
                x[i] = X[(size_t)a * ld + s];
                l[i] = lo[k * D + a];
                h[i] = hi[k * D + a];
            }
#pragma unroll
            for (int i = 0; i < AH; ++i) {
                if (a0 + i >= D) break;
                const double d = __dsub_rn((double)x[i], mid3d((double)l[i], (double)x[i], (double)h[i]));
                acc = __dadd_rn(acc, __dmul_rn(d, d));
            }
        }
        if (acc < e) e = acc;
    }
    return e;
}

struct HitArgs {
    PruneArgs A;
    int T;                 // samples of a tmax row
    int run;               // consecutive (node, tile) entries that a CTA looks over, a power of two <= 8
    double gam, cut;       // nodes whose float value proves an exact value >= cut are skipped
    ulonglong2 *best;      // [B] exact maxima, zero before the screen
};

// Float data (double data have no cut: gam < 0): the screen proves value >= cut.
__device__ __forceinline__ bool node_cut(float m, double gam, double cut)
{
    return gam >= 0.0 && screen_proves(m, gam, cut);
}

constexpr int kHitCtas = 4;      // CTAs per SM: the grid is resident at once
constexpr int kHitTile = 2048;   // most samples of a tmax row (of any kernel that fills tmax)

// A CTA looks over 256 (node, tile) entries at a time: does the tile hold a
// sample that may attain the node's maximum?  All its threads then go through
// each such tile in float, four samples a thread at a time, and list those that
// reach the floor; the listed ones are evaluated in double, one to a thread.
// Entries are dealt out in runs of at most eight, because the tiles of one sample
// far from everything are hits of every node, and all tiles of a node are hits
// where many samples attain its maximum: with 256 consecutive entries to a CTA, 16
// nodes of bound 0 over 1e5 samples (784 entries, all hits) kept four CTAs
// busy for 4.2 ms (now 0.05 ms a call; 64 double nodes of bound 0 over 1e6 samples 12.3,
// now 1.1 ms; 64 float center sets whose maximum 1e6 samples attain often 3.2, now 1.0).
//
// A node whose largest float value is within the margin of 0 keeps every sample
// (floor 0), but a sample inside a box has the exact value 0: it cannot beat the
// others, and among equal zeros the first sample wins, so that one alone is evaluated
// with those outside every box.  Being inside is decided on the ordered bits of the
// values (double comparisons would run at the rate of the double arithmetic that
// this saves).
template <typename T>
__global__ void __launch_bounds__(256, kHitCtas)
exact_hits_kernel(const HitArgs H)
{
    constexpr bool F64 = sizeof(T) == 8;
    // float data: a hit is bound by load latency, so four attributes are in flight (16
    // sets at N = 2e5, D = 29: 160 us a call, one attribute at a time 184); double
    // data: by the double arithmetic of the conversions
    constexpr int U = 4, AH = F64 ? 1 : 4;
    constexpr unsigned ALL = 0xffffffffu;
    using Ord = typename std::conditional<F64, uint64_t, uint32_t>::type;
    __shared__ int64_t hits[256];
    __shared__ float floors[256];
    __shared__ uint16_t list[kHitTile];   // samples of a hit that need the double value
    __shared__ int count, listed;
    // its node's boxes: float values, or (floor 0) ordered bits in the type's size
    extern __shared__ __align__(16) unsigned char boxes[];
    const PruneArgs &A = H.A;
    const int tid = threadIdx.x, lane = tid & 31, K = A.K, D = A.D, KD = K * D, run = H.run;
    float *flo = reinterpret_cast<float *>(boxes), *fhi = flo + KD;
    Ord *olo = reinterpret_cast<Ord *>(boxes), *ohi = olo + KD;
    auto ord = [](T v) {
        if constexpr (F64) return ord_f64(v);
        else return ord_f32(v);
    };
    const T *X = static_cast<const T *>(A.X);
    const int64_t total = A.rows * A.B;
    for (int64_t i0 = (int64_t)blockIdx.x * run; i0 < total; i0 += (int64_t)gridDim.x * 256) {
        if (tid == 0) count = 0;
        __syncthreads();
        const int64_t i = i0 + (int64_t)(tid / run) * gridDim.x * run + tid % run;
        if (i < total) {
            const float m = key_val(A.keys[i / A.rows]), t = screen_floor(m, A.c1, A.eps);
            if (A.tmax[i] >= t && !node_cut(m, H.gam, H.cut)) {
                const int o = atomicAdd(&count, 1);
                hits[o] = i;
                floors[o] = t > 0.f ? t : -1.f;   // -1: every sample outside the boxes
            }
        }
        __syncthreads();
        const int found = count;
        for (int o = 0; o < found; ++o) {
            const int64_t q = hits[o];
            const float tq = floors[o];
            const int b = (int)(q / A.rows);
            const int64_t s0 = q % A.rows * H.T, s1 = s0 + H.T < A.n ? s0 + H.T : A.n;
            const T *lo = static_cast<const T *>(A.lo) + (size_t)b * KD;
            const T *hi = static_cast<const T *>(A.hi) + (size_t)b * KD;
            if (tid == 0) listed = 0;
            for (int e = tid; e < KD; e += 256) {
                if (tq < 0.f) {
                    olo[e] = ord(lo[e]);
                    ohi[e] = ord(hi[e]);
                } else if constexpr (F64) {
                    const double f = A.off[e % D];
                    flo[e] = __double2float_ru(__dsub_ru(lo[e], f));
                    fhi[e] = __double2float_rd(__dsub_rd(hi[e], f));
                } else {
                    flo[e] = lo[e];
                    fhi[e] = hi[e];
                }
            }
            __syncthreads();
            for (int64_t s = s0 + tid; s - lane < s1; s += 256 * U) {   // (whole warps stay together)
                const int64_t left = s1 - (s - lane);
                const int nu = left > 256 * (U - 1) ? U : (int)((left + 255) / 256);   // of the U samples
                unsigned may = 0u;   // bit u: sample s + 256 u needs the double value
                if (tq < 0.f) {
                    unsigned in = 0u;
                    for (int k = 0; k < K && !__all_sync(ALL, in == (1u << nu) - 1u); ++k) {
                        unsigned inside = (1u << nu) - 1u;
                        for (int a = 0; a < D; ++a) {
                            const Ord l = olo[k * D + a], h = ohi[k * D + a];
#pragma unroll
                            for (int u = 0; u < U; ++u) {
                                if (u >= nu) break;
                                const int64_t w = s + u * 256;
                                const Ord x = ord(X[(size_t)a * A.ld + (w < s1 ? w : s1 - 1)]);
                                if (x < l || x > h) inside &= ~(1u << u);
                            }
                        }
                        in |= inside;
                    }
                    may = ~in;
                    if (s == 0) may |= 1u;
                } else {
                    unsigned reach = (1u << nu) - 1u;   // no distance below the floor so far
                    for (int k = 0; k < K && __any_sync(ALL, reach); ++k) {
                        // two chains over even and odd attributes, as the screen's
                        float acc[2][U];
#pragma unroll
                        for (int u = 0; u < U; ++u) acc[0][u] = acc[1][u] = 0.f;
                        for (int a0 = 0; a0 < D; a0 += AH) {
                            T x[AH][U];
#pragma unroll
                            for (int i = 0; i < AH; ++i)
#pragma unroll
                                for (int u = 0; u < U; ++u) {
                                    if (F64 && u >= nu) break;
                                    const int64_t w = s + u * 256;
                                    x[i][u] = X[(size_t)(a0 + i < D ? a0 + i : D - 1) * A.ld + (w < s1 ? w : s1 - 1)];
                                }
#pragma unroll
                            for (int i = 0; i < AH; ++i) {
                                if (a0 + i >= D) break;
                                const float l = flo[k * D + a0 + i], h = fhi[k * D + a0 + i];
#pragma unroll
                                for (int u = 0; u < U; ++u) {
                                    if (F64 && u >= nu) break;
                                    float c;
                                    if constexpr (F64) c = __double2float_rn(x[i][u] - A.off[a0 + i]);
                                    else c = x[i][u];
                                    const float m = max3f(l - c, c - h, 0.f);
                                    if ((a0 + i) & 1) acc[1][u] = fmaf(m, m, acc[1][u]);
                                    else acc[0][u] = fmaf(m, m, acc[0][u]);
                                }
                            }
                        }
#pragma unroll
                        for (int u = 0; u < U; ++u)
                            if (!(acc[0][u] + acc[1][u] >= tq)) reach &= ~(1u << u);
                    }
                    may = reach;
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int64_t w = s + u * 256;
                    const bool on = w < s1 && (may >> u & 1u);
                    const unsigned bal = __ballot_sync(ALL, on);
                    if (!bal) continue;
                    int at = 0;
                    if (lane == 0) at = atomicAdd(&listed, __popc(bal));
                    at = __shfl_sync(ALL, at, 0) + __popc(bal & ((1u << lane) - 1u));
                    if (on) list[at] = (uint16_t)(w - s0);
                }
            }
            __syncthreads();
            double v = -1.0;
            uint32_t pos = 0xFFFFFFFFu;
            for (int j = tid; j < listed; j += 256) {
                const int64_t w = s0 + list[j];
                const double e = exact_value<T>(X, A.ld, w, lo, hi, K, D);
                if (e > v || (e == v && (uint32_t)w < pos)) { v = e; pos = (uint32_t)w; }
            }
            if (__any_sync(ALL, v >= 0.0)) warp_raise128(&H.best[b], v, pos);
            __syncthreads();
        }
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
// evaluated directly.  Bounds, direct against screened, us: 0.1e6 terms 20 / 31, 1.9e6
// 36 / 37, 2.9e6 (D = 12) 61 / 65, 3.8e6 64 / 37, 7.7e6 117 / 41, 19e6 267 / 41.
constexpr double kDirectTerms = 3e6;

using DirectFn = void (*)(const double *, int64_t, int64_t, const double *, const double *, int, int, int, int, ulonglong2 *);

}  // namespace

static double exact_screen_gamma(int D)
{
    return gamma_n(f32_roundings(D), kU32) + 2 * gamma_n(f64_roundings(D), kU64) + 1e-15;
}

namespace {

// The screen of B nodes over n samples: the streaming kernel or e.
struct ScreenPlan {
    bool stream;
    const PruneEntry *e;
    int T;   // samples of a tmax row
};
ScreenPlan screen_plan(const kc_ctx *c, int64_t n, int B, int K)
{
    const bool f64 = c->dt == KC_F64;
    ScreenPlan p;
    p.e = f64 ? prune_pick(prune_table<true, true>(), c->D, n, c->num_sms, 0)
              : prune_pick(prune_table<false, true>(), c->D, n, c->num_sms, 0);
    p.stream = !f64 && use_stream_f32(B, K, c->D, n);
    p.T = p.stream ? kStreamTile : p.e->T;
    return p;
}

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
            const ScreenPlan plan = screen_plan(c, v.n, B, K);
            H.T = plan.T;
            const int64_t rows = (v.n + H.T - 1) / H.T;
            KC_TRY(ensure(c, c->tmax, (size_t)rows * B * 4));
            A.tmax = static_cast<float *>(c->tmax.p);
            A.rows = rows;
            if (plan.stream) KC_CUDA(c, launch_stream_f32(A, c->num_sms, c->stream));
            else KC_CUDA(c, prune_run(plan.e, A, true, c->num_sms, c->smem_optin > 0 ? c->smem_optin : 48 * 1024, 0, c->stream));
            ++c->launches;
            H.gam = f64 ? -1.0 : gam;
            H.cut = cut;
            H.best = best;
            if (H.T > kHitTile) return set_err(c, KC_EINTERNAL, "screen tile of %d samples", H.T);
            // short runs where there are few entries, so that they reach every SM; runs of
            // eight (one sector of tmax) where there are enough
            const int64_t most = (int64_t)c->num_sms * kHitCtas;
            H.run = 8;
            while (H.run > 1 && rows * B / H.run < 2 * most) H.run /= 2;
            const int grid = (int)std::min<int64_t>((rows * B + H.run - 1) / H.run, most);
            const auto fn = f64 ? exact_hits_kernel<double> : exact_hits_kernel<float>;
            const size_t smem = (size_t)2 * K * D * es;   // (at most 32 KiB, and 8 static)
            fn<<<grid, 256, smem, c->stream>>>(H);
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
    // batches whose tile maxima (one float per node and tile of the kernel that runs)
    // stay within 256 MiB; at most 65528 nodes, so that a launch's node ranges never
    // exceed its grid.  (N < 2^32 and tiles of at least 128 samples: at least one node.)
    const auto most = [&](int tile) {
        const int64_t s = ((int64_t)64 << 20) / ((v.n + tile - 1) / tile + 1);
        return (int)std::min<int64_t>({B, 65528, s >= 8 ? s / 8 * 8 : std::max<int64_t>(1, s)});
    };
    int step = most(screen_plan(c, v.n, B, K).T);
    if (step < B) step = std::min(step, most(screen_plan(c, v.n, step, K).T));   // (fewer nodes may be streamed)
    const size_t box = (size_t)K * c->D * c->esize;
    for (int b0 = 0; b0 < B; b0 += step)
        KC_TRY(exact_max_chunk(c, v, static_cast<const char *>(lo) + b0 * box, static_cast<const char *>(hi) + b0 * box,
                               std::min(step, B - b0), K, cut, lb ? lb + b0 : nullptr, val ? val + b0 : nullptr,
                               arg ? arg + b0 : nullptr));
    return KC_OK;
}

}  // namespace kc
