// kc_lb.cu -- node lower bound beta(M) = max_s min_k beta_s^k(M^k)
// (Section 3.1, Eqs. 9-11 with the closed-form minimiser mid{lo, x, hi}).
//
// Float data: batches of nodes take the pruning kernel (kc_prune.cuh), few
// nodes the streaming kernel (kc_stream.cu); both raise one (value, position)
// key per node with 64-bit atomics (the largest value, the smallest position
// on ties), which a small second kernel turns into the outputs.  Double data:
// the exact maxima of kc_exact.cu, in the serial order of operations.
#include <cuda_runtime.h>

#include <atomic>

#include "kc_device.cuh"
#include "kc_internal.cuh"
#include "kc_prune.cuh"

namespace kc {

namespace {

// Exact refinement of float-data lower bounds: each node comes with a float
// threshold below which no sample can attain the double maximum (from the
// float pass and its error bound); samples at or above it are re-evaluated in
// double in attribute order (mid{lo,x,hi}, separate multiply and add), so the
// node's value equals a serial double evaluation over all samples.
template <int DMAX>
__global__ void __launch_bounds__(kThreads)
lb_refine_f32(const float *__restrict__ X, int64_t ld, int64_t n, const float *__restrict__ lo,
              const float *__restrict__ hi, int B, int K, int D, const float *__restrict__ thr,
              double *__restrict__ pval, uint32_t *__restrict__ ppos)
{
    constexpr int NW = kThreads / 32;
    const int Dp = (D + 1) & ~1;
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t *sbox = reinterpret_cast<uint64_t *>(smem);                       // [B][K][Dp] (lo, -hi)
    float *sthr = reinterpret_cast<float *>(sbox + (size_t)B * K * Dp);
    double *wval = reinterpret_cast<double *>(sthr + ((B + 1) & ~1));          // [NW][B]
    uint32_t *wpos = reinterpret_cast<uint32_t *>(wval + NW * B);
    for (int i = threadIdx.x; i < B * K * Dp; i += kThreads) {
        const int a = i % Dp, bk = i / Dp;
        sbox[i] = a < D ? pk(lo[(size_t)bk * D + a], -hi[(size_t)bk * D + a]) : pk(0.f, -0.f);
    }
    for (int i = threadIdx.x; i < B; i += kThreads) sthr[i] = thr[i];
    for (int i = threadIdx.x; i < NW * B; i += kThreads) { wval[i] = -1.0; wpos[i] = 0xFFFFFFFFu; }
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int64_t s = (int64_t)blockIdx.x * kThreads + threadIdx.x; s - threadIdx.x < n;
         s += (int64_t)gridDim.x * kThreads) {
        const bool valid = s < n;
        uint64_t px[DMAX];
#pragma unroll
        for (int a = 0; a < DMAX; ++a) {
            const float v = (valid && a < D) ? X[(size_t)a * ld + s] : 0.f;
            px[a] = pk(v, -v);
        }
        for (int b = 0; b < B; ++b) {
            float best = __int_as_float(0x7f800000);
            for (int k = 0; k < K; ++k) {
                const uint64_t *bx = sbox + ((size_t)b * K + k) * Dp;
                uint64_t acc = 0;
#pragma unroll
                for (int a = 0; a < DMAX; a += 2)
                    if (a < Dp) {
                        const float2 t0 = upk(sub2(bx[a], px[a]));
                        const float2 t1 = upk(sub2(bx[a + 1], px[a + 1]));
                        const uint64_t m = pk(max3f(t0.x, t0.y, 0.f), max3f(t1.x, t1.y, 0.f));
                        acc = fma2(m, m, acc);
                    }
                const float2 sacc = upk(acc);
                best = fminf(best, sacc.x + sacc.y);
            }
            const bool cand = valid && best >= sthr[b];
            double e = -1.0;
            if (cand) {
                e = __longlong_as_double(0x7ff0000000000000ll);
                for (int k = 0; k < K; ++k) {
                    double acc = 0.0;
#pragma unroll
                    for (int a = 0; a < DMAX; ++a)
                        if (a < D) {
                            const double x = (double)upk(px[a]).x;
                            const double l = (double)lo[((size_t)b * K + k) * D + a];
                            const double h = (double)hi[((size_t)b * K + k) * D + a];
                            const double d = __dsub_rn(x, mid3d(l, x, h));
                            acc = __dadd_rn(acc, __dmul_rn(d, d));
                        }
                    if (acc < e) e = acc;
                }
            }
            const double cur = wval[w * B + b];
            const bool maybe = cand && e >= cur;
            if (__any_sync(0xffffffffu, maybe)) {
                double v = maybe ? e : -1.0;
                uint32_t p = maybe ? (uint32_t)s : 0xFFFFFFFFu;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const double v2 = __shfl_xor_sync(0xffffffffu, v, o);
                    const uint32_t p2 = __shfl_xor_sync(0xffffffffu, p, o);
                    if (v2 > v || (v2 == v && p2 < p)) { v = v2; p = p2; }
                }
                if (lane == 0 && (v > cur || (v == cur && p < wpos[w * B + b]))) {
                    wval[w * B + b] = v;
                    wpos[w * B + b] = p;
                }
                __syncwarp();
            }
        }
    }
    __syncthreads();
    for (int b = threadIdx.x; b < B; b += kThreads) {
        double v = -1.0;
        uint32_t p = 0xFFFFFFFFu;
        for (int q = 0; q < NW; ++q) {
            const double v2 = wval[q * B + b];
            const uint32_t p2 = wpos[q * B + b];
            if (v2 > v || (v2 == v && p2 < p)) { v = v2; p = p2; }
        }
        pval[(size_t)blockIdx.x * B + b] = v;
        ppos[(size_t)blockIdx.x * B + b] = p;
    }
}

constexpr int kMaxLeft = 256;   // flags of the pruning kernel's CTAs (an SM each) and one for all

// Keys (value bits, ~position) -> certified bound, value and sample per node.
// The keys (and the pruning kernel's flags) go back to zero, as the next launch
// wants them.
__global__ void lb_finalize_f32(unsigned long long *__restrict__ keys, int *__restrict__ left, int B,
                                const uint32_t *__restrict__ ids,
                                double defl, double slack, double *__restrict__ lb, double *__restrict__ lb_raw,
                                int64_t *__restrict__ arg)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (left && blockIdx.x == 0)
        for (int i = threadIdx.x; i < kMaxLeft; i += blockDim.x) left[i] = 0;
    if (b >= B) return;
    const unsigned long long m = keys[b];
    keys[b] = 0ull;
    const double raw = m ? (double)key_val(m) : 0.0;
    if (lb_raw) lb_raw[b] = raw;
    if (lb) lb[b] = certified_lb<float>(raw, defl, slack);
    if (arg) {
        const int64_t pos = m ? (int64_t)key_pos(m) : -1;
        arg[b] = (pos < 0 || !ids) ? pos : (int64_t)ids[pos];
    }
}

__global__ void lb_finalize_f64(const double *__restrict__ pval, const uint32_t *__restrict__ ppos,
                                int nparts, int B, const uint32_t *__restrict__ ids, double defl,
                                double slack, double *__restrict__ lb, double *__restrict__ lb_raw,
                                int64_t *__restrict__ arg)
{
    const int b = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (b >= B) return;
    double v = -1.0;
    uint32_t p = 0xFFFFFFFFu;
    for (int q = lane; q < nparts; q += 32) {
        const double v2 = pval[(size_t)q * B + b];
        const uint32_t p2 = ppos[(size_t)q * B + b];
        if (v2 > v || (v2 == v && p2 < p)) { v = v2; p = p2; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double v2 = __shfl_xor_sync(0xffffffffu, v, o);
        const uint32_t p2 = __shfl_xor_sync(0xffffffffu, p, o);
        if (v2 > v || (v2 == v && p2 < p)) { v = v2; p = p2; }
    }
    if (lane == 0) {
        const bool none = v < 0.0;
        const double raw = none ? 0.0 : v;
        if (lb_raw) lb_raw[b] = raw;
        if (lb) lb[b] = fmax(0.0, __dsub_rd(__dmul_rd(raw, defl), slack));
        if (arg) arg[b] = none ? -1 : (ids ? (int64_t)ids[p] : (int64_t)p);
    }
}

constexpr int64_t kSubsetBytes = (int64_t)128 << 20;   // of gathered rows at a time

// Rows of the samples named by ids: out[a * ldo + i] = X[a * ld + ids[i]].
__global__ void __launch_bounds__(256)
gather_rows_kernel(const float *__restrict__ X, int64_t ld, int D, const uint32_t *__restrict__ ids, int64_t n,
                   float *__restrict__ out, int64_t ldo)
{
    for (int64_t i0 = (int64_t)blockIdx.x * 1024; i0 < n; i0 += (int64_t)gridDim.x * 1024) {
        uint32_t id[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t i = i0 + j * 256 + threadIdx.x;
            id[j] = i < n ? ids[i] : 0u;
        }
        for (int a = 0; a < D; ++a)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int64_t i = i0 + j * 256 + threadIdx.x;
                if (i < n) out[(size_t)a * ldo + i] = __ldg(X + (size_t)a * ld + id[j]);
            }
    }
}

// ---------------------------------------------------------------- dispatch

// Launches the float maxima of A.B nodes into A.keys (zeroed by the caller, as
// A.left) on `stream`: full evaluation, or the pruning kernel and full evaluation
// of what it leaves.  st (samples per thread: 4 or 2, where both exist) and chunk (nodes
// per CTA) of 0 are chosen here.
cudaError_t launch_max_f32(PruneArgs A, int sms, size_t smem_cap, int st, int chunk, cudaStream_t stream,
                           int64_t *launches = nullptr)
{
    if (launches) ++*launches;
    A.vec = (uintptr_t)A.X % 16 == 0 && A.ld % 4 == 0;
    int *const left = A.left;
    A.left = nullptr;
    if (use_stream_f32(A.B, A.K, A.D, A.n)) return launch_stream_f32(A, sms, stream);
    const PruneEntry *e = prune_pick(prune_table<false, false>(), A.D, A.n, sms, st);
    A.T = e->T;
    A.gx = (int)std::min<int64_t>((A.n + e->T - 1) / e->T, sms);
    if (may_leave(A.B, A.D, (A.n + e->T - 1) / e->T <= sms) && A.gx < kMaxLeft) A.left = left;
    const cudaError_t r = prune_run(e, A, false, sms, smem_cap, chunk, stream);
    if (r != cudaSuccess || !A.left) return r;
    if (launches) ++*launches;
    return launch_stream_f32(A, sms, stream);
}

// The context's flags and keys of B nodes, all zero between calls.
kc_status ensure_keys(kc_ctx *c, int B)
{
    const size_t need = kMaxLeft * 4 + (size_t)B * 8;
    if (c->keys.bytes >= need) return KC_OK;
    KC_TRY(ensure(c, c->keys, need));
    KC_CUDA(c, cudaMemsetAsync(c->keys.p, 0, c->keys.bytes, c->stream));
    return KC_OK;
}
int *flags_of(const kc_ctx *c) { return static_cast<int *>(c->keys.p); }
unsigned long long *keys_of(const kc_ctx *c) { return reinterpret_cast<unsigned long long *>(flags_of(c) + kMaxLeft); }

template <typename F>
kc_status prep_kernel(kc_ctx *c, F fn, size_t smem, int *grid, int64_t tiles)
{
    if (smem > 48 * 1024)
        KC_CUDA(c, cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    KC_CUDA(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kThreads, smem));
    if (per_sm < 1) return set_err(c, KC_EINTERNAL, "lower-bound kernel does not fit (smem %zu)", smem);
    int64_t g = (int64_t)per_sm * c->num_sms;
    if (g > tiles) g = tiles;
    *grid = (int)(g < 1 ? 1 : g);
    return KC_OK;
}

}  // namespace

cudaError_t prune_run(const PruneEntry *e, PruneArgs A, bool tm, int sms, size_t smem_cap, int chunk, cudaStream_t stream)
{
    const int64_t tiles = (A.n + e->T - 1) / e->T;
    const auto bytes = [&](int nb) { return PruneLayout(nb, A.K, e->P, e->T, e->NT / 32, tm).end; };
    int per = std::min(A.B, 1 << 16);
    if (chunk > 0 && chunk < per) per = chunk;
    if (tiles < sms) {
        // few tiles: node ranges (whole groups) so that the last round of CTAs leaves
        // little idle; a range repeats the sort of its tile, about 16 nodes' worth (1e5
        // samples, D = 8, K = 5, 256 nodes: 280 us in one range, 212 in three; with more tiles than SMs
        // a second range cost up to 16 %)
        int64_t best = INT64_MAX;
        const int most = per;
        for (int64_t r = 1; r <= 4 * (int64_t)sms / tiles && r <= (A.B + kPG - 1) / kPG; ++r) {
            const int64_t nodes = std::min<int64_t>(most, ((A.B + r - 1) / r + kPG - 1) / kPG * kPG);
            const int64_t ranges = (A.B + nodes - 1) / nodes, cost = (tiles * ranges + sms - 1) / sms * (16 + nodes);
            if (cost < best) { best = cost; per = (int)nodes; }
        }
    }
    if (bytes(per) > smem_cap) {
        // as many nodes as fit, whole groups where there is more than one
        int fits = 0;   // (bytes(fits) <= smem_cap < bytes(per))
        while (per - fits > 1) {
            const int mid = fits + (per - fits) / 2;
            (bytes(mid) > smem_cap ? per : fits) = mid;
        }
        per = std::max(1, fits > kPG ? fits / kPG * kPG : fits);
    }
    A.per = per;
    const size_t smem = bytes(per);
    if (smem > smem_cap) return cudaErrorInvalidConfiguration;
    if (smem > 48 * 1024) {
        const cudaError_t r = cudaFuncSetAttribute(e->fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (r != cudaSuccess) return r;
    }
    // 512 threads at 128 registers fill an SM; of the smaller CTAs several fit (D = 128,
    // 3e5 samples, 8 nodes: 480 us with one, 286 with two)
    int per_sm = 1;
    if (e->NT < 512) {
        const cudaError_t r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, e->fn, e->NT, smem);
        if (r != cudaSuccess) return r;
        per_sm = std::max(1, per_sm);
    }
    // at most 65535 node ranges to a launch
    const int B = A.B, step = (int)std::min<int64_t>((int64_t)per * 65535, B);
    const size_t box = (size_t)A.K * A.D * (tm && A.off ? 8 : 4);
    if (tm && step < B) return cudaErrorInvalidConfiguration;   // (screens come in smaller batches)
    for (int b0 = 0; b0 < B; b0 += step) {
        PruneArgs C = A;
        C.B = std::min(step, B - b0);
        C.lo = static_cast<const char *>(A.lo) + b0 * box;
        C.hi = static_cast<const char *>(A.hi) + b0 * box;
        C.keys = A.keys + b0;
        const dim3 grid((unsigned)std::max<int64_t>(1, std::min<int64_t>(tiles, (int64_t)sms * per_sm)), (unsigned)((C.B + per - 1) / per));
        e->fn<<<grid, e->NT, smem, stream>>>(C);
        const cudaError_t r = cudaGetLastError();
        if (r != cudaSuccess) return r;
    }
    return cudaSuccess;
}

kc_status launch_lower_bounds_view(kc_ctx *c, const View &v, const void *lo, const void *hi, int B,
                                   double *lb, double *lb_raw, int64_t *arg, int st_override)
{
    return launch_lower_bounds_cfg(c, v, lo, hi, B, lb, lb_raw, arg, st_override, 0);
}

kc_status launch_lower_bounds_cfg(kc_ctx *c, const View &v, const void *lo, const void *hi, int B, double *lb,
                                  double *lb_raw, int64_t *arg, int st_override, int chunk_override)
{
    if (B <= 0) return KC_OK;
    const int D = c->D, K = c->K;
    const double defl = deflate_factor(c->dt, D), slack = underflow_slack(c->dt, D);
    const size_t smem_cap = c->smem_optin > 0 ? c->smem_optin : 48 * 1024;
    if (c->dt == KC_F32) {
        KC_TRY(ensure_keys(c, B));
        PruneArgs A{};
        A.X = v.X;
        A.ld = v.ld;
        A.n = v.n;
        A.lo = lo;
        A.hi = hi;
        A.B = B;
        A.K = K;
        A.D = D;
        A.keys = keys_of(c);
        A.left = flags_of(c);
        if (v.n > 0) {
            KC_CUDA(c, launch_max_f32(A, c->num_sms, smem_cap, st_override > 0 ? st_override : c->lb_st,
                                      chunk_override > 0 ? chunk_override : c->lb_chunk, c->stream,
                                      &c->launches));
        }
        lb_finalize_f32<<<(B + 127) / 128, 128, 0, c->stream>>>(A.keys, B > 2 && D <= 8 ? A.left : nullptr, B, v.ids, defl, slack, lb, lb_raw, arg);
        KC_TRY(after_launch(c, "lower bound finalize"));
    } else {
        KC_TRY(launch_exact_max(c, v, lo, hi, B, K, __builtin_huge_val(), lb, lb_raw, arg));
    }
    return KC_OK;
}

// Float bounds of B nodes over the samples named by ids [n] (device, D <= 8,
// every id below N): few nodes gather as they stream, batches gather the samples
// into rows of their own first (at most kSubsetBytes at a time, less where the device
// has no room for that) and prune.
kc_status launch_lower_bounds_subset(kc_ctx *c, const uint32_t *ids, int64_t n, const void *lo, const void *hi, int B,
                                     double *lb, double *lb_raw, int64_t *arg)
{
    const int D = c->D;
    KC_TRY(ensure_keys(c, B));
    PruneArgs A{};
    A.lo = lo;
    A.hi = hi;
    A.B = B;
    A.K = c->K;
    A.D = D;
    A.keys = keys_of(c);
    if (n > 0 && use_stream_f32(B, c->K, D, INT64_MAX)) {
        A.X = c->X;
        A.ld = c->ldx;
        A.n = n;
        A.ids = ids;
        A.vec = (uintptr_t)ids % 16 == 0;
        KC_CUDA(c, launch_stream_gather_f32(A, c->num_sms, c->stream));
        ++c->launches;
    } else if (n > 0) {
        int64_t chunk = std::min<int64_t>(n, kSubsetBytes / (4 * D) / 64 * 64), ld = 0;
        const std::string err = c->err;
        for (;; chunk = (chunk + 1) / 2) {
            ld = (chunk + 63) / 64 * 64;
            const kc_status st = ensure(c, c->work2, (size_t)ld * D * 4);
            if (st == KC_OK) break;
            if (st != KC_ENOMEM || chunk <= 4096) return st;
        }
        c->err = err;
        for (int64_t i0 = 0; i0 < n; i0 += chunk) {
            const int64_t m = std::min(chunk, n - i0);
            const int grid = (int)std::min<int64_t>((m + 1023) / 1024, (int64_t)c->num_sms * 8);
            gather_rows_kernel<<<grid, 256, 0, c->stream>>>(static_cast<const float *>(c->X), c->ldx, D, ids + i0, m,
                                                            static_cast<float *>(c->work2.p), ld);
            KC_TRY(after_launch(c, "subset gather"));
            A.X = c->work2.p;
            A.ld = ld;
            A.n = m;
            A.ids = ids + i0;
            A.vec = 1;
            KC_CUDA(c, prune_run(prune_pick(prune_table<false, false>(), D, m, c->num_sms, 0), A, false, c->num_sms,
                                 c->smem_optin > 0 ? c->smem_optin : 48 * 1024, 0, c->stream));
            ++c->launches;
        }
    }
    lb_finalize_f32<<<(B + 127) / 128, 128, 0, c->stream>>>(A.keys, nullptr, B, nullptr, deflate_factor(KC_F32, D),
                                                            underflow_slack(KC_F32, D), lb, lb_raw, arg);
    return after_launch(c, "lower bound finalize");
}

kc_status launch_lower_bounds(kc_ctx *c, const void *lo, const void *hi, int B, double *lb,
                              double *lb_raw, int64_t *argmax)
{
    return launch_lower_bounds_view(c, full_view(c), lo, hi, B, lb, lb_raw, argmax, 0);
}

// Double-precision refinement of float-data lower bounds (see lb_refine_f32):
// raw[b] is the float pass's value of node b; lb_out gets the certified bound
// from the serial double value, lb_exact_out (nullable) that double value.
kc_status launch_lower_bounds_refine(kc_ctx *c, const View &v, const void *lo, const void *hi, int B,
                                     const double *raw_host, double *lb_out, double *lb_exact_out, int64_t *arg)
{
    if (B <= 0) return KC_OK;
    if (c->dt != KC_F32) return set_err(c, KC_EINTERNAL, "refinement is for float data");
    const int D = c->D, K = c->K, NW = kThreads / 32, Dp = (D + 1) & ~1;
    const double gam = gamma_n(f32_roundings(D), kU32) + 2 * gamma_n(f64_roundings(D), kU64) + 1e-15;
    std::vector<float> thr(B);
    for (int b = 0; b < B; ++b) {
        double t = std::min(raw_host[b], 3.4028234663852886e38) / (1.0 + gam) * (1.0 - gam) * (1.0 - 1e-6) - 1e-37;
        float f = (float)t;
        if ((double)f > t) f = nextafterf(f, -1.f);
        thr[b] = t > 0 ? f : -1.f;
    }
    const size_t smem_cap = c->smem_optin > 0 ? c->smem_optin : 48 * 1024;
    const size_t per_node = (size_t)K * Dp * 8 + 4 + (size_t)NW * 12;
    const int chunk = (int)std::max<size_t>(1, std::min<size_t>((size_t)B, (smem_cap / 2) / per_node));
    const double defl = deflate_factor(KC_F64, D), slack = underflow_slack(KC_F64, D);
    for (int b0 = 0; b0 < B; b0 += chunk) {
        const int nb = std::min(chunk, B - b0);
        const size_t smem = (size_t)K * Dp * 8 * nb + (size_t)((nb + 1) & ~1) * 4 + (size_t)NW * 12 * nb;
        const int64_t tiles = (v.n + kThreads - 1) / kThreads;
        int grid = 1;
        auto kern = D <= 16 ? lb_refine_f32<16> : (D <= 64 ? lb_refine_f32<64> : lb_refine_f32<128>);
        KC_TRY(prep_kernel(c, kern, smem, &grid, tiles));
        const size_t thr_off = 0, part_off = 256 + (size_t)nb * 4;
        KC_TRY(ensure(c, c->part, part_off + (size_t)grid * nb * 12 + 256));
        char *pbuf = static_cast<char *>(c->part.p);
        float *dthr = reinterpret_cast<float *>(pbuf + thr_off);
        double *pval = reinterpret_cast<double *>(pbuf + ((part_off + 15) & ~(size_t)15));
        uint32_t *ppos = reinterpret_cast<uint32_t *>(pval + (size_t)grid * nb);
        KC_CUDA(c, cudaMemcpyAsync(dthr, thr.data() + b0, (size_t)nb * 4, cudaMemcpyHostToDevice, c->stream));
        const float *l = static_cast<const float *>(lo) + (size_t)b0 * K * D;
        const float *h = static_cast<const float *>(hi) + (size_t)b0 * K * D;
        if (v.n > 0) {
            kern<<<grid, kThreads, smem, c->stream>>>(static_cast<const float *>(v.X), v.ld, v.n, l, h, nb, K, D, dthr,
                                                      pval, ppos);
            KC_TRY(after_launch(c, "lower bound refinement"));
        }
        lb_finalize_f64<<<(nb + 3) / 4, 128, 0, c->stream>>>(pval, ppos, v.n > 0 ? grid : 0, nb, v.ids, defl, slack,
                                                             lb_out + b0, lb_exact_out ? lb_exact_out + b0 : nullptr,
                                                             arg ? arg + b0 : nullptr);
        KC_TRY(after_launch(c, "lower bound refinement finalize"));
        if (b0 + chunk < B) KC_CUDA(c, cudaStreamSynchronize(c->stream));   // thr upload reuses the buffer
    }
    return KC_OK;
}

// Times the launch shapes of the pruning kernel on the given node batch (samples
// per thread, where both exist, x nodes per CTA, whole groups) against the choice by
// size, and keeps one that is faster by more than timing noise in the context.
// Untimed work for the caller.
kc_status autotune_lower_bounds(kc_ctx *c, const void *lo, const void *hi, int B, double *lb_scratch, int *st_out,
                                int *chunk_out, float *ms_out)
{
    *st_out = 0;
    *chunk_out = 0;
    if (c->dt != KC_F32 || B <= 0) return KC_OK;
    const View v = full_view(c);
    const int D = c->D;
    const auto groups = [](int nodes) { return (nodes + kPG - 1) / kPG * kPG; };
    struct Shape {
        int st, chunk;
    };
    std::vector<Shape> shapes{{0, 0}};   // by size
    const bool fixed = use_stream_f32(B, c->K, D, v.n);   // evaluated in full: nothing to choose
    if (!fixed)
        for (int st : {4, 2}) {
            if (D > 8 && st == 2) break;   // one kernel
            for (int part = 1; part <= 4; ++part) {
                const int chunk = part == 1 ? B : groups((B + part - 1) / part);
                if (part == 1 || (chunk < B && chunk != shapes.back().chunk)) shapes.push_back({st, chunk});
            }
        }
    cudaEvent_t e0, e1;
    KC_CUDA(c, cudaEventCreate(&e0));
    if (cudaEventCreate(&e1) != cudaSuccess) {
        cudaEventDestroy(e0);
        return set_err(c, KC_ECUDA, "autotune: cudaEventCreate failed");
    }
    c->lb_st = c->lb_chunk = 0;
    float best = 0.f, limit = 0.f;
    Shape pick = shapes[0];
    kc_status st = KC_OK;
    for (const Shape &s : shapes) {
        st = launch_lower_bounds_cfg(c, v, lo, hi, B, lb_scratch, nullptr, nullptr, s.st, s.chunk);
        cudaEventRecord(e0, c->stream);
        for (int r = 0; r < 3 && st == KC_OK; ++r)
            st = launch_lower_bounds_cfg(c, v, lo, hi, B, lb_scratch, nullptr, nullptr, s.st, s.chunk);
        cudaEventRecord(e1, c->stream);
        if (st == KC_OK && cudaEventSynchronize(e1) != cudaSuccess) st = set_err(c, KC_ECUDA, "autotune: event sync failed");
        if (st != KC_OK) break;
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        ms /= 3.f;
        // (equal launches differ by less)
        if (&s == &shapes[0]) limit = 0.97f * (best = ms);
        else if (ms < limit && ms < best) { best = ms; pick = s; }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (st != KC_OK) return st;
    c->lb_st = D <= 8 ? pick.st : 0;
    c->lb_chunk = pick.chunk;
    if (!fixed) {
        *st_out = prune_pick(prune_table<false, false>(), D, v.n, c->num_sms, pick.st)->ST;
        *chunk_out = pick.chunk > 0 ? pick.chunk : B;
    }
    *ms_out = best;
    return KC_OK;
}

}  // namespace kc

// ------------------------------------------------------------------------
// kc_lower_bounds_noalloc: the float lower-bound kernels with their keys in a
// fixed device array instead of a context's buffers.
// Nothing here allocates; see include/kc.h for who needs this.

namespace kc {
namespace {

constexpr int kNoAllocMaxNodes = 4096;    // nodes per call
constexpr int kNoAllocMaxDevices = 64;

// The best key of each node of a call and the flags: 33 KiB, held by every GPU
// that loads the library until the process exits.
static __device__ __align__(256) unsigned long long g_noalloc_keys[kNoAllocMaxNodes + kMaxLeft / 2];   // (and the flags)

std::atomic<void *> g_noalloc_ptr[kNoAllocMaxDevices];

}  // namespace
}  // namespace kc

extern "C" kc_status kc_lower_bounds_noalloc(const float *X, int64_t N, int64_t ld, int32_t D, int32_t K,
                                             const float *lo, const float *hi, int32_t B, double *lb_out,
                                             double *lb_raw_out, int64_t *argmax_out, void *stream)
{
    using namespace kc;
    if (!X || !lo || !hi || !lb_out) return KC_EINVAL;
    if (K < 1 || K > kMaxK || D < 1 || D > kMaxD || N < 0 || ld < N || N > 4294967294ll) return KC_EINVAL;
    if (B < 0 || B > kNoAllocMaxNodes) return KC_EINVAL;   // more nodes than the fixed scratch is sized for
    if (B == 0) return KC_OK;
    // An error already pending in this thread belongs to earlier work: report
    // it without clearing it (cudaPeekAtLastError) and launch nothing.
    if (cudaPeekAtLastError() != cudaSuccess) return KC_ECUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoAllocMaxDevices) return KC_ECUDA;
    // Every array must be device memory of the current GPU: a host array
    // would make the kernels read or write through a host address.
    // cudaPointerGetAttributes allocates nothing.
    {
        const void *args[6] = {X, lo, hi, lb_out, lb_raw_out, argmax_out};
        for (const void *p : args) {
            if (!p) continue;
            cudaPointerAttributes a;
            if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
                cudaGetLastError();   // the error this query just raised
                return KC_EINVAL;
            }
            if ((a.type != cudaMemoryTypeDevice && a.type != cudaMemoryTypeManaged) || a.device != dev)
                return KC_EINVAL;
        }
    }
    // The host-side name of a __device__ array is not a device address: look
    // the address up once per device, with that device current.
    void *scratch = g_noalloc_ptr[dev].load();
    if (!scratch) {
        if (cudaGetSymbolAddress(&scratch, g_noalloc_keys) != cudaSuccess || !scratch) return KC_ECUDA;
        g_noalloc_ptr[dev].store(scratch);
    }
    int sms = 0, optin = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return KC_ECUDA;
    const double defl = deflate_factor(KC_F32, D), slack = underflow_slack(KC_F32, D);
    PruneArgs A{};
    A.X = X;
    A.ld = ld;
    A.n = N;
    A.lo = lo;
    A.hi = hi;
    A.B = B;
    A.K = K;
    A.D = D;
    A.keys = static_cast<unsigned long long *>(scratch);
    A.left = reinterpret_cast<int *>(A.keys + B);
    // the keys start from zero whatever an earlier call left (one whose last launch
    // failed): this array has no context that would end with the error
    if (cudaMemsetAsync(scratch, 0, (size_t)B * 8 + kMaxLeft * 4, st) != cudaSuccess) return KC_ECUDA;
    if (N > 0 && launch_max_f32(A, sms, (size_t)optin, 0, 0, st) != cudaSuccess) return KC_ECUDA;
    lb_finalize_f32<<<(B + 127) / 128, 128, 0, st>>>(A.keys, nullptr, B, nullptr, defl, slack, lb_out, lb_raw_out, argmax_out);
    if (cudaGetLastError() != cudaSuccess) return KC_ECUDA;
    return KC_OK;
}
