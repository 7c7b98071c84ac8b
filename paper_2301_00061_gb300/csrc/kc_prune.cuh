// kc_prune.cuh -- the max over samples of the min over clusters of a clamp (or
// point) distance, for a batch of nodes, without evaluating most of the
// (node, sample, cluster) terms.
//
// The result of a node is one maximum, so a sample only matters while its
// value may reach the largest value found so far, and one cluster's distance
// is enough to rule it out (the minimum over clusters is no larger).  Three
// tests use that, each on 32 ST samples of a warp at once:
//   supergroup (64 nodes), group (8 nodes): the distance to the box
//     [max lo, min hi] over the group's boxes of one cluster bounds the
//     distance to every one of them from above -- also when that box is
//     inverted, as max(lo - x, x - hi, 0) grows with lo and falls with hi; in
//     float the same holds of the evaluated values, because every rounding
//     involved (difference, maximum, fused multiply-add, sum) is monotone;
//   node: the distance to the node's own box of that cluster.
// A warp goes on to the remaining clusters only when some lane passes.  The
// tests dismiss only what cannot win (a value equal to the best is evaluated
// unless the best one's position lies before the tile), so the maximum and the
// smallest position attaining it are those of the full evaluation, bit for bit.
// Where the group tests dismiss nothing, the node tests cost one cluster's
// evaluation more; at few attributes such batches are left to the streaming kernel
// after the first group tests (may_leave).  Nodes of bound 0 (each sample in some
// box): 256 nodes at N = 1e7, D = 8, K = 5 take 8.9 ms, 17.4 when ties passed every
// test, 12.4 evaluated in full; at N = 1e6, D = 2, K = 4 0.44 ms, 1.19 and 0.43.
//
// For the one cluster to be the right one for a whole warp, a CTA sorts each
// tile of samples by the nearest of K reference points (the box centers of the
// middle node) in shared memory; first[b][r] names the cluster of node b
// nearest to reference r.  The group tests run first, on strips of 32 ST
// samples, and queue what they leave: (strip, group) items where many samples
// survive, (sample, group) pairs, packed one to a lane, where few do; the node
// tests queue (sample, node) pairs in the same way.  All warps share the
// queues, because the samples that matter are few and sorted together: with
// each warp going through its own samples, the one that held the far ones took
// 3.8 ms where the queues take 0.41 ms (N = 1e7, D = 8, K = 5, 256 nested nodes;
// every term evaluated: 11.5 ms).  Each CTA starts from the values of the 32
// samples of its first tile farthest from their references, and the CTAs share
// their best values once per tile through the global keys.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "kc_device.cuh"
#include "kc_internal.cuh"

namespace kc {

constexpr int kPG = 8;    // nodes per group
constexpr int kPSG = 8;   // groups per supergroup
constexpr int kSparse = 8;       // survivors of 32 samples up to which a group test packs them as pairs

struct PruneArgs {
    const void *X;            // attribute-major samples [D][ld]
    int64_t ld, n;
    const void *lo, *hi;      // [B][K][D] in the samples' type
    int B, K, D;
    int per;                  // nodes per CTA range (blockIdx.y)
    const uint32_t *ids;      // NULL, or the names of the samples: keys hold ids[position]
    int vec;                  // rows may be read with 16-byte loads (X 16-byte aligned, ld a multiple of 16 bytes)
    unsigned long long *keys; // [B] (value bits, ~position), zero before the launch
    // screens of an exact maximum (kc_exact.cu): the largest float value of each
    // node in each tile, of all samples that may attain the exact maximum
    float *tmax;              // [B][rows], a row a tile
    int64_t rows;
    // screens: a sample that may attain the maximum has a float value that reaches
    // screen_floor(best, c1, eps); off [D] is subtracted from double data before the
    // conversion to float.  Bounds: left, NULL or [gx + 1] zeros, says which of the
    // pruning kernel's gx CTAs (by blockIdx.x) left their samples, tiles of T, to the
    // streaming kernel, and at [gx] whether any did.  (One struct of the size it
    // had: with 16 bytes more the streaming kernel took 150 us for 146.)
    union { float c1; int gx; };
    union { float eps; int T; };
    float cut;                // screens: nodes proved to reach this float value are done
    union { const double *off; int *left; };
};

// Below this float value a sample cannot attain a maximum whose largest float
// value is m (rounded down; 0: any may): (c1 sqrt(m) - eps)^2.
__device__ __forceinline__ float screen_floor(float m, float c1, float eps)
{
    const float s = __fsub_rd(__fmul_rd(__fsqrt_rd(fminf(m, 3.0e38f)), c1), eps);
    return s > 0.f ? fmaxf(__fsub_rd(__fmul_rd(s, s), 1e-37f), 0.f) : 0.f;
}

// Threads and samples per thread of the kernel for P attribute pairs: the tile
// of NT ST samples stays in shared memory (8 P bytes each, 64 KB or so) beside
// the boxes; 512 threads at 128 registers fill the register file.
template <int P>
struct PruneShape {
    static constexpr int NT = P <= 16 ? 512 : (P <= 34 ? 256 : 128);
    static constexpr int ST = P <= 4 ? 4 : (P <= 8 ? 2 : 1);
};

// 16-byte words of a box row: odd, so that lanes reading the same word of
// different rows spread over the banks.
__host__ __device__ constexpr int row_words(int P) { return P | 1; }

// Entries of each pair queue.
__host__ __device__ constexpr int pair_cap(int P) { return P <= 2 ? 4096 : 2048; }

__host__ __device__ inline size_t al16(size_t v) { return (v + 15) & ~(size_t)15; }

// Shared memory of a CTA with nb nodes, K clusters, P pairs and a tile of T samples.
struct PruneLayout {
    size_t box, gbox, sbox, stage, ref, cand, key, thr, gmin, smin, hist, pos, queue, tmx, fk, fg, fs, rr, end;
    __host__ __device__ PruneLayout(int nb, int K, int P, int T, int warps, bool tm)
    {
        const int ng = (nb + kPG - 1) / kPG, ns = (ng + kPSG - 1) / kPSG;
        size_t o = 0;
        const size_t row = (size_t)row_words(P) * 16;
        box = o; o += nb * K * row;
        gbox = o; o += ng * K * row;
        sbox = o; o += ns * K * row;
        stage = o; o += (size_t)P * T * 8;
        ref = o; o += al16((size_t)K * P * 8);
        cand = o; o += 32 * 8;
        key = o; o += al16((size_t)nb * 8);
        thr = o; o += al16((size_t)nb * 4);
        gmin = o; o += al16((size_t)ng * 4);
        smin = o; o += al16((size_t)ns * 4);
        hist = o; o += (2 * kMaxK + 4) * 4;   // counts, bases, queue lengths
        pos = o; o += (size_t)T * 4;
        queue = o; o += al16((size_t)warps * ng * 4) + (size_t)2 * pair_cap(P) * 4;
        tmx = o; o += tm ? al16((size_t)nb * 4) : 0;
        fk = o; o += al16((size_t)nb * K);
        fg = o; o += al16((size_t)ng * K);
        fs = o; o += al16((size_t)ns * K);
        rr = o; o += al16(T);
        end = o;
    }
};

// Distances of ST samples to one box (q.x = (lo_2p, lo_2p+1), q.y = (hi_2p, hi_2p+1)).
// Each attribute's max(lo - x, x - hi, 0), squares in two interleaved fused
// chains: the evaluation of box_dist_f32, with half the registers per sample.
// PT: the box is the point q.x (lo = hi); the same value, as |x - c| squared.
template <int ST, int P, bool PT = false>
__device__ __forceinline__ void box_dists(const uint64_t (&x)[ST][P], const ulonglong2 *bx, float (&d)[ST])
{
    uint64_t acc[ST];
#pragma unroll
    for (int j = 0; j < ST; ++j) acc[j] = 0;
#pragma unroll
    for (int p = 0; p < P; ++p) {
        if constexpr (PT) {
            const uint64_t c = bx[p].x;
#pragma unroll
            for (int j = 0; j < ST; ++j) {
                const uint64_t t = sub2(x[j][p], c);
                acc[j] = fma2(t, t, acc[j]);
            }
            continue;
        }
        const ulonglong2 q = bx[p];
#pragma unroll
        for (int j = 0; j < ST; ++j) {
            const float2 t0 = upk(sub2(q.x, x[j][p])), t1 = upk(sub2(x[j][p], q.y));
            const uint64_t m = pk(max3f(t0.x, t1.x, 0.f), max3f(t0.y, t1.y, 0.f));
            acc[j] = fma2(m, m, acc[j]);
        }
    }
#pragma unroll
    for (int j = 0; j < ST; ++j) {
        const float2 s = upk(acc[j]);
        d[j] = s.x + s.y;
    }
}

// A key another CTA may be raising (never from L1).
__device__ __forceinline__ unsigned long long peek(const unsigned long long *p)
{
    return *reinterpret_cast<const volatile unsigned long long *>(p);
}

template <int ST>
__device__ __forceinline__ float max_of(const float (&d)[ST])
{
    float m = d[0];
#pragma unroll
    for (int j = 1; j < ST; ++j) m = fmaxf(m, d[j]);
    return m;
}

// ST consecutive samples from s0 as attribute pairs; positions past n - 1 read
// sample n - 1 again (the same key, so nothing changes).
template <int ST, int P>
__device__ __forceinline__ void load_samples(const float *__restrict__ X, int64_t ld, int64_t n, int D, bool vec,
                                             int64_t s0, uint64_t (&x)[ST][P])
{
    const bool full = vec && s0 + ST <= n;
#pragma unroll
    for (int p = 0; p < P; ++p) {
        float v[2][ST];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int a = 2 * p + h;
#pragma unroll
            for (int j = 0; j < ST; ++j) v[h][j] = 0.f;
            if (a < D) {
                const float *row = X + (size_t)a * ld;
                if (full) {
                    if constexpr (ST % 4 == 0) {
#pragma unroll
                        for (int j = 0; j < ST; j += 4) {
                            const float4 q = __ldg(reinterpret_cast<const float4 *>(row + s0 + j));
                            v[h][j] = q.x; v[h][j + 1] = q.y; v[h][j + 2] = q.z; v[h][j + 3] = q.w;
                        }
                    } else if constexpr (ST == 2) {
                        const float2 q = __ldg(reinterpret_cast<const float2 *>(row + s0));
                        v[h][0] = q.x; v[h][1] = q.y;
                    } else {
                        v[h][0] = __ldg(row + s0);
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < ST; ++j) v[h][j] = __ldg(row + (s0 + j < n ? s0 + j : n - 1));
                }
            }
        }
#pragma unroll
        for (int j = 0; j < ST; ++j) x[j][p] = pk(v[0][j], v[1][j]);
    }
}

// The references of a strip's samples (lane l: slots 32 j + l); true when the
// strip has only one (slots are sorted).
template <int ST>
__device__ __forceinline__ bool strip_refs(const uint8_t *rr, int lane, uint8_t (&rj)[ST])
{
#pragma unroll
    for (int j = 0; j < ST; ++j) rj[j] = rr[j * 32 + lane];
    return rr[0] == rr[32 * ST - 1];
}

// Distances of a strip to the boxes named by first[reference].
template <int ST, int P, bool PT = false>
__device__ __forceinline__ void strip_dists(const uint64_t (&x)[ST][P], const ulonglong2 *rows, const uint8_t *first,
                                            const uint8_t (&rj)[ST], bool one, float (&d)[ST])
{
    if (one) {
        box_dists<ST, P, PT>(x, rows + first[rj[0]] * row_words(P), d);
    } else {
#pragma unroll
        for (int j = 0; j < ST; ++j) {
            float e[1];
            box_dists<1, P, PT>(reinterpret_cast<const uint64_t (&)[1][P]>(x[j]), rows + first[rj[j]] * row_words(P), e);
            d[j] = e[0];
        }
    }
}

// Appends word(e) for every set bit e < E of the lanes' masks (c bits in the
// warp) to a queue of cap entries; when they do not fit, voids the entries they
// got and returns false.
template <int E, typename F>
__device__ __forceinline__ bool push_pairs(unsigned m, int c, int *count, uint32_t *queue, int cap, F word)
{
    const int lane = threadIdx.x & 31, own = __popc(m);
    int o = 0;
    if (lane == 0) o = atomicAdd(count, c);
    o = __shfl_sync(0xffffffffu, o, 0);
    const bool fits = o + c <= cap;
    int incl = own;
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, s);
        if (lane >= s) incl += v;
    }
    int e = o + incl - own;
    for (; m; m &= m - 1, ++e)
        if (e < cap) queue[e] = fits ? word(__ffs(m) - 1) : ~0u;
    return fits;
}

// The same for double data: the samples less off, rounded to float.
template <int ST, int P>
__device__ __forceinline__ void load_samples(const double *__restrict__ X, int64_t ld, int64_t n, int D, bool vec,
                                             int64_t s0, uint64_t (&x)[ST][P], const double *__restrict__ off)
{
    const bool full = vec && s0 + ST <= n;
#pragma unroll
    for (int p = 0; p < P; ++p) {
        float v[2][ST];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int a = 2 * p + h;
#pragma unroll
            for (int j = 0; j < ST; ++j) v[h][j] = 0.f;
            if (a < D) {
                const double *row = X + (size_t)a * ld, c = __ldg(off + a);
                double w[ST];
                if (full && ST % 2 == 0) {
#pragma unroll
                    for (int j = 0; j + 1 < ST; j += 2) {
                        const double2 q = __ldg(reinterpret_cast<const double2 *>(row + s0 + j));
                        w[j] = q.x;
                        w[j + 1] = q.y;
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < ST; ++j) w[j] = __ldg(row + (s0 + j < n ? s0 + j : n - 1));
                }
#pragma unroll
                for (int j = 0; j < ST; ++j) v[h][j] = __double2float_rn(w[j] - c);
            }
        }
#pragma unroll
        for (int j = 0; j < ST; ++j) x[j][p] = pk(v[0][j], v[1][j]);
    }
}

// F64: double data, boxes rounded inwards after the offset, so that the float
// values bound the exact ones (kc_exact.cu).  TM: a screen that fills A.tmax.
template <int P, int ST, int NT, bool F64, bool TM>
__global__ void __launch_bounds__(NT, 1)
prune_max_kernel(const PruneArgs A)
{
    constexpr int T = NT * ST, NWP = NT / 32, RW = row_words(P), CAP = pair_cap(P);
    constexpr bool PT = TM && !F64;   // float screens are of center sets
    constexpr unsigned ALL = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char smem[];
    const int K = A.K, D = A.D, KP = K * P, KR = K * RW;
    const int b0 = blockIdx.y * A.per, nb = min(A.per, A.B - b0);
    const int ng = (nb + kPG - 1) / kPG, ns = (ng + kPSG - 1) / kPSG;
    const PruneLayout L(nb, K, P, T, NWP, TM);
    ulonglong2 *box = reinterpret_cast<ulonglong2 *>(smem + L.box), *gbox = reinterpret_cast<ulonglong2 *>(smem + L.gbox);
    ulonglong2 *sbox = reinterpret_cast<ulonglong2 *>(smem + L.sbox);
    uint64_t *ref = reinterpret_cast<uint64_t *>(smem + L.ref), *stage = reinterpret_cast<uint64_t *>(smem + L.stage);
    volatile unsigned long long *key = reinterpret_cast<unsigned long long *>(smem + L.key);
    unsigned long long *cand = reinterpret_cast<unsigned long long *>(smem + L.cand);
    volatile float *thr = reinterpret_cast<float *>(smem + L.thr);
    float *gmin = reinterpret_cast<float *>(smem + L.gmin), *smin = reinterpret_cast<float *>(smem + L.smin);
    int *hist = reinterpret_cast<int *>(smem + L.hist), *base = hist + kMaxK, *qn = hist + 2 * kMaxK;   // lengths of queue, qb, qc
    uint32_t *spos = reinterpret_cast<uint32_t *>(smem + L.pos), *queue = reinterpret_cast<uint32_t *>(smem + L.queue);
    uint32_t *qb = queue + ((NWP * ng + 3) & ~3), *qc = qb + CAP;
    uint8_t *fk = smem + L.fk, *fg = smem + L.fg, *fs = smem + L.fs, *rr = smem + L.rr;
    using T_ = typename std::conditional<F64, double, float>::type;
    const T_ *lo = static_cast<const T_ *>(A.lo) + (size_t)b0 * K * D;
    const T_ *hi = static_cast<const T_ *>(A.hi) + (size_t)b0 * K * D;
    const T_ *X = static_cast<const T_ *>(A.X);
    auto load = [&](int64_t s0, uint64_t (&x)[ST][P]) {
        if constexpr (F64) load_samples<ST, P>(X, A.ld, A.n, D, A.vec != 0, s0, x, A.off);
        else load_samples<ST, P>(X, A.ld, A.n, D, A.vec != 0, s0, x);
    };
    auto floor_of = [&](float v) {   // values below it can be dismissed
        if constexpr (TM)
            return v >= A.cut && A.cut < __int_as_float(0x7f800000) ? __int_as_float(0x7f800000) : screen_floor(v, A.c1, A.eps);
        else return v;
    };
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float INF = __int_as_float(0x7f800000);

    // ---- the nodes of this CTA's range: boxes, group boxes, references
#pragma unroll 4
    for (int i = tid; i < nb * KP; i += NT) {
        const int p = i % P, bk = i / P, a = 2 * p;
        const size_t o = (size_t)bk * D + a;
        const bool two = a + 1 < D;
        if constexpr (F64) {
            auto in = [&](int e, float &l, float &h) {
                const double c = A.off[a + e];
                l = __double2float_ru(__dsub_ru(lo[o + e], c));
                h = __double2float_rd(__dsub_rd(hi[o + e], c));
            };
            float l0 = 0.f, h0 = 0.f, l1 = 0.f, h1 = 0.f;
            if (a < D) in(0, l0, h0);
            if (two) in(1, l1, h1);
            box[bk * RW + p] = make_ulonglong2(pk(l0, l1), pk(h0, h1));
        } else {
            box[bk * RW + p] = a < D ? make_ulonglong2(pk(lo[o], two ? lo[o + 1] : 0.f), pk(hi[o], two ? hi[o + 1] : 0.f))
                                     : make_ulonglong2(0ull, 0ull);
        }
    }
    unsigned *tmx = reinterpret_cast<unsigned *>(smem + L.tmx);
    if constexpr (TM)
        for (int i = tid; i < nb; i += NT) tmx[i] = 0u;
    if (tid < 32) cand[tid] = 0ull;
    __syncthreads();
    auto meet = [&](const ulonglong2 *src, int cnt, ulonglong2 *dst, int e) {
        // [max lo, min hi] of cnt nodes' boxes (pair e % P of cluster e / P)
        const int i = e / P * RW + e % P;
        float2 l = make_float2(-INF, -INF), h = make_float2(INF, INF);
        for (int q = 0; q < cnt; ++q) {
            const ulonglong2 v = src[(size_t)q * KR + i];
            const float2 a = upk(v.x), b = upk(v.y);
            l = make_float2(fmaxf(l.x, a.x), fmaxf(l.y, a.y));
            h = make_float2(fminf(h.x, b.x), fminf(h.y, b.y));
        }
        dst[i] = make_ulonglong2(pk(l.x, l.y), pk(h.x, h.y));
    };
    for (int i = tid; i < ng * KP; i += NT) {
        const int g = i / KP;
        meet(box + (size_t)g * kPG * KR, min(kPG, nb - g * kPG), gbox + (size_t)g * KR, i % KP);
    }
    for (int i = tid; i < KP; i += NT) {
        const ulonglong2 v = box[(size_t)(nb / 2) * KR + i / P * RW + i % P];
        const float2 a = upk(v.x), b = upk(v.y);
        ref[i] = pk(0.5f * a.x + 0.5f * b.x, 0.5f * a.y + 0.5f * b.y);
    }
    __syncthreads();
    for (int i = tid; i < ns * KP; i += NT) {
        const int g = i / KP;
        meet(gbox + (size_t)g * kPSG * KR, min(kPSG, ng - g * kPSG), sbox + (size_t)g * KR, i % KP);
    }
    auto first_of = [&](const ulonglong2 *bx, int r) {
        uint64_t x[1][P];
#pragma unroll
        for (int p = 0; p < P; ++p) x[0][p] = ref[r * P + p];
        float best = INF;
        int kb = 0;
#pragma unroll 2
        for (int k = 0; k < K; ++k) {
            float d[1];
            box_dists<1, P>(x, bx + k * RW, d);
            if (d[0] < best) { best = d[0]; kb = k; }
        }
        return (uint8_t)kb;
    };
    for (int i = tid; i < nb * K; i += NT) fk[i] = first_of(box + (size_t)(i / K) * KR, i % K);
    for (int i = tid; i < ng * K; i += NT) fg[i] = first_of(gbox + (size_t)(i / K) * KR, i % K);
    __syncthreads();
    for (int i = tid; i < ns * K; i += NT) fs[i] = first_of(sbox + (size_t)(i / K) * KR, i % K);

    uint32_t first = 0u;   // the tile's first position
    // What a sample of this tile has to reach where the best key is m.  An equal value
    // wins only at a smaller position: where m's lies before the tile, the next
    // float above is wanted.  (Nodes of bound 0, and values that many samples attain:
    // every sample passed every test.)
    auto thr_of = [&](unsigned long long m) {
        const float v = floor_of(key_val(m));
        if constexpr (!TM)
            if (!A.ids && m != 0ull && key_pos(m) <= first && v < __int_as_float(0x7f800000))
                return __uint_as_float(__float_as_uint(v) + 1u);
        return v;
    };

    // raise node b's best value by a warp whose lanes hold keys (0: none)
    auto raise = [&](int b, unsigned long long k) {
        k = warp_max_u64(k);
        if (TM && lane == 0) atomicMax(&tmx[b], (unsigned)(k >> 32));
        if (lane == 0 && k > key[b]) {
            atomicMax(const_cast<unsigned long long *>(&key[b]), k);
            atomicMax(reinterpret_cast<int *>(const_cast<float *>(&thr[b])), __float_as_int(thr_of(k)));
        }
        __syncwarp();
    };

    auto coord = [&](int a, int64_t s) {
        const T_ v = X[(size_t)a * A.ld + s];
        if constexpr (F64) return __double2float_rn(v - A.off[a]);
        else return v;
    };
    // the same for one lane's value
    auto lift = [&](int b, float v, uint32_t pos) {
        const unsigned long long k = key_max(v, pos);
        if (!(v >= thr[b])) return;
        if (TM) atomicMax(&tmx[b], __float_as_uint(v));
        if (k > key[b]) {
            atomicMax(const_cast<unsigned long long *>(&key[b]), k);
            atomicMax(reinterpret_cast<int *>(const_cast<float *>(&thr[b])), __float_as_int(thr_of(k)));
        }
    };
    // node b, all its clusters, over a strip's samples y (its slots from q0)
    auto finish = [&](const uint64_t (&y)[ST][P], int q0, int b) {
        float v[ST];
        box_dists<ST, P, PT>(y, box + b * KR, v);
        for (int k = 1; k < K; ++k) {
            float e[ST];
            box_dists<ST, P, PT>(y, box + b * KR + k * RW, e);
#pragma unroll
            for (int j = 0; j < ST; ++j) v[j] = fminf(v[j], e[j]);
        }
        if (!__any_sync(ALL, max_of<ST>(v) >= thr[b])) return;
        if constexpr (TM) {   // (the position of a screen's key is not used)
            raise(b, ((unsigned long long)__reduce_max_sync(ALL, __float_as_uint(max_of<ST>(v))) << 32) | 1ull);
        } else {
            const unsigned long long cur = key[b];
            unsigned long long top = 0ull;
#pragma unroll
            for (int j = 0; j < ST; ++j) {
                const unsigned long long q = key_max(v[j], spos[q0 + j * 32 + lane]);
                top = q > top ? q : top;
            }
            if (__any_sync(ALL, top > cur)) raise(b, top > cur ? top : 0ull);
        }
    };

    const int64_t tiles = (A.n + T - 1) / T;
    const int w0 = warp * 32 * ST;   // the warp's slots of the sorted tile
    uint64_t x[ST][P];
    load((int64_t)blockIdx.x * T + (int64_t)tid * ST, x);
    bool seed = true;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int64_t s0 = tile * T + (int64_t)tid * ST;
        first = (uint32_t)(tile * T);
        if (tid < kMaxK) hist[tid] = 0;
        if (tid >= kMaxK && tid < kMaxK + 3) qn[tid - kMaxK] = 0;
        // nearest reference of each sample, and the sample farthest from its reference
        int r[ST];
        {
            float u[ST];
#pragma unroll
            for (int j = 0; j < ST; ++j) { u[j] = INF; r[j] = 0; }
            for (int k = 0; k < K; ++k) {
                uint64_t acc[ST];
#pragma unroll
                for (int j = 0; j < ST; ++j) acc[j] = 0;
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    const uint64_t c = ref[k * P + p];
#pragma unroll
                    for (int j = 0; j < ST; ++j) {
                        const uint64_t t = sub2(x[j][p], c);
                        acc[j] = fma2(t, t, acc[j]);
                    }
                }
#pragma unroll
                for (int j = 0; j < ST; ++j) {
                    const float2 s = upk(acc[j]);
                    if (s.x + s.y < u[j]) { u[j] = s.x + s.y; r[j] = k; }
                }
            }
            if (seed) {
                unsigned long long m = 0ull;
#pragma unroll
                for (int j = 0; j < ST; ++j) {
                    const uint32_t pos = (uint32_t)(s0 + j < A.n ? s0 + j : A.n - 1);
                    const unsigned long long c = ((unsigned long long)__float_as_uint(u[j]) << 32) | pos;
                    m = c > m ? c : m;
                }
                if (m > cand[lane]) atomicMax(&cand[lane], m);
            }
        }
        __syncthreads();   // hist is zero; the previous tile's readers are done
        // best values so far, from every CTA
        for (int b = tid; b < nb; b += NT) {
            const unsigned long long g = peek(&A.keys[b0 + b]);
            unsigned long long m = seed ? 0ull : key[b];
            m = g > m ? g : m;
            key[b] = m;
            thr[b] = thr_of(m);
        }
        // slots of the samples, sorted by reference
        int off[ST];
#pragma unroll
        for (int j = 0; j < ST; ++j) {
            const unsigned grp = __match_any_sync(ALL, r[j]);
            const int leader = __ffs(grp) - 1;
            int o = 0;
            if (lane == leader) o = atomicAdd(&hist[r[j]], __popc(grp));
            off[j] = __shfl_sync(ALL, o, leader) + __popc(grp & ((1u << lane) - 1u));
        }
        __syncthreads();
        if (tid < K) {
            int s = 0;
            for (int k = 0; k < tid; ++k) s += hist[k];
            base[tid] = s;
        }
        if (seed) {
            // the first tile's farthest samples, against every node (and its first
            // sample: where no value is larger, none of the tile can win a tie)
            const int64_t cp = lane == 0 ? tile * T : (int64_t)(uint32_t)cand[lane];
            const uint32_t cid = A.ids ? A.ids[cp] : (uint32_t)cp;
            uint64_t xc[1][P];
#pragma unroll
            for (int p = 0; p < P; ++p)
                xc[0][p] = pk(2 * p < D ? coord(2 * p, cp) : 0.f, 2 * p + 1 < D ? coord(2 * p + 1, cp) : 0.f);
            for (int b = warp; b < nb; b += NWP) {
                float best = INF;
                for (int k = 0; k < K; ++k) {
                    float d[1];
                    box_dists<1, P, PT>(xc, box + ((size_t)b * K + k) * RW, d);
                    best = fminf(best, d[0]);
                }
                raise(b, key_max(best, cid));
            }
            seed = false;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < ST; ++j) {
            const int o = off[j] + base[r[j]];
            const int64_t w = s0 + j < A.n ? s0 + j : A.n - 1;
            spos[o] = A.ids ? A.ids[w] : (uint32_t)w;
            rr[o] = (uint8_t)r[j];
#pragma unroll
            for (int p = 0; p < P; ++p) stage[(size_t)p * T + o] = x[j][p];
        }
        for (int g = tid; g < ng; g += NT) {
            float m = INF;
            for (int b = g * kPG; b < min(nb, (g + 1) * kPG); ++b) m = fminf(m, thr[b]);
            gmin[g] = m;
        }
        __syncthreads();
        for (int s = tid; s < ns; s += NT) {
            float m = INF;
            for (int g = s * kPSG; g < min(ng, (s + 1) * kPSG); ++g) m = fminf(m, gmin[g]);
            smin[s] = m;
        }
#pragma unroll
        for (int p = 0; p < P; ++p)
#pragma unroll
            for (int j = 0; j < ST; ++j) x[j][p] = stage[(size_t)p * T + w0 + j * 32 + lane];
        __syncthreads();
        {
            // group tests of the warp's strip (32 ST slots): many survivors
            // make an item, few are packed as pairs
            uint8_t rj[ST];
            const bool one = strip_refs(rr + w0, lane, rj);
            for (int s = 0; s < ns; ++s) {
                float d[ST];
                strip_dists<ST, P>(x, sbox + s * KR, fs + s * K, rj, one, d);
                if (!__any_sync(ALL, max_of<ST>(d) >= smin[s])) continue;
                const int g1 = min(ng, (s + 1) * kPSG);
                for (int g = s * kPSG; g < g1; ++g) {
                    strip_dists<ST, P>(x, gbox + g * KR, fg + g * K, rj, one, d);
                    const float t = gmin[g];
                    unsigned m = 0u;
#pragma unroll
                    for (int j = 0; j < ST; ++j) m |= d[j] >= t ? 1u << j : 0u;
                    if (!__any_sync(ALL, m != 0u)) continue;
                    const int c = (int)__reduce_add_sync(ALL, (unsigned)__popc(m));
                    const uint32_t gw = (uint32_t)g << 16;
                    if (c > kSparse * ST || !push_pairs<ST>(m, c, &qn[1], qb, CAP, [&](int j) {
                            return gw | (uint32_t)(w0 + j * 32 + lane);
                        }))
                        if (lane == 0) queue[atomicAdd(&qn[0], 1)] = gw | (uint32_t)warp;
                }
            }
        }
        // the next tile's samples, in flight while the queue is worked off
        constexpr bool AHEAD = P < 48;   // (where the registers hold both)
        const bool more = tile + gridDim.x < tiles;
        if (AHEAD && more) load(s0 + (int64_t)gridDim.x * T, x);
        __syncthreads();
        // Where the group tests dismiss little (boxes that differ in every cluster: all
        // items), tests cost more than they save at few attributes; the streaming kernel
        // takes this CTA's samples.  (Inputs are one or the other: 0 to 5 % of the
        // items on nested boxes, all of them on open nodes of a branch and bound.)
        if (!TM && P <= 4 && A.left && tile == blockIdx.x && 2 * qn[0] > NWP * ng) {
            if (tid == 0) A.left[blockIdx.x] = A.left[gridDim.x] = 1;
            return;
        }
        const int items = qn[0], pairs = min(qn[1], CAP), units = items + (pairs + 31) / 32;
        // (strip, group) items: the node tests
        auto take_item = [&](int it) {
            const uint32_t w = queue[it];
            const int g = (int)(w >> 16), q0 = (int)(w & 0xFFFFu) * 32 * ST, bg = g * kPG, nn = min(kPG, nb - bg);
            uint64_t y[ST][P];
#pragma unroll
            for (int p = 0; p < P; ++p)
#pragma unroll
                for (int j = 0; j < ST; ++j) y[j][p] = stage[(size_t)p * T + q0 + j * 32 + lane];
            uint8_t rj[ST];
            const bool one = strip_refs(rr + q0, lane, rj);
            unsigned m = 0u;   // bit i ST + j: sample j may matter in node bg + i
#pragma unroll(P <= 4 ? 2 : 1)
            for (int i = 0; i < nn; ++i) {
                float d[ST];
                strip_dists<ST, P, PT>(y, box + (bg + i) * KR, fk + (bg + i) * K, rj, one, d);
                const float t = thr[bg + i];
                unsigned mi = 0u;
#pragma unroll
                for (int j = 0; j < ST; ++j) mi |= d[j] >= t ? 1u << j : 0u;
                m |= mi << (i * ST);
            }
            const int c = (int)__reduce_add_sync(ALL, (unsigned)__popc(m));
            if (c == 0) return;
            if (c <= CAP / 8 && push_pairs<ST * kPG>(m, c, &qn[2], qc, CAP, [&](int e) {
                    return ((uint32_t)(bg + e / ST) << 16) | (uint32_t)(q0 + (e % ST) * 32 + lane);
                }))
                return;
            // many: every cluster of the nodes that have any
            for (int i = 0; i < nn; ++i) {
                if (!__any_sync(ALL, (m >> (i * ST) & ((1u << ST) - 1u)) != 0u)) continue;
                finish(y, q0, bg + i);
            }
        };
        // (group, sample) pairs, one to a lane
        auto take_pairs = [&](int it) {
            const uint32_t w = it + lane < pairs ? qb[it + lane] : ~0u;
            const bool on = w != ~0u;
            const int bg = on ? (int)(w >> 16) * kPG : 0, slot = (int)(w & 0xFFFFu) & (T - 1);
            uint64_t y[1][P];
#pragma unroll
            for (int p = 0; p < P; ++p) y[0][p] = stage[(size_t)p * T + slot];
            const int rs = rr[slot];
            unsigned m = 0u;
            for (int i = 0; i < kPG; ++i) {
                const int b = min(bg + i, nb - 1);
                float d[1];
                box_dists<1, P, PT>(y, box + b * KR + fk[b * K + rs] * RW, d);
                if (on && bg + i < nb && d[0] >= thr[b]) m |= 1u << i;
            }
            const int c = (int)__reduce_add_sync(ALL, (unsigned)__popc(m));
            if (c == 0 || push_pairs<kPG>(m, c, &qn[2], qc, CAP,
                                          [&](int e) { return ((uint32_t)(bg + e) << 16) | (uint32_t)slot; }))
                return;
            for (; m; m &= m - 1) {
                const int b = bg + __ffs(m) - 1;
                float v = INF;
                for (int k = 0; k < K; ++k) {
                    float d[1];
                    box_dists<1, P, PT>(y, box + b * KR + k * RW, d);
                    v = fminf(v, d[0]);
                }
                lift(b, v, spos[slot]);
            }
        };
        // The warps take units in turn until none is left or the queue of (node, sample)
        // pairs fills up, work that queue off one pair to a lane, and go on.  (Pairs that did
        // not fit were evaluated in place by single lanes, where many samples survive
        // the group tests.)
        for (int u = warp;;) {
            for (; u < units && (u < items || *const_cast<volatile int *>(&qn[2]) < CAP / 2); u += NWP) {
                if (u < items) take_item(u);
                else take_pairs((u - items) * 32);
            }
            const bool done = __syncthreads_and(u >= units) != 0;
            const int last = min(qn[2], CAP);
            // (node, sample) pairs: the minimum over the clusters
            for (int it = tid; it < last; it += NT) {
                const uint32_t w = qc[it];
                if (w == ~0u) continue;
                const int b = (int)(w >> 16), slot = (int)(w & 0xFFFFu);
                uint64_t y[1][P];
#pragma unroll
                for (int p = 0; p < P; ++p) y[0][p] = stage[(size_t)p * T + slot];
                float v = INF;
                for (int k = 0; k < K; ++k) {
                    float d[1];
                    box_dists<1, P, PT>(y, box + b * KR + k * RW, d);
                    v = fminf(v, d[0]);
                }
                lift(b, v, spos[slot]);
            }
            if (done) break;
            __syncthreads();
            if (tid == 0) qn[2] = 0;
            __syncthreads();
        }
        if (!AHEAD && more) load(s0 + (int64_t)gridDim.x * T, x);
        __syncthreads();
        // publish what this tile raised
        for (int b = tid; b < nb; b += NT) {
            const unsigned long long k = key[b];
            if (k > peek(&A.keys[b0 + b])) atomicMax(&A.keys[b0 + b], k);
            if constexpr (TM) {
                A.tmax[(size_t)(b0 + b) * A.rows + tile] = __uint_as_float(tmx[b]);
                tmx[b] = 0u;
            }
        }
    }
}

// Attribute pairs with a compiled kernel (other D take the next larger one:
// padding pairs add exactly zero) and their launch.
struct PruneEntry {
    int P, ST, T, NT;
    void (*fn)(const PruneArgs);
};
template <int P, bool F64, bool TM, int ST = PruneShape<P>::ST>
PruneEntry prune_entry()
{
    constexpr int NT = PruneShape<P>::NT;
    return PruneEntry{P, ST, NT * ST, NT, prune_max_kernel<P, ST, NT, F64, TM>};
}
// Table of the kernels in ascending P, two entries (4 and 2 samples a thread)
// for each P <= 4.
template <bool F64, bool TM>
const PruneEntry *prune_table()
{
    static const PruneEntry t[] = {
        prune_entry<1, F64, TM>(),  prune_entry<1, F64, TM, 2>(), prune_entry<2, F64, TM>(), prune_entry<2, F64, TM, 2>(),
        prune_entry<3, F64, TM>(),  prune_entry<3, F64, TM, 2>(), prune_entry<4, F64, TM>(), prune_entry<4, F64, TM, 2>(),
        prune_entry<6, F64, TM>(),  prune_entry<8, F64, TM>(),    prune_entry<12, F64, TM>(), prune_entry<16, F64, TM>(),
        prune_entry<24, F64, TM>(), prune_entry<34, F64, TM>(),   prune_entry<48, F64, TM>(), prune_entry<64, F64, TM>()};
    return t;
}
// The entry for D attributes and n samples (st: 4 or 2 samples a thread where
// both exist, 0: by size -- 2 where the tiles of 4 would not fill 8 rounds).
inline const PruneEntry *prune_pick(const PruneEntry *e, int D, int64_t n, int sms, int st)
{
    const int P = (D + 1) / 2;
    while (e->P < P) ++e;
    if (P <= 4 && (st == 2 || (st != 4 && (n + e->T - 1) / e->T < 8 * (int64_t)sms))) ++e;
    return e;
}
// chunk: nodes per CTA at most (0: as many as fit).  A.B = all nodes.
cudaError_t prune_run(const PruneEntry *e, PruneArgs A, bool tm, int sms, size_t smem_cap, int chunk, cudaStream_t stream);

// The streaming path for few nodes (kc_stream.cu): taken at up to
// kStreamTerms node x cluster x attribute terms for D <= 8, and at up to two
// nodes and kStreamCols node x cluster columns for wider data.  Streaming
// against pruning, us, at 320 MB of samples: D = 8, K = 5, 4 nodes 216 / 283, 8
// nodes 427 / 386; D = 4, K = 3, 8 nodes 265 / 384, 16 nodes 508 / 515, 32 nodes
// 1086 / 760; D = 2, K = 4 (160 MB), 16 nodes 363 / 508, 32 nodes 808 / 678.
// With n <= kStreamSmall terms in all it is taken for any batch at D <= 8: the chip is
// not filled long enough for the sort to pay (1e5 samples, D = 4, K = 3, 64 nodes: 22 us
// against 49 without structure, 20 with nested boxes; 3e8 terms, 256 nodes: 65 against
// 117 and 39).
constexpr int kStreamTerms = 208, kStreamCols = 16;
constexpr double kStreamSmall = 1e8;
inline bool use_stream_f32(int B, int K, int D, int64_t n)
{
    return (D <= 8 && ((int64_t)B * K * D <= kStreamTerms || ((double)n * B * K * D <= kStreamSmall && B < 65536))) ||
           (B <= 2 && B * K <= kStreamCols);
}
// Batches whose unstructured form the pruning kernel leaves to the streaming one
// (PruneArgs::left): at few attributes full evaluation is cheaper than tests that
// dismiss nothing (open nodes of a branch and bound over 1e6 samples, pruned / full /
// pruned until the first group tests and then full, us: D = 2, K = 3, 64 nodes 224 /
// 98 / 115; D = 4 220 / 140 / 152); at D = 5 to 8 up to 32 nodes (D = 8, K = 5, 16
// nodes 120 / 93 / 107; 64 nodes 244 / 333) or where a CTA has one tile (1e5 samples,
// 64 nodes 72 / 48).
inline bool may_leave(int B, int D, bool one_tile)
{
    return B > 2 && B < 65536 && (D <= 4 || (D <= 8 && (B <= 32 || one_tile)));
}
cudaError_t launch_stream_f32(PruneArgs A, int sms, cudaStream_t stream);
// The same over the samples A.ids[0 .. A.n) of the rows A.X (D <= 8).
cudaError_t launch_stream_gather_f32(PruneArgs A, int sms, cudaStream_t stream);
constexpr int kStreamTile = 128;   // samples of a tmax row of the streaming screen

}  // namespace kc
