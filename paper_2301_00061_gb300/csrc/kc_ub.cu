// kc_ub.cu -- objective of Eq. 1 at center sets on samples: the upper bound
// alpha(M) of Eq. 12, the farthest-point queries of Algorithm 2, and the final
// double-precision certificate.  A center set is a node whose boxes are points;
// its exact maximum comes from kc_exact.cu.
#include <cuda_runtime.h>

#include "kc_device.cuh"
#include "kc_internal.cuh"

namespace kc {

namespace {

// Coordinates of the centers named by `centers` [count] -> out [count][D].
template <typename T>
__global__ void gather_centers_kernel(const T *__restrict__ X, int64_t ld, int D, const int64_t *__restrict__ centers,
                                      int64_t count, T *__restrict__ out)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count * D; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = X[(size_t)(i % D) * ld + centers[i / D]];
}

}  // namespace

kc_status launch_objective(kc_ctx *c, const View &v, const int64_t *centers, int S, int Kc,
                           double alpha_cut, double *val, int64_t *arg, const void *pts)
{
    if (S <= 0) return KC_OK;
    if (!pts) {
        const int64_t count = (int64_t)S * Kc;
        KC_TRY(ensure(c, c->obj, (size_t)count * c->D * c->esize));
        const int grid = (int)std::min<int64_t>((count * c->D + 255) / 256, (int64_t)c->num_sms * 8);
        if (c->dt == KC_F32)
            gather_centers_kernel<float><<<grid, 256, 0, c->stream>>>(static_cast<const float *>(c->X), c->ldx, c->D,
                                                                      centers, count, static_cast<float *>(c->obj.p));
        else
            gather_centers_kernel<double><<<grid, 256, 0, c->stream>>>(static_cast<const double *>(c->X), c->ldx, c->D,
                                                                       centers, count, static_cast<double *>(c->obj.p));
        KC_TRY(after_launch(c, "gather centers"));
        pts = c->obj.p;
    }
    // double data: every set's value, also those at or above alpha_cut
    const double cut = c->dt == KC_F32 ? alpha_cut : __builtin_huge_val();
    return launch_exact_max(c, v, pts, pts, S, Kc, cut, nullptr, val, arg);
}

}  // namespace kc
