// Reordering of per-cell device arrays into the caller's order, so that a
// read of the state is a device gather and plain copies (no per-cell host
// work).  The results are written in order, so that dst may be page-locked
// host memory: whole lines cross the link, and a small read needs no copy.
#include <cstdint>

#include <cuda_runtime.h>

#include "sweep.cuh"

namespace rich {
namespace {

// dst[f * n + u] = src_f[cell[u]] for the fields f < 6 (null sources are
// skipped): cell[u] is the internal cell of the caller's index u
__global__ void k_unpermute(int32_t n, const int32_t *__restrict__ cell, const double *s0, const double *s1,
                            const double *s2, const double *s3, const double *s4, const double *s5, double *dst)
{
    const int32_t u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= n) return;
    const int32_t k = cell[u];
    const double *src[6] = {s0, s1, s2, s3, s4, s5};
#pragma unroll
    for (int f = 0; f < 6; f++)
        if (src[f]) dst[(int64_t)f * n + u] = src[f][k];
}

// Seven fields of every cell for rich_get_state, in the caller's order: the
// points, the primitives (rho, vx, vy, p side by side per cell, in the
// simulation's precision) and the area
template <class R>
__global__ void k_unpermute_state(int32_t n, const int32_t *__restrict__ cell, const double *__restrict__ x,
                                  const double *__restrict__ y, const Vec4<R> *__restrict__ W,
                                  const double *__restrict__ area, double *__restrict__ dst)
{
    const int32_t u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= n) return;
    const int32_t k = cell[u];
    const int64_t N = n;
    const Vec4<R> w = W[k];
    dst[u] = x[k];
    dst[N + u] = y[k];
    dst[2 * N + u] = (double)w.x;
    dst[3 * N + u] = (double)w.y;
    dst[4 * N + u] = (double)w.z;
    dst[5 * N + u] = (double)w.w;
    dst[6 * N + u] = area[k];
}

}  // namespace

cudaError_t launch_unpermute_state(int32_t n, const int32_t *cell, const double *x, const double *y, const void *W,
                                   bool single, const double *area, double *dst, cudaStream_t st)
{
    const int b = (n + 255) / 256;
    if (n > 0 && single)
        k_unpermute_state<float><<<b, 256, 0, st>>>(n, cell, x, y, static_cast<const Vec4<float> *>(W), area, dst);
    else if (n > 0)
        k_unpermute_state<double><<<b, 256, 0, st>>>(n, cell, x, y, static_cast<const Vec4<double> *>(W), area, dst);
    return cudaGetLastError();
}

cudaError_t launch_unpermute(int32_t n, const int32_t *cell, const double *const src[6], double *dst,
                             cudaStream_t st)
{
    if (n > 0)
        k_unpermute<<<(n + 255) / 256, 256, 0, st>>>(n, cell, src[0], src[1], src[2], src[3], src[4], src[5], dst);
    return cudaGetLastError();
}

}  // namespace rich
