// resample.cu -- cell-centred trilinear resampling of mean fields onto the
// surrogate's grid (App. B: the simulated fields are scaled down to
// 128x64x64 before training).
//
// Output cell o of an axis with n source and m target cells samples the
// source at s = (o + 1/2) n/m - 1/2, clamped to [0, n - 1], linearly between
// floor(s) and floor(s) + 1; the 3D map is the product of the three axes.
// One thread per output cell: the eight source cells and their weights are
// found once for all channels, and four interleaved channels are one 16-byte
// load (one thread per value recomputed the map per channel and read every
// source sector four times: 192x128x96 -> 128x64x64 took 27.1 us, now 12.3).
#include <algorithm>
#include <cstdint>
#include <string>

#include "../../include/lbm.h"
#include "sm_count.h"

namespace lbm {
void set_global_error(const std::string &m);   // lbm_api.cu
}

namespace {

struct Axis {
    int i0, i1;
    float t;
};

__device__ __forceinline__ Axis axis_map(int o, int n, int m)
{
    float s = ((float)o + 0.5f) * ((float)n / (float)m) - 0.5f;
    s = fminf(fmaxf(s, 0.f), (float)(n - 1));
    const int i0 = (int)floorf(s);
    return Axis{i0, min(i0 + 1, n - 1), s - (float)i0};
}

// src: [nz][ny][nx][C] (cell-major, layout 0) or [C][nz][ny][nx] (layout 1);
// dst: [C][mz][my][mx].  PACK: layout 0 with 4 channels on 16-byte boundaries.
template <bool PACK>
__global__ void __launch_bounds__(256) k_resample(const float *__restrict__ src, int nx, int ny, int nz, int C,
                                                  int layout, float *__restrict__ dst, int mx, int my, int mz)
{
    const int ox = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if (ox >= mx) return;
    const int64_t nxyz = (int64_t)nx * ny * nz, plane = (int64_t)mx * my * mz;
    const Axis ax = axis_map(ox, nx, mx);
    const float wx[2] = {1.f - ax.t, ax.t};
    const int xs[2] = {ax.i0, ax.i1};
    for (int oy = (int)(blockIdx.y * blockDim.y + threadIdx.y); oy < my; oy += (int)(gridDim.y * blockDim.y))
    for (int oz = (int)blockIdx.z; oz < mz; oz += (int)gridDim.z) {
        const Axis ay = axis_map(oy, ny, my), az = axis_map(oz, nz, mz);
        const float wy[2] = {1.f - ay.t, ay.t}, wz[2] = {1.f - az.t, az.t};
        const int ys[2] = {ay.i0, ay.i1}, zs[2] = {az.i0, az.i1};
        float *d = dst + (int64_t)ox + (int64_t)mx * (oy + (int64_t)my * oz);
        int64_t cell[8];
        float w[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int a = q >> 2, b = (q >> 1) & 1, e = q & 1;
            cell[q] = (int64_t)xs[e] + (int64_t)nx * ((int64_t)ys[b] + (int64_t)ny * zs[a]);
            w[q] = wz[a] * wy[b] * wx[e];
        }
        if (PACK) {
            float4 v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = reinterpret_cast<const float4 *>(src)[cell[q]];
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                acc[0] += w[q] * v[q].x;
                acc[1] += w[q] * v[q].y;
                acc[2] += w[q] * v[q].z;
                acc[3] += w[q] * v[q].w;
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) d[c * plane] = acc[c];
        } else {
            for (int c = 0; c < C; ++c) {
                float acc = 0.f;
#pragma unroll
                for (int q = 0; q < 8; ++q) acc += w[q] * (layout == 0 ? src[cell[q] * C + c] : src[c * nxyz + cell[q]]);
                d[c * plane] = acc;
            }
        }
    }
}

bool on_device(const void *p)
{
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

}  // namespace

extern "C" lbm_status lbm_resample(const float *src, int32_t nx, int32_t ny, int32_t nz, int32_t channels,
                                   int32_t src_layout, float *dst, int32_t mx, int32_t my, int32_t mz,
                                   void *cuda_stream)
{
    if (!src || !dst || nx < 1 || ny < 1 || nz < 1 || mx < 1 || my < 1 || mz < 1 || channels < 1 ||
        (src_layout != 0 && src_layout != 1)) {
        lbm::set_global_error("lbm_resample: null pointer, empty grid or unknown layout");
        return LBM_ERR_ARG;
    }
    if (!on_device(src) || !on_device(dst)) {
        lbm::set_global_error("lbm_resample: src and dst must be device (or managed) memory");
        return LBM_ERR_ARG;
    }
    const dim3 blk(32, 8), grd((unsigned)((mx + 31) / 32), (unsigned)std::min((my + 7) / 8, 65535), (unsigned)std::min(mz, 65535));
    auto k = src_layout == 0 && channels == 4 && ((uintptr_t)src & 15) == 0 ? k_resample<true> : k_resample<false>;
    k<<<grd, blk, 0, static_cast<cudaStream_t>(cuda_stream)>>>(src, nx, ny, nz, channels, src_layout, dst, mx, my, mz);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        lbm::set_global_error(std::string("lbm_resample: ") + cudaGetErrorString(e));
        return LBM_ERR_CUDA;
    }
    return LBM_OK;
}
