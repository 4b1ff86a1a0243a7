// resample.cu -- cell-centred trilinear resampling of mean fields onto the
// surrogate's grid (App. B: the simulated fields are scaled down to
// 128x64x64 before training).
//
// Output cell o of an axis with n source and m target cells samples the
// source at s = (o + 1/2) n/m - 1/2, clamped to [0, n - 1], linearly between
// floor(s) and floor(s) + 1; the 3D map is the product of the three axes.
// One thread per output cell and group of channels: the eight source cells and
// their weights are found once for the group, and four interleaved channels are
// one 16-byte load (one thread per value recomputed the map per channel and read
// every source sector four times: 192x128x96 -> 128x64x64 took 27.1 us, now
// 12.3).  Small targets split their channels over more threads, and blocks take
// the shape of narrow targets (one thread for all of 256 channels on 4x4x4: 28.7
// us, one per value 4.6, now 4.3; 2x2x20000, 4 channels: 34.8, 8.2, now 4.9).
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
// dst: [C][mz][my][mx].  READ: ONE value at a time; FOUR, the four channels of
// layout 0 in 16 bytes; FOURS, the same for any multiple of 4 channels.  SPLIT:
// a thread takes `cpt` of the channels (whole fours), the groups behind each
// other along grid z, `ztiles` apart; else all of them.
enum { ONE, FOUR, FOURS };

template <int READ, bool SPLIT>
__global__ void __launch_bounds__(256) k_resample(const float *__restrict__ src, int nx, int ny, int nz, int C,
                                                  int layout, float *__restrict__ dst, int mx, int my, int mz, int cpt,
                                                  unsigned ztiles, unsigned ztotal)
{
    const int ox = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if (ox >= mx) return;
    const int64_t nxyz = (int64_t)nx * ny * nz, plane = (int64_t)mx * my * mz;
    const Axis ax = axis_map(ox, nx, mx);
    const float wx[2] = {1.f - ax.t, ax.t};
    const int xs[2] = {ax.i0, ax.i1};
    for (int oy = (int)(blockIdx.y * blockDim.y + threadIdx.y); oy < my; oy += (int)(gridDim.y * blockDim.y))
    for (unsigned zt = blockIdx.z; zt < ztotal; zt += gridDim.z) {
        const unsigned group = SPLIT ? zt / ztiles : 0u;
        const int c0 = SPLIT ? (int)group * cpt : 0, c1 = SPLIT ? min(C, c0 + cpt) : C;
        const int oz = (int)((zt - group * ztiles) * blockDim.z + threadIdx.z);
        if (oz >= mz) continue;
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
        if (READ == ONE) {
            for (int c = c0; c < c1; ++c) {
                float acc = 0.f;
#pragma unroll
                for (int q = 0; q < 8; ++q) acc += w[q] * (layout == 0 ? src[cell[q] * C + c] : src[c * nxyz + cell[q]]);
                d[c * plane] = acc;
            }
        } else {
            for (int c = c0; c < (READ == FOUR ? 4 : c1); c += 4) {
                float4 v[8];
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    v[q] = *reinterpret_cast<const float4 *>(src + cell[q] * (READ == FOUR ? 4 : C) + c);
                float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    acc[0] += w[q] * v[q].x;
                    acc[1] += w[q] * v[q].y;
                    acc[2] += w[q] * v[q].z;
                    acc[3] += w[q] * v[q].w;
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) d[(c + e) * plane] = acc[e];
            }
        }
    }
}

// smallest power of two that holds v, at most `most` (a power of two)
unsigned pow2_for(int v, unsigned most)
{
    unsigned p = 1;
    while (p < most && p < (unsigned)v) p <<= 1;
    return p;
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
    // rows of up to 32 cells per block, then rows, then planes
    const unsigned bx = pow2_for(mx, 32), by = pow2_for(my, 256 / bx), bz = pow2_for(mz, std::min(64u, 256 / (bx * by)));
    const bool fours = src_layout == 0 && channels % 4 == 0 && ((uintptr_t)src & 15) == 0;
    // groups of channels: where the cells alone are less than a quarter of the
    // threads that the chip holds, enough for that many (and grid z stays a
    // 32-bit count)
    const int64_t cells = (int64_t)mx * my * mz, steps = fours ? channels / 4 : channels;
    const int64_t ztiles = ((int64_t)mz + bz - 1) / bz;
    const int64_t most = std::min<int64_t>(gb300::sm_count() * 512 / cells, ((int64_t)1 << 31) / ztiles);
    const int64_t per = (steps + std::max<int64_t>(1, std::min(steps, most)) - 1) / std::max<int64_t>(1, std::min(steps, most));
    const int64_t groups = (steps + per - 1) / per, ztotal = ztiles * groups;
    const dim3 blk(bx, by, bz), grd((unsigned)(((int64_t)mx + bx - 1) / bx), (unsigned)std::min<int64_t>(((int64_t)my + by - 1) / by, 65535),
                                    (unsigned)std::min<int64_t>(ztotal, 65535));
    auto k = groups > 1 ? (fours ? k_resample<FOURS, true> : k_resample<ONE, true>)
                        : !fours ? k_resample<ONE, false> : channels == 4 ? k_resample<FOUR, false> : k_resample<FOURS, false>;
    k<<<grd, blk, 0, static_cast<cudaStream_t>(cuda_stream)>>>(src, nx, ny, nz, channels, src_layout, dst, mx, my, mz,
                                                              (int)(fours ? 4 * per : per), (unsigned)ztiles, (unsigned)ztotal);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        lbm::set_global_error(std::string("lbm_resample: ") + cudaGetErrorString(e));
        return LBM_ERR_CUDA;
    }
    return LBM_OK;
}
