// ffno_fast.h -- the factorised surrogate's tiled kernels (ffno_fast.cu):
// one axis's spectral convolution in one pass, the pointwise networks and
// their backward, and the spectral weights' gradient.
#pragma once
#include <cstddef>
#include <cstdint>
#include <vector>

#include <cuda_runtime.h>

namespace ffno {

enum { ACT_NONE = 0, ACT_GELU = 1, ACT_SIREN = 2 };
constexpr int MAXW = 32;                 // channels the tiled kernels take

// One axis of the spectral convolution: L samples, the first m wave numbers.
// The transforms use the symmetries of the real DFT: samples n and L - n are
// folded into even and odd parts and, where 4 divides L, n and L/2 - n once
// more (q = 2 parities of the wave number), which leaves nq terms per sum.
struct Axis {
    int L, m;
    int rows;                            // 1: the samples are contiguous (x); 0: S apart
    int64_t S, outer;                    // lines: outer x S (rows: outer, S = 1)
    int reg;                             // 1: a register kernel exists for this length
    int T;                               // lines per block
    int q, nq;                           // parities, terms per folded sum
    int mk, KG, NG;                      // wave numbers per parity, groups of 4 of them, groups of 4 terms
    uint32_t dnq, dKG, dNG;              // reciprocals of nq, KG, NG
    int DS, KS;                          // shared-memory strides: folded channel, wave number
    size_t smem;
    const float4 *ctab, *stab;           // [q][nq][KG] cos, sin of 4 wave numbers
    const float4 *cinv, *sinv;           // [q][mk][NG] cos, sin of 4 terms (NG apart)
    int64_t lines() const { return outer * S; }
};

// Fill in the tiling; false: a line's channels do not fit shared memory.
bool axis_plan(Axis &a, int L, int m, int rows, int64_t S, int64_t outer, int W);
// Host tables in the order ctab, stab, cinv, sinv (floats); `count` each.
void axis_tables(const Axis &a, std::vector<float> &out, size_t count[4]);

bool set_attrs();

// u [+]= IDFT(R . DFT(v)) along one axis: v, u [B][W][N]; R packed [m][W][Wp]
// complex (Wp = W rounded up to 4); wk scales the spectrum, ak what goes into
// the inverse (null: 1); spec, if given, receives the scaled spectrum as
// [m][W][B lines] real parts, then imaginary parts.
void spectral(const Axis &a, const float *v, float *u, int B, int W, int64_t N, const float2 *R, const float *wk,
              const float *ak, float *spec, bool accumulate, cudaStream_t s);

// R [i][o][m] complex (parameter layout, floats) of the three axes ->
// rf [m][i][Wp], ra [m][o][Wp] conjugated (rows in the order the mixing reads)
struct PackR {
    struct { const float *R; int m; float2 *rf, *ra; } a[3];
};
void pack_r(const PackR &p, int W, cudaStream_t s);

// gR(i, o, k) = sum over lines of G(o) conj V(i), both as `spec` above; part:
// grad_r_parts(...) x m W W float2 of scratch
int grad_r_parts(int m, int64_t lines);
void grad_r(const float *G, const float *V, int W, int m, int64_t lines, float2 *part, float *gR, cudaStream_t s);

// y = W2 act(W1 x + b1) + b2 [+ res] per cell; fields [B][c][N]
struct Mlp {
    int ci, ch, co, act;
    float w0;
    const float *W1, *b1, *W2, *b2;
};
bool mlp_fits(int ci, int ch, int co);
void mlp(const Mlp &p, const float *x, const float *res, float *y, int B, int64_t N, cudaStream_t s);
// gx = dL/dx (may be null with ACT_GELU) and the gradients of (W1, b1, W2, b2), contiguous at
// gw, from g = dL/dy; part: mlp_parts() x (sizes of the four) floats
int mlp_parts();
void mlp_bwd(const Mlp &p, const float *x, const float *g, float *gx, float *part, float *gw, int B, int64_t N,
             cudaStream_t s);

}  // namespace ffno
