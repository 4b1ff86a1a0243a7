// ffno_fast.cu -- tiled kernels of the factorised surrogate (FP32 activations
// and arithmetic).
//   k_spectral   one axis of u [+]= IDFT(R . DFT(v)): a block takes T lines of
//                all channels through the folded transform, the channel mixing
//                and the inverse in shared memory
//   k_grad_r     the spectral weights' gradient, a split reduction over lines
//   k_mlp        the pointwise networks, two cells per thread in registers
//   k_mlp_bwd    their backward: hidden values recomputed, weight gradients
//                accumulated per block and summed in a fixed order
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "ffno_fast.h"
#include "sm_count.h"

namespace ffno {
namespace {

constexpr int TPB = 256;
constexpr size_t SMEM_TWO = 113 * 1024;      // two blocks per SM
constexpr size_t SMEM_MAX = 226 * 1024;

__device__ __forceinline__ float4 f4(float v) { return make_float4(v, v, v, v); }
__device__ __forceinline__ float4 operator+(float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
__device__ __forceinline__ float4 operator-(float4 a, float4 b) { return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w); }
__device__ __forceinline__ void fma4(float4 &d, float s, const float4 &v)
{
    d.x = fmaf(s, v.x, d.x);
    d.y = fmaf(s, v.y, d.y);
    d.z = fmaf(s, v.z, d.z);
    d.w = fmaf(s, v.w, d.w);
}
__device__ __forceinline__ float4 mul4(float s, const float4 &v) { return make_float4(s * v.x, s * v.y, s * v.z, s * v.w); }

// ---------------------------------------------------------------------------
// spectral convolution along one axis
// ---------------------------------------------------------------------------
// Four neighbouring lines of sample n of a channel: contiguous along the lines
// (ROWS = 0), or one element of each of four rows (ROWS = 1).
struct Tile {
    int64_t base;        // element of sample 0, line 0 of channel 0
    int64_t sn;          // between samples
    int64_t sl;          // between lines
    int valid;           // lines of this tile that exist
};

__device__ __forceinline__ void async16(float *dst, const float *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

__device__ __forceinline__ void async8(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

__device__ __forceinline__ void async4(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

__device__ __forceinline__ void async_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// copy the four lines into shared memory (this thread's own 16 bytes), zeros
// past the tile's lines
template <int ROWS>
__device__ __forceinline__ void fetch4(float *dst, const float *p, const Tile &t, int64_t off, int l, bool vec)
{
    if (!ROWS && vec) {
        if (l < t.valid) async16(dst, p + off);
        else *reinterpret_cast<float4 *>(dst) = f4(0.f);
        return;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (l + q < t.valid) async4(dst + q, p + off + q * t.sl);
        else dst[q] = 0.f;
}

// Store, or add without reading back: one kernel at a time adds to a field, one
// addition per element, so the sum does not depend on the order of the blocks.
template <int ROWS>
__device__ __forceinline__ void store4(float *p, const Tile &t, int64_t off, int l, bool vec, bool add, const float4 &v)
{
    if (!ROWS && vec) {
        if (l >= t.valid) return;
        if (add) atomicAdd(reinterpret_cast<float4 *>(p + off), v);
        else *reinterpret_cast<float4 *>(p + off) = v;
        return;
    }
    const float w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (l + q < t.valid) {
            if (add) atomicAdd(p + off + q * t.sl, w[q]);
            else p[off + q * t.sl] = w[q];
        }
}

// n / d for n, d < 2^16: mul = ceil(2^32 / d) (0 stands for d = 1)
__device__ __forceinline__ int fdiv(int n, uint32_t mul) { return mul ? (int)__umulhi((uint32_t)n, mul) : n; }

// V(o) += R(i, o) V(i) for 4 lines and 4 outputs: re, im of the input's lines
__device__ __forceinline__ void mix4(float4 *gr, float4 *gi, const float4 *w, const float4 &x, const float4 &y)
{
    const float c[8] = {w[0].x, w[0].y, w[0].z, w[0].w, w[1].x, w[1].y, w[1].z, w[1].w};
#pragma unroll
    for (int o = 0; o < 4; ++o) {
        fma4(gr[o], c[2 * o], x);
        fma4(gr[o], -c[2 * o + 1], y);
        fma4(gi[o], c[2 * o + 1], x);
        fma4(gi[o], c[2 * o], y);
    }
}

// Channel mixing of a tile in place: V [k][c][T], V(o) <- ak sum_i V(i) R(i, o).
// Thread = 4 lines x 4 outputs (complex), 64 multiply-adds per two operands
// from shared memory and two from L2 (read two steps ahead); the lanes of one
// wave number and 4 lines (a power of two of them) sit in one warp, read all
// inputs, then write.  WC: the width when it is a constant, else 0.
template <int WC>
__device__ __forceinline__ void mix_phase(float *Vre, float *Vim, int m, int KS, int T, int W,
                                          const float2 *__restrict__ R, const float *__restrict__ ak)
{
    const int TQ = T >> 2, tqs = TQ == 1 ? 0 : (TQ == 2 ? 1 : 2);
    const int OG = (W + 3) >> 2, ogs = OG > 4 ? 3 : (OG > 2 ? 2 : (OG > 1 ? 1 : 0)), units = (m * TQ) << ogs;
    for (int i0 = 0; i0 < units; i0 += TPB) {
        const int idx = i0 + (int)threadIdx.x, r = idx >> ogs;
        const int og = idx & ((1 << ogs) - 1);
        const bool on = idx < units && og < OG;
        const int l = (r & (TQ - 1)) << 2, k = on ? r >> tqs : 0;
        const float4 *rp = reinterpret_cast<const float4 *>(R + (int64_t)k * W * OG * 4) + og;
        float *vr = Vre + k * KS + l, *vi = Vim + k * KS + l;
        float4 gr[4], gi[4];
#pragma unroll
        for (int o = 0; o < 4; ++o) gr[o] = gi[o] = f4(0.f);
        if (on) {
            if (WC) {
                float4 b[3][2][2];              // two inputs' weights per step, two steps ahead
#pragma unroll
                for (int st = 0; st < 2; ++st)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        b[st][h][0] = __ldg(rp + (2 * st + h) * OG * 2);
                        b[st][h][1] = __ldg(rp + (2 * st + h) * OG * 2 + OG);
                    }
#pragma unroll
                for (int st = 0; st < WC / 2; ++st) {
                    if (st + 2 < WC / 2)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            b[(st + 2) % 3][h][0] = __ldg(rp + (2 * st + 4 + h) * OG * 2);
                            b[(st + 2) % 3][h][1] = __ldg(rp + (2 * st + 4 + h) * OG * 2 + OG);
                        }
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        mix4(gr, gi, b[st % 3][h], *reinterpret_cast<const float4 *>(vr + (2 * st + h) * T),
                             *reinterpret_cast<const float4 *>(vi + (2 * st + h) * T));
                }
            } else {
#pragma unroll 4
                for (int i = 0; i < W; ++i) {
                    const float4 c[2] = {__ldg(rp + i * OG * 2), __ldg(rp + i * OG * 2 + OG)};
                    mix4(gr, gi, c, *reinterpret_cast<const float4 *>(vr + i * T),
                         *reinterpret_cast<const float4 *>(vi + i * T));
                }
            }
        }
        __syncwarp();
        if (on) {
            const float sc = ak ? ak[k] : 1.f;
#pragma unroll
            for (int o = 0; o < 4; ++o) {
                if (4 * og + o >= W) break;
                *reinterpret_cast<float4 *>(vr + (4 * og + o) * T) = mul4(sc, gr[o]);
                *reinterpret_cast<float4 *>(vi + (4 * og + o) * T) = mul4(sc, gi[o]);
            }
        }
    }
}

// A persistent block over tiles of T lines x W channels x L samples.  Phases,
// a barrier between them:
//   fold     D [c][class][n][T]: even and odd parts of the lines, split by the
//            parity of the wave number they serve; each thread folds in place
//            what it copied itself
//   forward  V [k][c][T]: thread = 4 wave numbers x 4 lines, real and
//            imaginary part: 32 multiply-adds per four 16-byte operands
//   mix      in place on V
//   inverse  thread = 4 terms x 4 lines of all four symmetric sums, unfolded
//            into 16 samples and stored
// D is free after the forward phase: the next tile's copies are issued there
// and land behind the mixing and the inverse.
// WC: the width when it is a constant (full unrolling), else 0.
template <int ROWS, int WC>
__global__ void __launch_bounds__(TPB, 2) k_spectral(const Axis a, const float *__restrict__ v, float *u, int Wr,
                                                     int64_t N, const float2 *__restrict__ R,
                                                     const float *__restrict__ wk, const float *__restrict__ ak,
                                                     float *__restrict__ spec, int64_t NL, int tiles, int total,
                                                     int accumulate)
{
    extern __shared__ float4 raw[];
    const int W = WC ? WC : Wr;
    float *D = reinterpret_cast<float *>(raw);
    float *Vre = D + W * a.DS, *Vim = Vre + a.m * a.KS;
    const int T = a.T, TQ = T >> 2, tid = threadIdx.x;
    const int tqs = TQ == 1 ? 0 : (TQ == 2 ? 1 : 2);
    const bool vec = !ROWS && (a.S & 3) == 0;
    const int L = a.L, nq = a.nq, cls = nq * T;

    auto lines_of = [&](int64_t w, int64_t &line0) {
        Tile t;
        const int64_t ti = w % tiles;
        w /= tiles;
        if (ROWS) {
            t.base = w * W * N + ti * T * L;
            t.sn = 1;
            t.sl = L;
            t.valid = (int)min((int64_t)T, a.outer - ti * T);
            line0 = w * a.outer + ti * T;
        } else {
            const int64_t o = w % a.outer, b = w / a.outer;
            t.base = b * W * N + o * L * a.S + ti * T;
            t.sn = a.S;
            t.sl = 1;
            t.valid = (int)min((int64_t)T, a.S - ti * T);
            line0 = (b * a.outer + o) * a.S + ti * T;
        }
        return t;
    };
    auto place = [&](int idx, int &j, int &l, int &c) {
        if (ROWS) {                                 // neighbouring threads: neighbouring samples
            const int r = fdiv(idx, a.dnq);
            j = idx - r * nq;
            l = (r & (TQ - 1)) << 2;
            c = r >> tqs;
        } else {
            l = (idx & (TQ - 1)) << 2;
            const int r = idx >> tqs;
            c = fdiv(r, a.dnq);
            j = r - c * nq;
        }
    };
    // each thread copies its own (n, L - n, L/2 - n, L/2 + n) into the places
    // of its four folded values
    auto fetch = [&](const Tile &t) {
        for (int idx = tid; idx < W * nq * TQ; idx += TPB) {
            int j, l, c;
            place(idx, j, l, c);
            const int64_t p0 = t.base + (int64_t)c * N + (int64_t)l * t.sl;
            auto ld = [&](float *dst, int n) { fetch4<ROWS>(dst, v, t, p0 + (int64_t)n * t.sn, l, vec); };
            float *d = D + c * a.DS + j * T + l;
            ld(d, j);
            if (a.q == 2) {
                ld(d + cls, j == 0 ? L / 2 : L - j);
                if (j > 0 && 4 * j < L) {
                    ld(d + 2 * cls, L / 2 - j);
                    ld(d + 3 * cls, L / 2 + j);
                }
            } else if (j > 0 && 2 * j != L) {
                ld(d + cls, L - j);
            }
        }
    };

    int64_t line0 = 0, line_next = 0;
    Tile t = lines_of(blockIdx.x, line0), tn = t;
    fetch(t);
    for (int w = blockIdx.x; w < total; w += gridDim.x, t = tn, line0 = line_next) {
        async_wait();
        for (int idx = tid; idx < W * nq * TQ; idx += TPB) {
            int j, l, c;
            place(idx, j, l, c);
            float4 *d0 = reinterpret_cast<float4 *>(D + c * a.DS + j * T + l);
            float4 *d1 = d0 + cls / 4, *d2 = d1 + cls / 4, *d3 = d2 + cls / 4;
            const float4 x = *d0;
            if (a.q == 2) {
                const float4 y = *d1, e = x + y, o = x - y;
                if (j == 0) {                       // x(0), x(L/2)
                    *d0 = e;
                    *d1 = o;
                    *d2 = *d3 = f4(0.f);
                } else if (4 * j == L) {            // x(L/4), x(3L/4)
                    *d0 = e;
                    *d1 = *d2 = f4(0.f);
                    *d3 = o;
                } else {
                    const float4 z = *d2, q = *d3, eb = z + q, ob = z - q;
                    *d0 = e + eb;
                    *d1 = e - eb;
                    *d2 = o - ob;
                    *d3 = o + ob;
                }
            } else if (j > 0 && 2 * j != L) {
                const float4 y = *d1;
                *d0 = x + y;
                *d1 = x - y;
            } else {
                *d1 = f4(0.f);
            }
        }
        __syncthreads();

        // forward: V(k) = wk (sum_n E cos - i sum_n O sin)
        for (int idx = tid; idx < W * TQ * a.q * a.KG; idx += TPB) {
            int r = fdiv(idx, a.dKG);
            const int kg = idx - r * a.KG;
            const int par = a.q == 2 ? (r & 1) : 0;
            r = a.q == 2 ? r >> 1 : r;
            const int l = (r & (TQ - 1)) << 2, c = r >> tqs;
            const float *e = D + c * a.DS + par * cls + l, *o = e + a.q * cls;
            const float4 *ct = a.ctab + par * nq * a.KG + kg, *st = a.stab + par * nq * a.KG + kg;
            float4 re[4], im[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) re[k] = im[k] = f4(0.f);
#pragma unroll 4
            for (int n = 0; n < nq; ++n) {
                const float4 cw = __ldg(ct + n * a.KG), sw = __ldg(st + n * a.KG);
                const float4 x = *reinterpret_cast<const float4 *>(e + n * T);
                const float4 y = *reinterpret_cast<const float4 *>(o + n * T);
                fma4(re[0], cw.x, x);
                fma4(re[1], cw.y, x);
                fma4(re[2], cw.z, x);
                fma4(re[3], cw.w, x);
                fma4(im[0], sw.x, y);
                fma4(im[1], sw.y, y);
                fma4(im[2], sw.z, y);
                fma4(im[3], sw.w, y);
            }
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                const int k = par + a.q * (4 * kg + kk);
                if (k >= a.m) break;
                const float sc = wk ? wk[k] : 1.f;
                const float4 vr = mul4(sc, re[kk]), vi = mul4(-sc, im[kk]);
                *reinterpret_cast<float4 *>(Vre + k * a.KS + c * T + l) = vr;
                *reinterpret_cast<float4 *>(Vim + k * a.KS + c * T + l) = vi;
                if (spec) {
                    const int64_t at = ((int64_t)k * W + c) * NL + line0 + l;
                    float *sr = spec + at, *si = sr + (int64_t)a.m * W * NL;
                    if (l + 4 <= t.valid && (at & 3) == 0 && (NL & 3) == 0) {
                        *reinterpret_cast<float4 *>(sr) = vr;
                        *reinterpret_cast<float4 *>(si) = vi;
                    } else {
                        const float pr[4] = {vr.x, vr.y, vr.z, vr.w}, pi[4] = {vi.x, vi.y, vi.z, vi.w};
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            if (l + q < t.valid) {
                                sr[q] = pr[q];
                                si[q] = pi[q];
                            }
                    }
                }
            }
        }
        __syncthreads();
        if (w + (int)gridDim.x < total) {
            tn = lines_of(w + (int)gridDim.x, line_next);
            fetch(tn);
        }

        mix_phase<WC>(Vre, Vim, a.m, a.KS, T, W, R, ak);
        __syncthreads();

        // inverse: u(n) = sum_k (Gre cos - Gim sin)
        for (int idx = tid; idx < W * TQ * a.NG; idx += TPB) {
            const int r = fdiv(idx, a.dNG), ng = idx - r * a.NG;
            const int l = (r & (TQ - 1)) << 2, c = r >> tqs;
            const float *gr = Vre + c * T + l, *gi = Vim + c * T + l;
            const float4 *ct = a.cinv + ng, *st = a.sinv + ng;
            const int64_t p0 = t.base + (int64_t)c * N + (int64_t)l * t.sl;
            auto put = [&](int n, const float4 &x) {
                store4<ROWS>(u, t, p0 + (int64_t)n * t.sn, l, vec, accumulate != 0, x);
            };
            if (a.q == 2) {
                float4 ce[4], co[4], se[4], so[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) ce[j] = co[j] = se[j] = so[j] = f4(0.f);
#pragma unroll 2
                for (int kk = 0; kk < a.mk; ++kk) {
                    const int k0 = 2 * kk, k1 = min(2 * kk + 1, a.m - 1);       // past the end: zero tables
                    const float4 x0 = *reinterpret_cast<const float4 *>(gr + k0 * a.KS);
                    const float4 y0 = *reinterpret_cast<const float4 *>(gi + k0 * a.KS);
                    const float4 x1 = *reinterpret_cast<const float4 *>(gr + k1 * a.KS);
                    const float4 y1 = *reinterpret_cast<const float4 *>(gi + k1 * a.KS);
                    const float4 c0 = __ldg(ct + kk * a.NG), s0 = __ldg(st + kk * a.NG);
                    const float4 c1 = __ldg(ct + (a.mk + kk) * a.NG), s1 = __ldg(st + (a.mk + kk) * a.NG);
                    fma4(ce[0], c0.x, x0);
                    fma4(ce[1], c0.y, x0);
                    fma4(ce[2], c0.z, x0);
                    fma4(ce[3], c0.w, x0);
                    fma4(se[0], s0.x, y0);
                    fma4(se[1], s0.y, y0);
                    fma4(se[2], s0.z, y0);
                    fma4(se[3], s0.w, y0);
                    fma4(co[0], c1.x, x1);
                    fma4(co[1], c1.y, x1);
                    fma4(co[2], c1.z, x1);
                    fma4(co[3], c1.w, x1);
                    fma4(so[0], s1.x, y1);
                    fma4(so[1], s1.y, y1);
                    fma4(so[2], s1.z, y1);
                    fma4(so[3], s1.w, y1);
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int n = ng + j * a.NG;
                    if (4 * n >= L) break;
                    const float4 p = ce[j] + co[j], m = ce[j] - co[j], s = se[j] + so[j], d = se[j] - so[j];
                    put(n, p - s);
                    if (n == 0) {
                        put(L / 2, m);
                    } else {
                        put(L - n, p + s);
                        put(L / 2 - n, m + d);
                        put(L / 2 + n, m - d);
                    }
                }
            } else {
                float4 ce[4], se[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) ce[j] = se[j] = f4(0.f);
                for (int kk = 0; kk < a.mk; ++kk) {
                    const float4 x = *reinterpret_cast<const float4 *>(gr + kk * a.KS);
                    const float4 y = *reinterpret_cast<const float4 *>(gi + kk * a.KS);
                    const float4 c0 = __ldg(ct + kk * a.NG), s0 = __ldg(st + kk * a.NG);
                    fma4(ce[0], c0.x, x);
                    fma4(ce[1], c0.y, x);
                    fma4(ce[2], c0.z, x);
                    fma4(ce[3], c0.w, x);
                    fma4(se[0], s0.x, y);
                    fma4(se[1], s0.y, y);
                    fma4(se[2], s0.z, y);
                    fma4(se[3], s0.w, y);
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int n = ng + j * a.NG;
                    if (n >= nq) break;
                    put(n, ce[j] - se[j]);
                    if (n > 0 && 2 * n != L) put(L - n, ce[j] + se[j]);
                }
            }
        }
        // the self-symmetric term n = L/4 (its cosines and sines are 0, 1, -1),
        // one thread per channel and 4 lines
        if (a.q == 2)
            for (int idx = TPB - 1 - tid; idx < W * TQ; idx += TPB) {
                const int l = (idx & (TQ - 1)) << 2, c = idx >> tqs;
                const float *gr = Vre + c * T + l, *gi = Vim + c * T + l;
                float4 p = f4(0.f), s = f4(0.f);
                for (int k = 0; k < a.m; k += 4) {
                    p = p + *reinterpret_cast<const float4 *>(gr + k * a.KS);
                    if (k + 2 < a.m) p = p - *reinterpret_cast<const float4 *>(gr + (k + 2) * a.KS);
                    if (k + 1 < a.m) s = s + *reinterpret_cast<const float4 *>(gi + (k + 1) * a.KS);
                    if (k + 3 < a.m) s = s - *reinterpret_cast<const float4 *>(gi + (k + 3) * a.KS);
                }
                const int64_t p0 = t.base + (int64_t)c * N + (int64_t)l * t.sl;
                store4<ROWS>(u, t, p0 + (int64_t)(L / 4) * t.sn, l, vec, accumulate != 0, p - s);
                store4<ROWS>(u, t, p0 + (int64_t)(L - L / 4) * t.sn, l, vec, accumulate != 0, p + s);
            }
    }
}

// ---------------------------------------------------------------------------
// the same for the usual lengths, with the transform in registers
// ---------------------------------------------------------------------------
// cos(2 pi j / n) and sin(2 pi j / n) from their Taylor series at the argument
// reduced to [0, pi/4] (double; 20 terms leave less than 1e-20)
constexpr double taylor(double x, bool sine)
{
    double t = sine ? x : 1.0, s = t;
    for (int k = sine ? 2 : 1; k < 40; k += 2) {
        t *= -x * x / (k * (k + 1.0));
        s += t;
    }
    return s;
}
constexpr double sincos_of(int j, int n, bool sine)
{
    j %= n;
    if (sine) return 2 * j > n ? -sincos_of(n - j, n, true)
                   : 4 * j > n ? (8 * j > 3 * n ? taylor(2 * M_PI * (n - 2 * j) / (2.0 * n), true)
                                                : taylor(2 * M_PI * (4 * j - n) / (4.0 * n), false))
                   : 8 * j > n ? taylor(2 * M_PI * (n - 4 * j) / (4.0 * n), false)
                               : taylor(2 * M_PI * j / n, true);
    return 2 * j > n ? sincos_of(n - j, n, false)
         : 4 * j > n ? -(8 * j > 3 * n ? taylor(2 * M_PI * (n - 2 * j) / (2.0 * n), false)
                                       : taylor(2 * M_PI * (4 * j - n) / (4.0 * n), true))
         : 8 * j > n ? taylor(2 * M_PI * (n - 4 * j) / (4.0 * n), true)
                     : taylor(2 * M_PI * j / n, false);
}

template <int A, int B, int STEP = 1, class F>
__device__ __forceinline__ void each(const F &f)
{
    if constexpr (A < B) {
        f(std::integral_constant<int, A>());
        each<A + STEP, B, STEP>(f);
    }
}

// s += c x with the constant c (nothing where it is 0)
template <int J, int N, bool SINE>
__device__ __forceinline__ void cfma(float &s, float x)
{
    constexpr double d = sincos_of(J, N, SINE);
    constexpr float c = d < 1e-12 && d > -1e-12 ? 0.f : (float)d;
    if constexpr (c == 1.f) s += x;
    else if constexpr (c == -1.f) s -= x;
    else if constexpr (c != 0.f) s = fmaf(c, x, s);
}

// The wave numbers of parity PAR (-1: all) below M of one line whose folded
// samples are E0, E1 (even parts), O0, O1 (odd parts): st(k, re, im).
template <int L, int M, int PAR, class F>
__device__ __forceinline__ void forward_line(const float *E, const float *O, const F &st)
{
    each<0, M>([&](auto kc) {
        constexpr int k = kc;
        if constexpr (PAR < 0 || (k & 1) == PAR) {
            constexpr int Q = L / 4 + 1, off = PAR < 0 ? (k & 1) * Q : 0;
            float re = 0.f, im = 0.f;
            each<0, Q>([&](auto nc) {
                constexpr int n = nc;
                cfma<(k * n) % L, L, false>(re, E[off + n]);
                cfma<(k * n) % L, L, true>(im, O[off + n]);
            });
            st(kc, re, im);
        }
    });
}

// The samples n, L - n, L/2 - n, L/2 + n of one line for FIRST <= n < LAST
// (n <= L/4) from its wave numbers: put(index, value), in this order.
template <int L, int M, int FIRST, int LAST, class F>
__device__ __forceinline__ void inverse_line(const float *re, const float *im, const F &put)
{
    each<FIRST, LAST>([&](auto nc) {
        constexpr int n = nc;
        float ce = 0.f, co = 0.f, se = 0.f, so = 0.f;
        each<0, M>([&](auto kc) {
            constexpr int k = kc;
            if constexpr (k & 1) {
                cfma<(k * n) % L, L, false>(co, re[k]);
                cfma<(k * n) % L, L, true>(so, im[k]);
            } else {
                cfma<(k * n) % L, L, false>(ce, re[k]);
                cfma<(k * n) % L, L, true>(se, im[k]);
            }
        });
        const float p = ce + co, s = se + so;
        put(nc, p - s);
        if constexpr (n > 0) put(std::integral_constant<int, L - n>(), p + s);
        if constexpr (n == 0) put(std::integral_constant<int, L / 2>(), ce - co);
        if constexpr (n > 0 && 4 * n != L) {
            const float m = ce - co, d = se - so;
            put(std::integral_constant<int, L / 2 - n>(), m + d);
            put(std::integral_constant<int, L / 2 + n>(), m - d);
        }
    });
}

__device__ __forceinline__ void put1(float *p, float v, bool add)
{
    if (add) atomicAdd(p, v);
    else *p = v;
}

__device__ __forceinline__ void put4(float *p, const float4 &v, bool add)
{
    if (add) atomicAdd(reinterpret_cast<float4 *>(p), v);
    else *reinterpret_cast<float4 *>(p) = v;
}

// One thread per line (c, t), its samples in registers: the transforms'
// cosines are immediate operands, so they take one instruction per
// multiply-add and shared memory carries the samples and spectra once (the
// tabulated kernel above is bound by shared-memory reads: 32 multiply-adds per
// four 16-byte operands).  The next tile's samples are copied behind the
// mixing and the inverse.
//   ROWS = 0 (samples S apart): X [c][n][8 lines]; stores run along the lines
//   ROWS = 1 (contiguous samples): X [c, row][L + 4], read 16 bytes at a time;
//     a line is shared by two threads (wave numbers of even and odd parity;
//     the lower and the upper half of the terms back, 16 bytes per store)
template <int L, int M, int ROWS>
__global__ void __launch_bounds__(TPB, 2) k_spectral_reg(const Axis a, const float *__restrict__ v, float *u, int W,
                                                         int64_t N, const float2 *__restrict__ R,
                                                         const float *__restrict__ wk, const float *__restrict__ ak,
                                                         float *__restrict__ spec, int64_t NL, int tiles, int total,
                                                         int accumulate)
{
    extern __shared__ float4 raw[];
    constexpr int T = ROWS ? 4 : 8, TS = ROWS ? 2 : 3, P = L + 4, CS = L * T + 8, Q = L / 4 + 1, H = L / 8;
    const int tid = threadIdx.x;
    float *X = reinterpret_cast<float *>(raw), *Vre = X + W * (ROWS ? T * P : CS), *Vim = Vre + a.m * a.KS;
    const int64_t plane = (int64_t)a.m * W * NL;
    const bool vec = ROWS || (a.S & 3) == 0, add = accumulate != 0;

    auto lines_of = [&](int w, int64_t &line0) {
        Tile t;
        const int64_t ti = w % tiles, ob = w / tiles;
        if (ROWS) {
            t.base = ob * W * N + ti * T * L;
            t.valid = (int)min((int64_t)T, a.outer - ti * T);
            line0 = ob * a.outer + ti * T;
        } else {
            const int64_t o = ob % a.outer, b = ob / a.outer;
            t.base = b * W * N + o * L * a.S + ti * T;
            t.valid = (int)min((int64_t)T, a.S - ti * T);
            line0 = ob * a.S + ti * T;
        }
        t.sn = a.S;
        t.sl = 1;
        return t;
    };
    auto fetch = [&](const Tile &t) {
        if (ROWS) {                                  // 16 bytes along a row
            for (int idx = tid; idx < W * T * (L / 4); idx += TPB) {
                const int x = (idx % (L / 4)) * 4, r = idx / (L / 4);
                if ((r & (T - 1)) < t.valid)
                    async16(X + r * P + x, v + t.base + (int64_t)(r >> TS) * N + (r & (T - 1)) * L + x);
            }
        } else {                                     // 16 bytes along the lines
            for (int idx = tid; idx < W * L * (T / 4); idx += TPB) {
                const int l = (idx & (T / 4 - 1)) * 4, r = idx / (T / 4), n = r % L, c = r / L;
                fetch4<0>(X + c * CS + n * T + l, v, t, t.base + (int64_t)c * N + n * a.S + l, l, vec);
            }
        }
    };

    int64_t line0 = 0, line_next = 0;
    Tile t = lines_of(blockIdx.x, line0), tn = t;
    fetch(t);
    for (int w = blockIdx.x; w < total; w += gridDim.x, t = tn, line0 = line_next) {
        async_wait();
        __syncthreads();

        // forward: one line, or one parity of a line, per thread
        constexpr int SPLIT = ROWS ? 2 : 1;
        for (int i0 = 0; i0 < W * T * SPLIT; i0 += TPB) {
            // the parity is uniform over half a block
            const int par = ROWS ? tid / (TPB / 2) : 0;
            const int ln = ROWS ? i0 / 2 + tid % (TPB / 2) : i0 + tid;
            const int c = ln >> TS, l = ln & (T - 1);
            if (ln >= W * T) continue;
            const bool ok = l < t.valid;
            auto out = [&](auto kc, float re, float im) {
                constexpr int k = kc;
                if (k < a.m) {
                    const float sc = wk ? wk[k] : 1.f;
                    const float x = ok ? sc * re : 0.f, y = ok ? -sc * im : 0.f;
                    Vre[k * a.KS + ln] = x;
                    Vim[k * a.KS + ln] = y;
                    if (spec && ok) {
                        float *s = spec + ((int64_t)k * W + c) * NL + line0 + l;
                        s[0] = x;
                        s[plane] = y;
                    }
                }
            };
            float x[L];
            if constexpr (ROWS) {
                const float4 *src = reinterpret_cast<const float4 *>(X + ln * P);
#pragma unroll
                for (int n = 0; n < L / 4; ++n) {
                    const float4 q = src[n];
                    x[4 * n] = q.x;
                    x[4 * n + 1] = q.y;
                    x[4 * n + 2] = q.z;
                    x[4 * n + 3] = q.w;
                }
                float E[Q], O[Q];
                const float sg = par ? -1.f : 1.f;
#pragma unroll
                for (int n = 0; n < Q; ++n) {
                    if (n == 0) {
                        E[0] = fmaf(sg, x[L / 2], x[0]);
                        O[0] = 0.f;
                    } else if (4 * n == L) {
                        E[n] = par ? 0.f : x[n] + x[L - n];
                        O[n] = par ? x[n] - x[L - n] : 0.f;
                    } else {
                        E[n] = fmaf(sg, x[L / 2 - n] + x[L / 2 + n], x[n] + x[L - n]);
                        O[n] = fmaf(-sg, x[L / 2 - n] - x[L / 2 + n], x[n] - x[L - n]);
                    }
                }
                if (par) forward_line<L, M, 1>(E, O, out);
                else forward_line<L, M, 0>(E, O, out);
            } else {
                float E[2 * Q], O[2 * Q];
                const float *src = X + c * CS + l;
#pragma unroll
                for (int n = 0; n < L; ++n) x[n] = src[n * T];
#pragma unroll
                for (int n = 0; n < Q; ++n) {
                    if (n == 0) {
                        E[0] = x[0] + x[L / 2];
                        E[Q] = x[0] - x[L / 2];
                        O[0] = O[Q] = 0.f;
                    } else if (4 * n == L) {
                        E[n] = x[n] + x[L - n];
                        O[Q + n] = x[n] - x[L - n];
                        E[Q + n] = O[n] = 0.f;
                    } else {
                        const float ea = x[n] + x[L - n], eb = x[L / 2 - n] + x[L / 2 + n];
                        const float oa = x[n] - x[L - n], ob = x[L / 2 - n] - x[L / 2 + n];
                        E[n] = ea + eb;
                        E[Q + n] = ea - eb;
                        O[n] = oa - ob;
                        O[Q + n] = oa + ob;
                    }
                }
                forward_line<L, M, -1>(E, O, out);
            }
        }
        __syncthreads();
        if (w + (int)gridDim.x < total) {
            tn = lines_of(w + (int)gridDim.x, line_next);
            fetch(tn);
        }
        if (W == MAXW) mix_phase<MAXW>(Vre, Vim, a.m, a.KS, T, W, R, ak);
        else mix_phase<0>(Vre, Vim, a.m, a.KS, T, W, R, ak);
        __syncthreads();

        // inverse
        for (int i0 = 0; i0 < W * T * SPLIT; i0 += TPB) {
            const int par = ROWS ? tid / (TPB / 2) : 0;
            const int ln = ROWS ? i0 / 2 + tid % (TPB / 2) : i0 + tid;
            const int c = ln >> TS, l = ln & (T - 1);
            if (ln >= W * T || l >= t.valid) continue;
            float re[M], im[M];
#pragma unroll
            for (int k = 0; k < M; ++k) {
                re[k] = k < a.m ? Vre[k * a.KS + ln] : 0.f;
                im[k] = k < a.m ? Vim[k * a.KS + ln] : 0.f;
            }
            if constexpr (ROWS) {
                // the terms below L/8 give the samples within L/8 of 0 and L/2,
                // the others those around L/4 and 3L/4; 16 bytes are stored
                // once their four samples are there
                float *dst = u + t.base + (int64_t)c * N + (int64_t)l * L;
                float x[L];
                auto run = [&](auto fc, auto lc) {
                    constexpr int F = fc, E = lc;
                    inverse_line<L, M, F, E>(re, im, [&](auto nc, float val) {
                        constexpr int n = nc;
                        x[n] = val;
                    });
                    each<0, L / 4>([&](auto qc) {
                        constexpr int q = 4 * qc;
                        // the term that gives sample n: its distance to the nearest multiple of L/2
                        constexpr auto term = [](int n) { const int r = n % (L / 2); return r > L / 4 ? L / 2 - r : r; };
                        constexpr bool all = term(q) >= F && term(q) < E && term(q + 1) >= F && term(q + 1) < E &&
                                             term(q + 2) >= F && term(q + 2) < E && term(q + 3) >= F && term(q + 3) < E;
                        if constexpr (all) {
                            put4(dst + q, make_float4(x[q], x[q + 1], x[q + 2], x[q + 3]), add);
                        } else {
                            each<0, 4>([&](auto ic) {
                                constexpr int n = q + ic;
                                if constexpr (term(n) >= F && term(n) < E) put1(dst + n, x[n], add);
                            });
                        }
                    });
                };
                if (par) run(std::integral_constant<int, H>(), std::integral_constant<int, Q>());
                else run(std::integral_constant<int, 0>(), std::integral_constant<int, H>());
            } else {
                float *dst = u + t.base + (int64_t)c * N + l;
                if (add) inverse_line<L, M, 0, Q>(re, im, [&](auto nc, float val) { constexpr int n = nc; atomicAdd(dst + n * a.S, val); });
                else inverse_line<L, M, 0, Q>(re, im, [&](auto nc, float val) { constexpr int n = nc; dst[n * a.S] = val; });
            }
        }
    }
}

// R [i][o][m] -> rf [m][i] and the conjugate transpose ra [m][o], each row of
// Wp entries in the order the mixing reads them: entries 4g, 4g + 1 of every
// group g, then entries 4g + 2, 4g + 3 (neighbouring lanes read neighbouring
// 16 bytes)
__global__ void k_pack_r(const PackR pr, int W, int Wp)
{
    const float *R = pr.a[blockIdx.y].R;
    float2 *rf = pr.a[blockIdx.y].rf, *ra = pr.a[blockIdx.y].ra;
    const int m = pr.a[blockIdx.y].m, n = m * W * Wp;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
        const int e = t % Wp, r = (t / Wp) % W, k = t / (Wp * W);
        const int half = e / (Wp / 2), x = e % (Wp / 2), p = (x >> 1) * 4 + half * 2 + (x & 1);
        float2 f = make_float2(0.f, 0.f), g = f;
        if (p < W) {
            const int64_t j = (((int64_t)r * W + p) * m + k) * 2, h = (((int64_t)p * W + r) * m + k) * 2;
            f = make_float2(R[j], R[j + 1]);
            g = make_float2(R[h], -R[h + 1]);
        }
        rf[t] = f;
        ra[t] = g;
    }
}

// ---------------------------------------------------------------------------
// gradient of the spectral weights
// ---------------------------------------------------------------------------
constexpr int GL = 64, GLP = GL + 4;         // lines per shared-memory tile, row stride
constexpr size_t GRAD_SMEM = sizeof(float) * 2 * 4 * MAXW * GLP;

// Block (k, split): a W x W complex product over the split's lines, thread =
// 4 x 4 entries of one of four line groups (rows n4 apart keep the 16-byte
// operand reads free of bank conflicts); 256 multiply-adds per 16 operands.
// The next tile is copied behind the products (without that the reads'
// latency was exposed: 442 against 260 us for 32 x 32 x 16 wave numbers of
// 65,536 lines).
__global__ void __launch_bounds__(TPB, 2) k_grad_r(const float *__restrict__ G, const float *__restrict__ V, int W,
                                                   int m, int64_t NL, int splits, float2 *__restrict__ part)
{
    extern __shared__ float4 raw[];
    float (*tiles)[4][MAXW][GLP] = reinterpret_cast<float (*)[4][MAXW][GLP]>(raw);       // [2]: G re, G im, V re, V im
    const int k = blockIdx.x % m, sp = blockIdx.x / m, tid = threadIdx.x;
    const int64_t quads = (NL + GL - 1) / GL;
    const int64_t l0 = quads * sp / splits * GL, l1 = min(NL, quads * (sp + 1) / splits * GL);
    const int64_t plane = (int64_t)m * W * NL;
    const float *src[4] = {G + (int64_t)k * W * NL, G + plane + (int64_t)k * W * NL, V + (int64_t)k * W * NL,
                           V + plane + (int64_t)k * W * NL};
    const int n4 = (W + 3) >> 2, grp = tid >> 6, e = tid & 63;
    const int ig = e % n4, og = e / n4;
    const bool active = og < n4;
    const bool vec = (NL & 3) == 0;
    float re[4][4], im[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int o = 0; o < 4; ++o) re[i][o] = im[i][o] = 0.f;
    for (int q = tid; q < 2 * 4 * MAXW * GLP; q += TPB) (&tiles[0][0][0][0])[q] = 0.f;
    __syncthreads();
    auto copy = [&](int64_t l, float (*sh)[MAXW][GLP]) {
        for (int q = tid; q < 4 * W * (GL / 4); q += TPB) {
            const int x = (q % (GL / 4)) * 4, c = (q / (GL / 4)) % W, f = q / (GL / 4 * W);
            const float *p = src[f] + (int64_t)c * NL + l + x;
            float *d = &sh[f][c][x];
            if (vec && l + x < l1) {
                async16(d, p);
            } else {
                float4 w = f4(0.f);
                if (l + x < l1) w.x = p[0];
                if (l + x + 1 < l1) w.y = p[1];
                if (l + x + 2 < l1) w.z = p[2];
                if (l + x + 3 < l1) w.w = p[3];
                *reinterpret_cast<float4 *>(d) = w;
            }
        }
    };
    int buf = 0;
    if (l0 < l1) copy(l0, tiles[0]);
    for (int64_t l = l0; l < l1; l += GL, buf ^= 1) {
        async_wait();
        __syncthreads();                                     // the tile is there, the other one free
        if (l + GL < l1) copy(l + GL, tiles[buf ^ 1]);
        float (*sh)[MAXW][GLP] = tiles[buf];
        if (active) {
            for (int x = grp * 4; x < GL; x += 16) {
                float4 gr[4], gi[4];
#pragma unroll
                for (int o = 0; o < 4; ++o) {
                    const int row = min(og + n4 * o, MAXW - 1);
                    gr[o] = *reinterpret_cast<const float4 *>(&sh[0][row][x]);
                    gi[o] = *reinterpret_cast<const float4 *>(&sh[1][row][x]);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int row = min(ig + n4 * i, MAXW - 1);
                    const float4 vr = *reinterpret_cast<const float4 *>(&sh[2][row][x]);
                    const float4 vi = *reinterpret_cast<const float4 *>(&sh[3][row][x]);
#pragma unroll
                    for (int o = 0; o < 4; ++o) {           // g conj(v)
                        float a = re[i][o], b = im[i][o];
                        a = fmaf(gr[o].x, vr.x, a); a = fmaf(gi[o].x, vi.x, a);
                        b = fmaf(gi[o].x, vr.x, b); b = fmaf(-gr[o].x, vi.x, b);
                        a = fmaf(gr[o].y, vr.y, a); a = fmaf(gi[o].y, vi.y, a);
                        b = fmaf(gi[o].y, vr.y, b); b = fmaf(-gr[o].y, vi.y, b);
                        a = fmaf(gr[o].z, vr.z, a); a = fmaf(gi[o].z, vi.z, a);
                        b = fmaf(gi[o].z, vr.z, b); b = fmaf(-gr[o].z, vi.z, b);
                        a = fmaf(gr[o].w, vr.w, a); a = fmaf(gi[o].w, vi.w, a);
                        b = fmaf(gi[o].w, vr.w, b); b = fmaf(-gr[o].w, vi.w, b);
                        re[i][o] = a;
                        im[i][o] = b;
                    }
                }
            }
        }
    }
    __syncthreads();
    // the four line groups' sums, in order
    float2 *acc = reinterpret_cast<float2 *>(raw);                     // [MAXW][MAXW]
    for (int g = 0; g < 4; ++g) {
        if (active && grp == g)
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int o = 0; o < 4; ++o) {
                    const int ri = ig + n4 * i, ro = og + n4 * o;
                    if (ri >= W || ro >= W) continue;
                    float2 *d = acc + ri * MAXW + ro;
                    *d = g == 0 ? make_float2(re[i][o], im[i][o]) : make_float2(d->x + re[i][o], d->y + im[i][o]);
                }
        __syncthreads();
    }
    float2 *out = part + ((int64_t)sp * m + k) * W * W;
    for (int q = tid; q < W * W; q += TPB) out[q] = acc[q / W * MAXW + q % W];
}

// part [splits][k][i][o] -> gR [i][o][k]
__global__ void k_grad_r_sum(const float2 *__restrict__ part, int W, int m, int splits, float *__restrict__ gR)
{
    const int n = m * W * W, t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    float re = 0.f, im = 0.f;
    for (int s = 0; s < splits; ++s) {
        const float2 p = part[(int64_t)s * n + t];
        re += p.x;
        im += p.y;
    }
    const int k = t / (W * W), io = t % (W * W);
    gR[((int64_t)io * m + k) * 2] = re;
    gR[((int64_t)io * m + k) * 2 + 1] = im;
}

// ---------------------------------------------------------------------------
// pointwise networks
// ---------------------------------------------------------------------------
template <int ACT>
__device__ __forceinline__ float act_of(float z, float w0)
{
    if (ACT == ACT_GELU) return 0.5f * z * (1.f + erff(z * 0.70710678118654752f));
    return sinf(w0 * z);
}

// value and derivative
template <int ACT>
__device__ __forceinline__ void act_both(float z, float w0, float &h, float &dh)
{
    if (ACT == ACT_GELU) {
        const float c = 0.5f * (1.f + erff(z * 0.70710678118654752f));
        h = z * c;
        dh = c + z * expf(-0.5f * z * z) * 0.39894228040143268f;
    } else {
        float sn, cs;
        sincosf(w0 * z, &sn, &cs);
        h = sn;
        dh = w0 * cs;
    }
}

// weights into shared memory: W1 [ch][CI], W2 transposed [ch][CO], zeros in
// the padding (chp rows)
template <int CI, int CO>
__device__ __forceinline__ void stage_weights(const Mlp &p, int chp, float *w1, float *w2, float *b1, float *b2)
{
    for (int q = threadIdx.x; q < chp * CI; q += blockDim.x) {
        const int j = q / CI, c = q % CI;
        w1[q] = j < p.ch && c < p.ci ? p.W1[j * p.ci + c] : 0.f;
    }
    for (int q = threadIdx.x; q < chp * CO; q += blockDim.x) {
        const int j = q / CO, o = q % CO;
        w2[q] = j < p.ch && o < p.co ? p.W2[o * p.ch + j] : 0.f;
    }
    for (int q = threadIdx.x; q < chp; q += blockDim.x) b1[q] = q < p.ch ? p.b1[q] : 0.f;
    if (b2)
        for (int q = threadIdx.x; q < CO; q += blockDim.x) b2[q] = q < p.co ? p.b2[q] : 0.f;
}

template <int V> struct Vec;
template <> struct Vec<1> { using T = float; };
template <> struct Vec<2> { using T = float2; };

constexpr int MT = 128;                      // threads of the forward kernel

// A thread's V cells keep their CI inputs and CO outputs in registers; the
// weights are broadcast from shared memory, so the kernel is bound by the
// multiply-adds and the activation.  Each thread copies its next cells' inputs
// into its own places of shared memory while it computes (no barrier: nobody
// else reads them), which 12 warps per SM would not hide otherwise.
template <int CI, int CO, int ACT, int V>
__global__ void __launch_bounds__(MT, 3) k_mlp(const Mlp p, const float *__restrict__ x, const float *res, float *y,
                                               int B, int64_t N)
{
    extern __shared__ float4 raw[];
    using T = typename Vec<V>::T;
    const int chp = (p.ch + 1) & ~1;
    float *w1 = reinterpret_cast<float *>(raw), *w2 = w1 + chp * CI, *b1 = w2 + chp * CO, *b2 = b1 + ((chp + 3) & ~3);
    T *next = reinterpret_cast<T *>(b2 + CO) + threadIdx.x;
    stage_weights<CI, CO>(p, chp, w1, w2, b1, b2);
    __syncthreads();
    const int64_t items = B * N / V, step = (int64_t)gridDim.x * MT;
    auto fetch = [&](int64_t it) {
        if (it >= items) return;
        const int64_t cell = it * V, b = cell / N, n = cell - b * N;
        const float *src = x + b * p.ci * N + n;
#pragma unroll 8
        for (int c = 0; c < p.ci; ++c, src += N) {
            if (V == 2) async8(next + c * MT, src);
            else async4(next + c * MT, src);
        }
    };
    int64_t it = (int64_t)blockIdx.x * MT + threadIdx.x;
    fetch(it);
    for (; it < items; it += step) {
        const int64_t cell = it * V, b = cell / N, n = cell - b * N;
        float in[CI][V], out[CO][V];
        async_wait();
#pragma unroll
        for (int c = 0; c < CI; ++c) {
            if (c < p.ci) *reinterpret_cast<T *>(in[c]) = next[c * MT];
            else
#pragma unroll
                for (int q = 0; q < V; ++q) in[c][q] = 0.f;
        }
        fetch(it + step);
#pragma unroll
        for (int o = 0; o < CO; ++o)
#pragma unroll
            for (int q = 0; q < V; ++q) out[o][q] = b2[o];
#pragma unroll 1
        for (int j = 0; j < chp; j += 2) {
            float z[2][V];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
#pragma unroll
                for (int q = 0; q < V; ++q) z[h][q] = b1[j + h];
            }
#pragma unroll
            for (int c = 0; c < CI; c += 4)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float4 w = *reinterpret_cast<const float4 *>(w1 + (j + h) * CI + c);
#pragma unroll
                    for (int q = 0; q < V; ++q) {
                        z[h][q] = fmaf(w.x, in[c][q], z[h][q]);
                        z[h][q] = fmaf(w.y, in[c + 1][q], z[h][q]);
                        z[h][q] = fmaf(w.z, in[c + 2][q], z[h][q]);
                        z[h][q] = fmaf(w.w, in[c + 3][q], z[h][q]);
                    }
                }
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int q = 0; q < V; ++q) z[h][q] = act_of<ACT>(z[h][q], p.w0);
#pragma unroll
            for (int o = 0; o < CO; o += 4)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float4 w = *reinterpret_cast<const float4 *>(w2 + (j + h) * CO + o);
#pragma unroll
                    for (int q = 0; q < V; ++q) {
                        out[o][q] = fmaf(w.x, z[h][q], out[o][q]);
                        out[o + 1][q] = fmaf(w.y, z[h][q], out[o + 1][q]);
                        out[o + 2][q] = fmaf(w.z, z[h][q], out[o + 2][q]);
                        out[o + 3][q] = fmaf(w.w, z[h][q], out[o + 3][q]);
                    }
                }
        }
        float *dst = y + b * p.co * N + n;
        if (res) {                               // `in` is free: sixteen residuals in flight at once
            const float *r = res + b * p.co * N + n;
#pragma unroll
            for (int o = 0; o < CO; o += 16) {
                float v[16][V];
#pragma unroll
                for (int k = 0; k < 16 && o + k < CO; ++k, r += N)
                    if (o + k < p.co) *reinterpret_cast<T *>(v[k]) = *reinterpret_cast<const T *>(r);
#pragma unroll
                for (int k = 0; k < 16 && o + k < CO; ++k)
                    if (o + k < p.co)
#pragma unroll
                        for (int q = 0; q < V; ++q) out[o + k][q] += v[k][q];
            }
        }
#pragma unroll
        for (int o = 0; o < CO; ++o, dst += N)
            if (o < p.co) *reinterpret_cast<T *>(dst) = *reinterpret_cast<const T *>(out[o]);
    }
}

constexpr int BT = 128;                      // threads of the backward kernel = cells of a tile
constexpr int BTP = BT + 4;                  // row stride of its tiles
constexpr int HC = 32;                       // hidden units per chunk

// Backward of the same network, a persistent block over tiles of 128 cells; the
// hidden values are recomputed (cheaper than keeping two fields per layer), 32
// hidden units at a time.  All five products (hidden values and their
// gradients, the input gradient, both weight gradients) read their operands
// from shared memory in register tiles of 8 rows x 4 cells or 4 x 4 sums of
// four cells, 32 multiply-adds per three 16-byte operands and 64 per eight: one
// cell per thread was bound by those reads (4 multiply-adds per broadcast
// weight).  32 -> 32 -> 32 at 8 x 524,288 cells:
// 1.16 ms, where the multiply-adds alone take 0.60 ms; 32 -> 128 -> 4: 3.63 ms
// (three blocks per SM with some spills; two without: 5.10); the six networks
// of a training step 13.4 -> 9.1 ms.
// A warp owns 32 cells up to the input gradient: lanes = 8 quadruples of cells
// x 4 groups of rows.  The weight gradients take all cells: 64 threads x (4
// hidden units x N1 or N2 rows) in each half of the cells, rows 8 apart (row
// stride of 132: conflict-free).
template <int CI, int CO, int ACT, int NCH, bool GX>
__global__ void __launch_bounds__(BT, NCH == 4 && CO > 8 ? 2 : 3) k_mlp_bwd(const Mlp p, const float *__restrict__ x,
                                                                  const float *__restrict__ g, float *__restrict__ gx,
                                                                  int B, int64_t N, int vec, float *__restrict__ part)
{
    extern __shared__ float4 raw[];
    constexpr int chp = NCH * HC, N1 = CI / 8, N2 = CO / 8;
    constexpr int WS = chp + 4;                              // row stride of W1 transposed
    float *w1 = reinterpret_cast<float *>(raw), *w2 = w1 + CI * WS, *b1 = w2 + CO * chp;
    float *X = b1 + chp, *G = X + CI * BTP, *H = G + CO * BTP, *GH = H + HC * BTP;
    const int tid = threadIdx.x;
    for (int q = tid; q < chp * CI; q += BT) {               // W1 transposed [CI][ch], W2 [CO][ch]
        const int j = q / CI, c = q % CI;
        w1[c * WS + j] = j < p.ch && c < p.ci ? p.W1[j * p.ci + c] : 0.f;
    }
    for (int q = tid; q < CO * chp; q += BT) {
        const int o = q / chp, j = q % chp;
        w2[q] = j < p.ch && o < p.co ? p.W2[o * p.ch + j] : 0.f;
    }
    for (int q = tid; q < chp; q += BT) b1[q] = q < p.ch ? p.b1[q] : 0.f;
    const int lane = tid & 31, r4 = lane >> 3, r8 = r4 * 8, cq = (tid >> 5) * 32 + (lane & 7) * 4;      // 8 rows, 4 cells
    const int hg = (tid >> 3) & 7, cg = tid & 7, half = tid >> 6;
    const int sr = tid >> 2, sq = (tid & 3) * 4;             // row and cells of the bias sums
    float a1[NCH][4][N1], a2[NCH][4][N2], s1[NCH], s2 = 0.f;
#pragma unroll
    for (int k = 0; k < NCH; ++k) {
        s1[k] = 0.f;
#pragma unroll
        for (int h = 0; h < 4; ++h) {
#pragma unroll
            for (int c = 0; c < N1; ++c) a1[k][h][c] = 0.f;
#pragma unroll
            for (int c = 0; c < N2; ++c) a2[k][h][c] = 0.f;
        }
    }
    const int64_t cells = B * N;
    for (int64_t c0 = (int64_t)blockIdx.x * BT; c0 < cells; c0 += (int64_t)gridDim.x * BT) {
        if (vec) {                                           // N % 4 == 0: a quadruple lies in one sample
            const int qd = 4 * lane;
            const int64_t cell = c0 + qd, b = cell / N, n = cell - b * N;
            const bool ok = cell < cells;
            for (int c = tid >> 5; c < CI; c += BT / 32) {
                if (ok && c < p.ci) async16(X + c * BTP + qd, x + (b * p.ci + c) * N + n);
                else *reinterpret_cast<float4 *>(X + c * BTP + qd) = f4(0.f);
            }
            for (int o = tid >> 5; o < CO; o += BT / 32) {
                if (ok && o < p.co) async16(G + o * BTP + qd, g + (b * p.co + o) * N + n);
                else *reinterpret_cast<float4 *>(G + o * BTP + qd) = f4(0.f);
            }
            async_wait();
        } else {
            const int64_t cell = c0 + tid, b = cell / N, n = cell - b * N;
            const bool ok = cell < cells;
#pragma unroll 8
            for (int c = 0; c < CI; ++c) X[c * BTP + tid] = ok && c < p.ci ? x[(b * p.ci + c) * N + n] : 0.f;
#pragma unroll 8
            for (int o = 0; o < CO; ++o) G[o * BTP + tid] = ok && o < p.co ? g[(b * p.co + o) * N + n] : 0.f;
        }
        __syncthreads();
        float4 gi[GX ? 8 : 1];
        if (GX)
#pragma unroll
            for (int i = 0; i < 8; ++i) gi[i] = f4(0.f);
#pragma unroll
        for (int k = 0; k < NCH; ++k) {
            // z and dL/dh of 8 hidden units and 4 cells, into H and GH
            {
                float4 z[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) z[i] = f4(b1[k * HC + r8 + i]);
#pragma unroll 4
                for (int c = 0; c < CI; ++c) {
                    const float4 v = *reinterpret_cast<const float4 *>(X + c * BTP + cq);
                    const float *w = w1 + c * WS + k * HC + r8;
                    const float4 wa = *reinterpret_cast<const float4 *>(w), wb = *reinterpret_cast<const float4 *>(w + 4);
                    fma4(z[0], wa.x, v); fma4(z[1], wa.y, v); fma4(z[2], wa.z, v); fma4(z[3], wa.w, v);
                    fma4(z[4], wb.x, v); fma4(z[5], wb.y, v); fma4(z[6], wb.z, v); fma4(z[7], wb.w, v);
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) *reinterpret_cast<float4 *>(H + (r8 + i) * BTP + cq) = z[i];
#pragma unroll
                for (int i = 0; i < 8; ++i) z[i] = f4(0.f);
#pragma unroll 4
                for (int o = 0; o < CO; ++o) {
                    const float4 v = *reinterpret_cast<const float4 *>(G + o * BTP + cq);
                    const float *w = w2 + o * chp + k * HC + r8;
                    const float4 wa = *reinterpret_cast<const float4 *>(w), wb = *reinterpret_cast<const float4 *>(w + 4);
                    fma4(z[0], wa.x, v); fma4(z[1], wa.y, v); fma4(z[2], wa.z, v); fma4(z[3], wa.w, v);
                    fma4(z[4], wb.x, v); fma4(z[5], wb.y, v); fma4(z[6], wb.z, v); fma4(z[7], wb.w, v);
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) *reinterpret_cast<float4 *>(GH + (r8 + i) * BTP + cq) = z[i];
            }
            // the activation, on this thread's own entries (rolled: 32 inlined
            // copies would not fit the instruction cache)
#pragma unroll 1
            for (int i = 0; i < 8; ++i) {
                float4 *hp = reinterpret_cast<float4 *>(H + (r8 + i) * BTP + cq);
                float4 *gp = reinterpret_cast<float4 *>(GH + (r8 + i) * BTP + cq);
                const float4 z = *hp, d = *gp;
                float4 v, dv;
                act_both<ACT>(z.x, p.w0, v.x, dv.x);
                act_both<ACT>(z.y, p.w0, v.y, dv.y);
                act_both<ACT>(z.z, p.w0, v.z, dv.z);
                act_both<ACT>(z.w, p.w0, v.w, dv.w);
                *hp = v;
                *gp = make_float4(d.x * dv.x, d.y * dv.y, d.z * dv.z, d.w * dv.w);
            }
            __syncthreads();
            if (GX) {
#pragma unroll 2
                for (int h = 0; h < HC; h += 4) {            // channels r4 + 4 i
                    float4 v[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) v[u] = *reinterpret_cast<const float4 *>(GH + (h + u) * BTP + cq);
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float4 w = *reinterpret_cast<const float4 *>(w1 + (r4 + 4 * i) * WS + k * HC + h);
                        fma4(gi[i], w.x, v[0]); fma4(gi[i], w.y, v[1]); fma4(gi[i], w.z, v[2]); fma4(gi[i], w.w, v[3]);
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < BT; q += 16) {
                const float4 v = *reinterpret_cast<const float4 *>(GH + sr * BTP + q + sq);
                s1[k] += (v.x + v.y) + (v.z + v.w);
            }
            if (k == 0 && sr < CO)
#pragma unroll
                for (int q = 0; q < BT; q += 16) {
                    const float4 v = *reinterpret_cast<const float4 *>(G + sr * BTP + q + sq);
                    s2 += (v.x + v.y) + (v.z + v.w);
                }
#pragma unroll 1
            for (int q = half * (BT / 2); q < (half + 1) * (BT / 2); q += 4) {
                float4 v[4];
#pragma unroll
                for (int h = 0; h < 4; ++h) v[h] = *reinterpret_cast<const float4 *>(GH + (hg + 8 * h) * BTP + q);
#pragma unroll
                for (int c = 0; c < N1; ++c) {
                    const float4 w = *reinterpret_cast<const float4 *>(X + (cg + 8 * c) * BTP + q);
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        float t = a1[k][h][c];
                        t = fmaf(v[h].x, w.x, t);
                        t = fmaf(v[h].y, w.y, t);
                        t = fmaf(v[h].z, w.z, t);
                        a1[k][h][c] = fmaf(v[h].w, w.w, t);
                    }
                }
#pragma unroll
                for (int h = 0; h < 4; ++h) v[h] = *reinterpret_cast<const float4 *>(H + (hg + 8 * h) * BTP + q);
#pragma unroll
                for (int c = 0; c < N2; ++c) {
                    const float4 w = *reinterpret_cast<const float4 *>(G + (cg + 8 * c) * BTP + q);
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        float t = a2[k][h][c];
                        t = fmaf(v[h].x, w.x, t);
                        t = fmaf(v[h].y, w.y, t);
                        t = fmaf(v[h].z, w.z, t);
                        a2[k][h][c] = fmaf(v[h].w, w.w, t);
                    }
                }
            }
            __syncthreads();
        }
        if (GX && vec) {
            const int64_t cell = c0 + cq, b = cell / N, n = cell - b * N;
            if (cell < cells)
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (r4 + 4 * i < p.ci) *reinterpret_cast<float4 *>(gx + (b * p.ci + r4 + 4 * i) * N + n) = gi[i];
        } else if (GX) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int64_t cell = c0 + cq + e, b = cell / N, n = cell - b * N;
                if (cell < cells)
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        if (r4 + 4 * i < p.ci)
                            gx[(b * p.ci + r4 + 4 * i) * N + n] = e == 0 ? gi[i].x : e == 1 ? gi[i].y : e == 2 ? gi[i].z : gi[i].w;
            }
        }
    }
    // this block's sums, in the parameters' order: W1 [ch][ci], b1, W2 [co][ch],
    // b2; the second half of the cells through shared memory
    const int n1 = p.ch * p.ci, n2 = p.co * p.ch;
    float *d = part + (int64_t)blockIdx.x * (n1 + p.ch + n2 + p.co);
    float *red = X + (tid & 63);
    if (half)
#pragma unroll
        for (int k = 0; k < NCH; ++k)
#pragma unroll
            for (int h = 0; h < 4; ++h) {
#pragma unroll
                for (int c = 0; c < N1; ++c) red[((k * 4 + h) * (N1 + N2) + c) * 64] = a1[k][h][c];
#pragma unroll
                for (int c = 0; c < N2; ++c) red[((k * 4 + h) * (N1 + N2) + N1 + c) * 64] = a2[k][h][c];
            }
    __syncthreads();
    if (!half)
#pragma unroll
        for (int k = 0; k < NCH; ++k)
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int j = k * HC + hg + 8 * h;
                if (j >= p.ch) continue;
#pragma unroll
                for (int c = 0; c < N1; ++c)
                    if (cg + 8 * c < p.ci)
                        d[j * p.ci + cg + 8 * c] = a1[k][h][c] + red[((k * 4 + h) * (N1 + N2) + c) * 64];
#pragma unroll
                for (int c = 0; c < N2; ++c)
                    if (cg + 8 * c < p.co)
                        d[n1 + p.ch + (cg + 8 * c) * p.ch + j] =
                            a2[k][h][c] + red[((k * 4 + h) * (N1 + N2) + N1 + c) * 64];
            }
#pragma unroll
    for (int k = 0; k < NCH; ++k) {
        float t = s1[k];
        t += __shfl_xor_sync(0xffffffffu, t, 1);
        t += __shfl_xor_sync(0xffffffffu, t, 2);
        if ((tid & 3) == 0 && k * HC + sr < p.ch) d[n1 + k * HC + sr] = t;
    }
    s2 += __shfl_xor_sync(0xffffffffu, s2, 1);
    s2 += __shfl_xor_sync(0xffffffffu, s2, 2);
    if ((tid & 3) == 0 && sr < p.co) d[n1 + p.ch + n2 + sr] = s2;
}

// out[q] = sum over the parts, 8 interleaved FP64 sums added in order
__global__ void __launch_bounds__(256) k_sum_parts(const float *__restrict__ part, int P, int n, float *__restrict__ out)
{
    __shared__ double sh[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, q = blockIdx.x * 32 + lane;
    double s = 0.0;
    if (q < n)
        for (int p = w; p < P; p += 8) s += part[(int64_t)p * n + q];
    sh[w][lane] = s;
    __syncthreads();
    if (w == 0 && q < n) {
        for (int k = 1; k < 8; ++k) s += sh[k][lane];
        out[q] = (float)s;
    }
}

int round4(int v) { return (v + 3) & ~3; }

// smallest stride >= v, a multiple of 4, that leaves `rem` on division by 32
int stride_for(int v, int rem)
{
    v = round4(v);
    while (v % 32 != rem) v += 4;
    return v;
}

}  // namespace

namespace {

typedef void (*SpecKernel)(Axis, const float *, float *, int, int64_t, const float2 *, const float *, const float *,
                           float *, int64_t, int, int, int);

// the register kernel of a length, or null: the lengths of the surrogate grids
// (samples S apart: a line fits a thread's registers up to 64)
SpecKernel k_reg(const Axis &a)
{
    switch (a.m > 32 ? 0 : a.L * 2 + (a.m > 16)) {
    case 64: return a.rows ? k_spectral_reg<32, 16, 1> : k_spectral_reg<32, 16, 0>;
    case 96: return a.rows ? k_spectral_reg<48, 16, 1> : k_spectral_reg<48, 16, 0>;
    case 128: return a.rows ? k_spectral_reg<64, 16, 1> : k_spectral_reg<64, 16, 0>;
    case 129: return a.rows ? k_spectral_reg<64, 32, 1> : nullptr;
    case 192:
    case 193: return a.rows ? k_spectral_reg<96, 32, 1> : nullptr;
    case 256:
    case 257: return a.rows ? k_spectral_reg<128, 32, 1> : nullptr;
    default: return nullptr;
    }
}

}  // namespace

// T: as many lines as leave room for two blocks per SM (long runs along the
// lines and fewer reads of the weights), 4 lines in one block where they do not.
bool axis_plan(Axis &a, int L, int m, int rows, int64_t S, int64_t outer, int W)
{
    if (W < 1 || W > MAXW) return false;
    a = Axis{};
    a.L = L; a.m = m; a.rows = rows; a.S = S; a.outer = outer;
    a.q = L % 4 == 0 ? 2 : 1;
    a.nq = a.q == 2 ? L / 4 + 1 : L / 2 + 1;
    a.mk = (m + a.q - 1) / a.q;
    a.KG = (a.mk + 3) / 4;
    a.NG = a.q == 2 ? (L / 4 + 3) / 4 : (a.nq + 3) / 4;
    auto recip = [](int d) { return d > 1 ? (uint32_t)((((uint64_t)1 << 32) + d - 1) / d) : 0u; };
    a.dnq = recip(a.nq);
    a.dKG = recip(a.KG);
    a.dNG = recip(a.NG);
    if (k_reg(a)) {
        a.reg = 1;
        a.T = rows ? 4 : 8;
        a.KS = stride_for(W * a.T, 0) + 4;
        a.smem = sizeof(float) * ((size_t)2 * m * a.KS + (size_t)W * (rows ? a.T * (L + 4) : a.T * L + 8));
        if (a.smem <= SMEM_TWO) return true;
        a.reg = 0;
    }
    for (int T = 16; T >= 4; T /= 2) {
        a.T = T;
        a.DS = stride_for(2 * a.q * a.nq * T, T);
        a.KS = stride_for(W * T, 4);
        a.smem = sizeof(float) * ((size_t)W * a.DS + (size_t)2 * m * a.KS);
        if (a.smem <= SMEM_TWO) return true;
    }
    return a.smem <= SMEM_MAX && (int64_t)W * a.nq * 4 < 65536;
}

void axis_tables(const Axis &a, std::vector<float> &out, size_t count[4])
{
    out.clear();
    auto ang = [&](int k, int n) { return 2.0 * M_PI * (double)(((int64_t)k * n) % a.L) / a.L; };
    for (int f = 0; f < 4; ++f) {
        const size_t before = out.size();
        const bool sine = f & 1;
        for (int par = 0; par < a.q; ++par) {
            if (f < 2) {
                for (int n = 0; n < a.nq; ++n)
                    for (int kk = 0; kk < 4 * a.KG; ++kk) {
                        const int k = par + a.q * kk;
                        out.push_back(k < a.m ? (float)(sine ? std::sin(ang(k, n)) : std::cos(ang(k, n))) : 0.f);
                    }
            } else {
                for (int kk = 0; kk < a.mk; ++kk)
                    for (int g = 0; g < a.NG; ++g)
                        for (int j = 0; j < 4; ++j) {
                            const int k = par + a.q * kk, n = g + j * a.NG;
                            const bool in = k < a.m && n < a.nq;
                            out.push_back(in ? (float)(sine ? std::sin(ang(k, n)) : std::cos(ang(k, n))) : 0.f);
                        }
            }
        }
        count[f] = out.size() - before;
    }
}

void spectral(const Axis &a, const float *v, float *u, int B, int W, int64_t N, const float2 *R, const float *wk,
              const float *ak, float *spec, bool accumulate, cudaStream_t s)
{
    const int64_t run = a.rows ? a.outer : a.S;
    const int tiles = (int)((run + a.T - 1) / a.T);
    const int64_t total = (int64_t)B * tiles * (a.rows ? 1 : a.outer), NL = B * a.lines();
    const int grid = (int)std::min<int64_t>(total, (int64_t)gb300::sm_count() * (a.smem <= SMEM_TWO ? 2 : 1));
    if (a.reg) {
        k_reg(a)<<<grid, TPB, a.smem, s>>>(a, v, u, W, N, R, wk, ak, spec, NL, tiles, (int)total, accumulate);
        return;
    }
    auto k = a.rows ? (W == MAXW ? k_spectral<1, MAXW> : k_spectral<1, 0>)
                    : (W == MAXW ? k_spectral<0, MAXW> : k_spectral<0, 0>);
    k<<<grid, TPB, a.smem, s>>>(a, v, u, W, N, R, wk, ak, spec, NL, tiles, (int)total, accumulate);
}

void pack_r(const PackR &p, int W, cudaStream_t s)
{
    const int Wp = round4(W), m = std::max({p.a[0].m, p.a[1].m, p.a[2].m});
    k_pack_r<<<dim3((unsigned)std::min(gb300::sm_count() * 4, (m * W * Wp + TPB - 1) / TPB), 3), TPB, 0, s>>>(p, W, Wp);
}

int grad_r_parts(int m, int64_t lines)
{
    const int want = std::max(1, 4 * gb300::sm_count() / std::max(1, m));
    return (int)std::max<int64_t>(1, std::min<int64_t>(want, (lines + GL - 1) / GL));
}

void grad_r(const float *G, const float *V, int W, int m, int64_t lines, float2 *part, float *gR, cudaStream_t s)
{
    const int sp = grad_r_parts(m, lines);
    k_grad_r<<<m * sp, TPB, GRAD_SMEM, s>>>(G, V, W, m, lines, sp, part);
    k_grad_r_sum<<<(m * W * W + TPB - 1) / TPB, TPB, 0, s>>>(part, W, m, sp, gR);
}

bool mlp_fits(int ci, int ch, int co) { return ci <= MAXW && co <= MAXW && ch <= 128; }

namespace {

template <int CI, int CO, int ACT>
void mlp_v(const Mlp &p, const float *x, const float *res, float *y, int B, int64_t N, cudaStream_t s)
{
    const int chp = (p.ch + 1) & ~1;
    const size_t smem = sizeof(float) * (size_t)(chp * (CI + CO) + round4(chp) + CO + 2 * CI * MT);
    const uintptr_t al = (uintptr_t)x | (uintptr_t)res | (uintptr_t)y;
    const bool two = N % 2 == 0 && (al & 7) == 0;
    const int64_t items = B * N / (two ? 2 : 1);
    const int grid = (int)std::min<int64_t>((items + MT - 1) / MT, (int64_t)gb300::sm_count() * 3);
    if (two) k_mlp<CI, CO, ACT, 2><<<grid, MT, smem, s>>>(p, x, res, y, B, N);
    else k_mlp<CI, CO, ACT, 1><<<grid, MT, smem, s>>>(p, x, res, y, B, N);
}

template <int ACT>
void mlp_act(const Mlp &p, const float *x, const float *res, float *y, int B, int64_t N, cudaStream_t s)
{
    if (p.ci <= 8) mlp_v<8, 32, ACT>(p, x, res, y, B, N, s);
    else if (p.co <= 8) mlp_v<32, 8, ACT>(p, x, res, y, B, N, s);
    else mlp_v<32, 32, ACT>(p, x, res, y, B, N, s);
}

template <int CI, int CO, int ACT, int NCH, bool GX>
size_t bwd_smem() { return sizeof(float) * (size_t)(NCH * HC * (CI + CO + 1) + 4 * CI + (CI + CO + 2 * HC) * BTP); }

int bwd_grid(int64_t cells) { return (int)std::min<int64_t>((cells + BT - 1) / BT, mlp_parts()); }

template <int CI, int CO, int ACT, int NCH, bool GX>
void bwd_k(const Mlp &p, const float *x, const float *g, float *gx, float *part, int B, int64_t N, cudaStream_t s)
{
    // 16-byte copies where a quadruple of cells stays in a sample and is aligned
    const int vec = N % 4 == 0 && (((uintptr_t)x | (uintptr_t)g | (uintptr_t)gx) & 15) == 0;
    k_mlp_bwd<CI, CO, ACT, NCH, GX><<<bwd_grid(B * N), BT, bwd_smem<CI, CO, ACT, NCH, GX>(), s>>>(p, x, g, gx, B, N, vec, part);
}

template <int CI, int CO, int ACT, bool GX>
void bwd_n(const Mlp &p, const float *x, const float *g, float *gx, float *part, int B, int64_t N, cudaStream_t s)
{
    if (p.ch <= HC) bwd_k<CI, CO, ACT, 1, GX>(p, x, g, gx, part, B, N, s);
    else if (p.ch <= 2 * HC) bwd_k<CI, CO, ACT, 2, GX>(p, x, g, gx, part, B, N, s);
    else bwd_k<CI, CO, ACT, 4, GX>(p, x, g, gx, part, B, N, s);
}

template <int ACT>
void bwd_act(const Mlp &p, const float *x, const float *g, float *gx, float *part, int B, int64_t N, cudaStream_t s)
{
    if constexpr (ACT == ACT_GELU)             // the lift, the one network without an input gradient
        if (!gx) {
            if (p.ci <= 8) bwd_n<8, 32, ACT, false>(p, x, g, gx, part, B, N, s);
            else bwd_n<32, 32, ACT, false>(p, x, g, gx, part, B, N, s);
            return;
        }
    if (p.co <= 8) bwd_n<32, 8, ACT, true>(p, x, g, gx, part, B, N, s);
    else bwd_n<32, 32, ACT, true>(p, x, g, gx, part, B, N, s);
}

template <class K>
bool big(K k, size_t bytes)
{
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
}

template <int CI, int CO, int ACT, bool GX>
bool big_bwd()
{
    return big(k_mlp_bwd<CI, CO, ACT, 1, GX>, bwd_smem<CI, CO, ACT, 1, GX>()) &&
           big(k_mlp_bwd<CI, CO, ACT, 2, GX>, bwd_smem<CI, CO, ACT, 2, GX>()) &&
           big(k_mlp_bwd<CI, CO, ACT, 4, GX>, bwd_smem<CI, CO, ACT, 4, GX>());
}

template <int CI, int CO, int ACT>
bool big_mlp()
{
    constexpr size_t most = sizeof(float) * (size_t)(128 * (CI + CO + 1) + CO + 2 * CI * MT);
    return big(k_mlp<CI, CO, ACT, 1>, most) && big(k_mlp<CI, CO, ACT, 2>, most);
}

template <int ACT>
bool big_act()
{
    if constexpr (ACT == ACT_GELU)
        if (!big_bwd<8, 32, ACT, false>() || !big_bwd<32, 32, ACT, false>()) return false;
    return big_mlp<8, 32, ACT>() && big_mlp<32, 8, ACT>() && big_mlp<32, 32, ACT>() && big_bwd<32, 8, ACT, true>() &&
           big_bwd<32, 32, ACT, true>();
}

}  // namespace

void mlp(const Mlp &p, const float *x, const float *res, float *y, int B, int64_t N, cudaStream_t s)
{
    if (p.act == ACT_SIREN) mlp_act<ACT_SIREN>(p, x, res, y, B, N, s);
    else mlp_act<ACT_GELU>(p, x, res, y, B, N, s);
}

int mlp_parts() { return gb300::sm_count() * 3; }

void mlp_bwd(const Mlp &p, const float *x, const float *g, float *gx, float *part, float *gw, int B, int64_t N,
             cudaStream_t s)
{
    if (p.act == ACT_SIREN) bwd_act<ACT_SIREN>(p, x, g, gx, part, B, N, s);
    else bwd_act<ACT_GELU>(p, x, g, gx, part, B, N, s);
    const int n = p.ch * p.ci + p.ch + p.co * p.ch + p.co;
    k_sum_parts<<<(n + 31) / 32, 256, 0, s>>>(part, bwd_grid(B * N), n, gw);
}

// The dynamic shared-memory limits are per device: set on every creation.
bool set_attrs()
{
    for (int L : {32, 48, 64, 96, 128})
        for (int m : {16, 32})
            for (int rows : {0, 1}) {
                Axis a{};
                a.L = L; a.m = m; a.rows = rows;
                SpecKernel k = k_reg(a);
                if (k && !big(k, SMEM_TWO)) return false;
            }
    return big(k_grad_r, GRAD_SMEM) && big(k_spectral<0, 0>, SMEM_MAX) && big(k_spectral<1, 0>, SMEM_MAX) &&
           big(k_spectral<0, MAXW>, SMEM_MAX) && big(k_spectral<1, MAXW>, SMEM_MAX) && big_act<ACT_GELU>() && big_act<ACT_SIREN>();
}

}  // namespace ffno
