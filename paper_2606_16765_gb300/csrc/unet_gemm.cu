// unet_gemm.cu -- the U-Net's 3x3x3 convolutions on the fifth-generation
// tensor cores (tcgen05.mma, kind::f16, BF16 operands, FP32 accumulators in
// tensor memory), fed by tensor-map copies (cp.async.bulk.tensor).
//
// Forward and input gradient: an implicit GEMM with M = 128 output cells (a
// box of the channel-last activation: bx x by x bz cells x bb samples), N =
// output channels (<= 256 per tile) and K = 27 taps x input channels.  For
// tap (dz, dy, dx) the A tile is the same box shifted by (dz-1, dy-1, dx-1):
// one 5-D tensor-map copy whose out-of-range cells arrive as zeros, which is
// the convolution's zero padding.  The B tile is the tap's [N][K-chunk] slice
// of the weights.  Both operands are K-major, 64 channels per 128-byte
// swizzled row (or 32 channels per 64-byte row when the channel count is not a
// multiple of 64).  The input gradient is the same product with the weights
// transposed and the taps reversed.
//
// Where the input has 32 or 64 channels on a large grid, those 27 shifted
// copies are what the kernel waits for (8 KB of cells for two products): the
// halo kernel below keeps a block of cells with its halo in shared memory
// instead and takes every tap's operand from it.
//
// Weight gradient: G[(tap, i)][o] = sum over cells of X[cell + tap - 1][i] *
// GZ[cell][o]: M = 128 (tap, input-channel) rows taken as four 32-channel
// atoms, N = output channels, K = cells.  Here both operands are MN-major: the
// same channel-last boxes, rows of 32 or 64 channels, consecutive cells
// the contraction index.  The cell range is split over CTAs, each adding its
// FP32 tile into G atomically.
//
// A persistent CTA of six warps: warp 0 issues the copies into a ring of
// stages, warp 1 (after allocating tensor memory) issues the MMAs and commits
// each stage back to the producer, warps 2-5 read the accumulator (two
// accumulators alternate, so the epilogue of one tile overlaps the products of
// the next) and write the outputs.  Every mbarrier wait is bounded (about a
// second): on expiry the CTA records a status code, every role stops, the
// copies in flight and the issued products are waited for (bounded again),
// tensor memory is freed and the kernel returns.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "unet_gemm.h"

namespace unet {
namespace {

constexpr int NT = 192;                                // six warps
constexpr long long WAIT_CYCLES = 2000000000LL;        // about a second at the SM clock
constexpr size_t SMEM_MAX = 232448;                    // 227 KB
constexpr size_t SMEM_ONE_CTA = 120 * 1024;            // at least this much: one CTA per SM

__device__ __forceinline__ uint32_t saddr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Operands arrive by copies that complete on the barrier (or are fenced by
// their writers), so the issuing thread needs no tensor-core fence per stage;
// the accumulators' barriers keep theirs.
//
// Wait for the phase of parity `parity`; false after WAIT_CYCLES or, when
// `abort` is given, as soon as another role has set it.
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, volatile int *abort)
{
    if (mbar_try(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try(bar, parity)) {
        if (abort && *abort) return false;
        if (clock64() - t0 > WAIT_CYCLES) return false;
    }
    return true;
}

__device__ __forceinline__ void fail(volatile int *abort, int *status, int code)
{
    *abort = 1;
    atomicCAS(status, 0, code);
}

__device__ __forceinline__ void tma5(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, int c3, int c4,
                                     uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, "
        "%6}], [%7];\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void tma3(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
        : "memory");
}

// Shared-memory matrix descriptor, K-major, swizzled rows of `row_bytes`
// (128: swizzle mode 2; 64: mode 4); 8-row atoms row_bytes * 8 apart (stride
// field), leading field unused by these layouts, version 1 (bit 46).
__device__ __forceinline__ uint64_t desc_k(uint32_t addr, uint32_t row_bytes)
{
    const uint64_t mode = row_bytes == 128 ? 2 : 4;
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)((row_bytes * 8) >> 4) << 32) |
           ((uint64_t)1 << 46) | (mode << 61);
}

// MN-major, rows of W channels: atoms of W MN elements x 8 K rows with the 64-
// or 128-byte swizzle (W = 32, 64); `lbo` bytes between atoms along MN (leading
// field), an atom's 16 W bytes between 8-row groups along K (stride field).
template <int W>
__device__ __forceinline__ uint64_t desc_mn(uint32_t addr, uint32_t lbo)
{
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)W << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)(W == 64 ? 2 : 4) << 61);
}

// One lane of a full warp.  The issuing loops run inside `if (elect_one())`:
// there the compiler knows that a single thread runs and moves descriptors and
// addresses straight to uniform registers (at most 60 cycles per product; 65
// is what N = 128 takes in the tensor cores), while a lane == 0 branch costs a
// loop over the active lanes around every instruction, 143 cycles per product
// whatever its size.
__device__ __forceinline__ bool elect_one()
{
    uint32_t one = 0;
    asm volatile(
        "{\n\t.reg .b32 r;\n\t.reg .pred p;\n\t"
        "elect.sync r|p, 0xffffffff;\n\t"
        "@p mov.b32 %0, 1;\n\t}\n"
        : "+r"(one));
    return one != 0;
}

__device__ __forceinline__ void umma(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}

// The same with the descriptors' halves apart (only the low ones change).
template <bool ACC>
__device__ __forceinline__ void umma_lo(uint32_t tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                        uint32_t idesc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "mov.b64 da, {%1, %2};\n\tmov.b64 db, {%3, %4};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n\t}\n" ::"r"(tmem),
        "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "n"(ACC ? 1 : 0)
        : "memory");
}

// One tap of a halo block: NT tiles x CK / 16 products, all
// unrolled so that only the A address is formed per product (the tensor cores
// take 32 + N / 4 cycles each, 40 at N = 32; a rolled loop issues one per 90).
template <int NT, int CK, bool FIRST>
__device__ __forceinline__ void halo_tap(const uint32_t *d, const uint32_t *off, uint32_t a_lo, uint32_t a_hi,
                                         uint32_t kstep, uint32_t b_lo, uint32_t b_hi, uint32_t idesc)
{
#pragma unroll
    for (int t = 0; t < NT; ++t) {
        umma_lo<!FIRST>(d[t], a_lo + off[t], a_hi, b_lo, b_hi, idesc);
#pragma unroll
        for (int k = 1; k < CK / 16; ++k) umma_lo<true>(d[t], a_lo + off[t] + k * kstep, a_hi, b_lo + 2 * k, b_hi, idesc);
    }
}

__device__ __forceinline__ void commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar)
                 : "memory");
}

// a value every lane holds, marked as the same for the whole warp
__device__ __forceinline__ uint32_t uniform(uint32_t v) { return __shfl_sync(0xffffffffu, v, 0); }

__device__ __forceinline__ void tc_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tc_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }

__device__ __forceinline__ void tmem_ld16(uint32_t addr, float *v)
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = __uint_as_float(r[k]);
}

__device__ __forceinline__ void store16(float *dst, const float *v)
{
    float4 *d = reinterpret_cast<float4 *>(dst);
#pragma unroll
    for (int q = 0; q < 4; ++q) d[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
}

__device__ __forceinline__ void store16(__nv_bfloat16 *dst, const float *v)
{
    uint32_t w[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
        w[q] = *reinterpret_cast<const uint32_t *>(&h);
    }
    uint4 *d = reinterpret_cast<uint4 *>(dst);
    d[0] = make_uint4(w[0], w[1], w[2], w[3]);
    d[1] = make_uint4(w[4], w[5], w[6], w[7]);
}

// Position in a ring of S stages: the stage and the parity of its round (kept
// by counting: a division by S takes the issuing thread longer than a product).
struct Ring {
    uint32_t s = 0, round = 0;
    __device__ __forceinline__ void next(int S)
    {
        if (++s == (uint32_t)S) {
            s = 0;
            round ^= 1;
        }
    }
};

struct Box {
    int x0, y0, z0, b0;
};

__device__ __forceinline__ Box box_origin(int64_t mt, int tx, int ty, int tz, int bx, int by, int bz, int bb)
{
    Box o;
    o.x0 = (int)(mt % tx) * bx;
    mt /= tx;
    o.y0 = (int)(mt % ty) * by;
    mt /= ty;
    o.z0 = (int)(mt % tz) * bz;
    o.b0 = (int)(mt / tz) * bb;
    return o;
}

// Shared memory after the 1024-aligned operand ring: barriers, the tensor
// memory address, the abort flag.
struct Ctl {
    uint64_t *full, *empty, *accf, *acce, *drain;
    uint32_t *tslot;
    volatile int *abort;
};

__device__ __forceinline__ Ctl ctl_at(unsigned char *p, int S)
{
    Ctl c;
    uint64_t *b = reinterpret_cast<uint64_t *>(p);
    c.full = b;
    c.empty = b + S;
    c.accf = b + 2 * S;
    c.acce = b + 2 * S + 2;
    c.drain = b + 2 * S + 4;
    c.tslot = reinterpret_cast<uint32_t *>(b + 2 * S + 5);
    c.abort = reinterpret_cast<volatile int *>(c.tslot + 1);
    return c;
}

__device__ __forceinline__ void ctl_init(const Ctl &c, int S, uint32_t tmem_cols)
{
    const int warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(saddr(&c.full[s]), 1);
            mbar_init(saddr(&c.empty[s]), 1);
        }
        for (int q = 0; q < 2; ++q) {
            mbar_init(saddr(&c.accf[q]), 1);
            mbar_init(saddr(&c.acce[q]), 128);
        }
        mbar_init(saddr(c.drain), 1);
        *c.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(saddr(c.tslot)),
                     "r"(tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    tc_before();
    __syncthreads();
    tc_after();
}

__device__ __forceinline__ void ctl_finish(const Ctl &c, uint32_t tmem, uint32_t tmem_cols)
{
    tc_before();
    __syncthreads();
    tc_after();
    if ((threadIdx.x >> 5) == 1) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(tmem_cols) : "memory");
    }
}

// The producer's copies still in flight must land before the CTA exits.
__device__ __forceinline__ void drain_loads(const Ctl &c, uint32_t issued, int S, int *status)
{
    for (uint32_t j = issued > (uint32_t)S ? issued - S : 0; j < issued; ++j)
        if (!wait_bar(saddr(&c.full[j % S]), (j / S) & 1, nullptr)) atomicCAS(status, 0, 3);
}

// Every product issued must complete before tensor memory is freed.
__device__ __forceinline__ void drain_mma(const Ctl &c, int *status)
{
    commit(saddr(c.drain));
    if (!wait_bar(saddr(c.drain), 0, nullptr)) atomicCAS(status, 0, 4);
}

// ---------------------------------------------------------------------------
// forward / input-gradient convolution
// ---------------------------------------------------------------------------
template <int CK, class TO>
__global__ void __launch_bounds__(NT, 1) k_conv_umma(const __grid_constant__ CUtensorMap amap,
                                                     const __grid_constant__ CUtensorMap wmap, const ConvArgs a,
                                                     TO *__restrict__ out, int *status)
{
    extern __shared__ unsigned char raw[];
    unsigned char *sm = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~uintptr_t(1023));
    const int S = a.stages;
    unsigned char *sA = sm;
    unsigned char *sB = sm + (size_t)S * a.a_bytes;
    const Ctl c = ctl_at(sB + (size_t)S * a.b_bytes, S);
    const int warp = (int)uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    ctl_init(c, S, a.tmem_cols);
    const uint32_t tmem = uniform(*c.tslot);
    const int nk = a.ntaps * a.kchunks;
    // work item: (cell tile, channel tile, slice of the taps and chunks)
    auto q_of = [&](int sp) { return nk * sp / a.ksplit; };

    if (warp == 0) {
        if (elect_one()) {
            uint32_t it = 0;
            Ring r;
            bool ok = true;
            for (int64_t w = blockIdx.x; ok && w < a.nwork; w += gridDim.x) {
                const int sp = (int)(w % a.ksplit);
                const int64_t wt = w / a.ksplit;
                const Box o = box_origin(wt / a.nntiles, a.tx, a.ty, a.tz, a.bx, a.by, a.bz, a.bb);
                const int n0 = (int)(wt % a.nntiles) * a.ntile, q0 = q_of(sp), q1 = q_of(sp + 1);
                for (int q = q0, tap = q0 / a.kchunks, kc = q0 % a.kchunks; q < q1; ++q) {
                    const int dz = a.ntaps == 1 ? 1 : tap / 9, dy = a.ntaps == 1 ? 1 : (tap / 3) % 3,
                              dx = a.ntaps == 1 ? 1 : tap % 3;
                    const uint32_t s = r.s;
                    if (!wait_bar(saddr(&c.empty[s]), r.round ^ 1, c.abort)) {
                        fail(c.abort, status, 1);
                        ok = false;
                        break;
                    }
                    const uint32_t fb = saddr(&c.full[s]);
                    mbar_expect_tx(fb, a.a_bytes + a.b_bytes);
                    tma5(saddr(sA + (size_t)s * a.a_bytes), &amap, kc * CK, o.x0 + dx - 1, o.y0 + dy - 1,
                         o.z0 + dz - 1, o.b0, fb);
                    tma3(saddr(sB + (size_t)s * a.b_bytes), &wmap, kc * CK, n0, tap, fb);
                    ++it;
                    r.next(S);
                    if (++kc == a.kchunks) {
                        kc = 0;
                        ++tap;
                    }
                }
            }
            drain_loads(c, it, S, status);
        }
    } else if (warp == 1) {
        if (elect_one()) {
            uint32_t tc = 0;
            Ring r;
            bool ok = true;
            for (int64_t w = blockIdx.x; ok && w < a.nwork; w += gridDim.x, ++tc) {
                const uint32_t acc = tc & 1;
                if (!wait_bar(saddr(&c.acce[acc]), ((tc >> 1) & 1) ^ 1, c.abort)) {
                    fail(c.abort, status, 2);
                    break;
                }
                tc_after();
                const uint32_t d = tmem + acc * (uint32_t)a.ntile;
                const int sp = (int)(w % a.ksplit), q0 = q_of(sp), q1 = q_of(sp + 1);
                for (int q = q0; q < q1; ++q, r.next(S)) {
                    const uint32_t s = r.s;
                    if (!wait_bar(saddr(&c.full[s]), r.round, c.abort)) {
                        fail(c.abort, status, 2);
                        ok = false;
                        break;
                    }
                    const uint64_t ad = desc_k(saddr(sA + (size_t)s * a.a_bytes), CK * 2);
                    const uint64_t bd = desc_k(saddr(sB + (size_t)s * a.b_bytes), CK * 2);
#pragma unroll
                    for (int k = 0; k < CK / 16; ++k)          // K = 16 per product: 32 bytes along the row
                        umma(d, ad + 2 * k, bd + 2 * k, a.idesc, (q > q0 || k > 0) ? 1u : 0u);
                    commit(saddr(&c.empty[s]));
                }
                if (ok) commit(saddr(&c.accf[acc]));
            }
            drain_mma(c, status);
        }
        __syncwarp();
    } else {
        const int quad = warp & 3;                 // tensor-memory lanes 32 quad .. 32 quad + 31
        const int row = quad * 32 + lane;
        const int rx = row % a.bx, ry = (row / a.bx) % a.by, rz = (row / (a.bx * a.by)) % a.bz,
                  rb = row / (a.bx * a.by * a.bz);
        uint32_t tc = 0;
        for (int64_t w = blockIdx.x; w < a.nwork; w += gridDim.x, ++tc) {
            const uint32_t acc = tc & 1;
            if (!wait_bar(saddr(&c.accf[acc]), (tc >> 1) & 1, c.abort)) {
                fail(c.abort, status, 5);
                break;
            }
            tc_after();
            const int64_t wt = w / a.ksplit;
            const Box o = box_origin(wt / a.nntiles, a.tx, a.ty, a.tz, a.bx, a.by, a.bz, a.bb);
            const int n0 = (int)(wt % a.nntiles) * a.ntile;
            const int b = o.b0 + rb;
            const bool valid = b < a.B;
            TO *dst = out + (w % a.ksplit) * a.split_stride + ((((int64_t)(valid ? b : 0) * a.Z + o.z0 + rz) * a.Y + o.y0 + ry) * a.X + o.x0 + rx) * a.ldo +
                      a.ooff + n0;
            const uint32_t base = tmem + ((uint32_t)(quad * 32) << 16) + acc * (uint32_t)a.ntile;
            for (int cc = 0; cc < a.ntile; cc += 16) {
                float v[16];
                tmem_ld16(base + cc, v);
                if (valid) store16(dst + cc, v);
            }
            tc_before();
            mbar_arrive(saddr(&c.acce[acc]));
        }
    }
    ctl_finish(c, tmem, a.tmem_cols);
}

// ---------------------------------------------------------------------------
// forward / input-gradient convolution from a halo block
// ---------------------------------------------------------------------------
// A block of bz x sy rows of X cells with its halo lies in shared memory as
// [8-channel group][plane][row][P = X + 2 cells][16 bytes]: the unswizzled
// K-major operand layout whose 8-row groups are 128 bytes apart, so that any
// run of 128 cells is an A tile and a tap is an offset of the start address
// by whole cells (16 bytes).  A plane's rows are one run of sy P cells cut
// into tiles of 128 (one row each where X = 128); the two cells between rows
// give results that are not stored.  Each input cell is fetched
// (bz + 2)(sy + 2) / (bz sy) times instead of 27, and a tap's weights serve
// all the block's tiles.  The products of an output are added in the order of
// the kernel above (tap, channel chunk, 16 channels): the same bits.
// Ten warps: four fetch the block (16-byte copies, zeros outside the grid),
// one the weights (tensor map, a ring of stages), one issues, four store.  A
// plane is handed back as soon as no later tap reads it.
constexpr int HT = 320;

struct HCtl {
    uint64_t *afull, *aempty, *full, *empty, *accf, *acce, *drain;
    uint32_t *tslot;
    volatile int *abort;
};

constexpr int HPL = 6;                       // most planes of a block (bz + 2)

__device__ __forceinline__ HCtl hctl_at(unsigned char *p, int S)
{
    HCtl c;
    uint64_t *b = reinterpret_cast<uint64_t *>(p);
    c.afull = b;
    c.aempty = b + HPL;
    c.accf = b + 2 * HPL;
    c.acce = b + 2 * HPL + 2;
    c.drain = b + 2 * HPL + 4;
    c.full = b + 2 * HPL + 5;
    c.empty = c.full + S;
    c.tslot = reinterpret_cast<uint32_t *>(c.empty + S);
    c.abort = reinterpret_cast<volatile int *>(c.tslot + 1);
    return c;
}

// unswizzled K-major: `lbo` bytes between 8-channel groups, 128 between 8-row groups
__device__ __forceinline__ uint64_t desc_plain(uint32_t addr, uint32_t lbo)
{
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(128 >> 4) << 32) |
           ((uint64_t)1 << 46);
}

struct HItem {
    int b, z0, y0, n0;
};

__device__ __forceinline__ HItem hitem(const HaloArgs &a, int64_t w)
{
    HItem it;
    it.n0 = (int)(w % a.nntiles) * a.ntile;
    w /= a.nntiles;
    it.y0 = (int)(w % a.ty) * a.sy;
    w /= a.ty;
    it.z0 = (int)(w % a.tz) * a.bz;
    it.b = (int)(w / a.tz);
    return it;
}

constexpr int HALO_TILES = 8;                // most tiles of a block

// The issuing thread's loop over its blocks.
template <int NT, int CK>
__device__ __forceinline__ void halo_issue(const HaloArgs &a, const HCtl &c, unsigned char *sA, unsigned char *sB,
                                           uint32_t tmem, int *status)
{
    const int S = a.stages, planes = a.bz + 2, rows = a.sy + 2, P = a.X + 2;
    const uint64_t a0 = desc_plain(saddr(sA), a.lbo);
    const uint32_t kstep = a.lbo >> 3;                     // two 8-channel groups, in 16 bytes
    const uint32_t a_lo = (uint32_t)a0, a_hi = (uint32_t)(a0 >> 32);
    uint32_t off[NT];
#pragma unroll
    for (int t = 0; t < NT; ++t) off[t] = (uint32_t)((t / a.ptiles) * rows * P + (t % a.ptiles) * a.tstep);
    uint32_t n = 0;
    Ring r;
    for (int64_t w = blockIdx.x; w < a.nwork; w += gridDim.x, ++n) {
        const uint32_t set = a.sets == 2 ? n & 1 : 0, use = a.sets == 2 ? n >> 1 : n;
        if (!wait_bar(saddr(&c.acce[set]), (use & 1) ^ 1, c.abort)) {
            fail(c.abort, status, 2);
            return;
        }
        tc_after();
        uint32_t d[NT];
#pragma unroll
        for (int t = 0; t < NT; ++t) d[t] = tmem + (set * NT + t) * (uint32_t)a.ntile;
        int have = 0;                                      // planes that have arrived
        for (int dz = 0; dz < 3; ++dz) {
            for (; have < dz + a.bz; ++have)
                if (!wait_bar(saddr(&c.afull[have]), n & 1, c.abort)) {
                    fail(c.abort, status, 7);
                    return;
                }
            for (int yx = 0; yx < 9; yx += a.tps, r.next(S)) {
                if (!wait_bar(saddr(&c.full[r.s]), r.round, c.abort)) {
                    fail(c.abort, status, 2);
                    return;
                }
                const uint64_t bd = desc_k(saddr(sB + (size_t)r.s * a.b_bytes), CK * 2);
                const uint32_t b_hi = (uint32_t)(bd >> 32);
                uint32_t b_lo = (uint32_t)bd;
                for (int j = yx; j < yx + a.tps; ++j, b_lo += a.tap_bytes >> 4) {
                    const uint32_t al = a_lo + (uint32_t)((dz * rows + j / 3) * P + j % 3);
                    if (dz + j == 0) halo_tap<NT, CK, true>(d, off, al, a_hi, kstep, b_lo, b_hi, a.idesc);
                    else halo_tap<NT, CK, false>(d, off, al, a_hi, kstep, b_lo, b_hi, a.idesc);
                }
                commit(saddr(&c.empty[r.s]));
            }
            // planes 0 and 1 have no reader after the taps of dz = 0 and 1
            if (dz < 2) commit(saddr(&c.aempty[dz]));
        }
        for (int p = 2; p < planes; ++p) commit(saddr(&c.aempty[p]));
        commit(saddr(&c.accf[set]));
    }
}

template <int CK, class TO>
__global__ void __launch_bounds__(HT, 1) k_conv_halo(const __nv_bfloat16 *__restrict__ x,
                                                     const __grid_constant__ CUtensorMap wmap, const HaloArgs a,
                                                     TO *__restrict__ out, int *status)
{
    extern __shared__ unsigned char raw[];
    unsigned char *sm = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~uintptr_t(1023));
    const int S = a.stages;
    unsigned char *sB = sm, *sA = sm + (size_t)S * a.b_bytes;
    const HCtl c = hctl_at(sA + a.a_bytes, S);
    const int warp = (int)uniform(threadIdx.x >> 5), lane = threadIdx.x & 31, planes = a.bz + 2;
    if (threadIdx.x == 0) {
        for (int p = 0; p < planes; ++p) {
            mbar_init(saddr(&c.afull[p]), 128);
            mbar_init(saddr(&c.aempty[p]), 1);
        }
        for (int s = 0; s < S; ++s) {
            mbar_init(saddr(&c.full[s]), 1);
            mbar_init(saddr(&c.empty[s]), 1);
        }
        for (int q = 0; q < 2; ++q) {
            mbar_init(saddr(&c.accf[q]), 1);
            mbar_init(saddr(&c.acce[q]), 128);
        }
        mbar_init(saddr(c.drain), 1);
        *c.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 5) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(saddr(c.tslot)),
                     "r"(a.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    // zeros once: the cells beside every row stay zero
    for (uint32_t q = threadIdx.x; q < a.a_bytes / 16; q += HT) reinterpret_cast<uint4 *>(sA)[q] = make_uint4(0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    tc_before();
    __syncthreads();
    tc_after();
    const uint32_t tmem = uniform(*c.tslot);
    const int rows = a.sy + 2, P = a.X + 2;

    if (warp < 4) {
        // 16 bytes (8 channels of a cell) per copy; a plane's copies are in
        // flight while the next plane's are issued
        constexpr int G = CK / 8, STEP = 128 / G;
        const int g = (int)threadIdx.x & (G - 1), cell0 = (int)threadIdx.x / G;
        uint32_t n = 0;
        int pending = -1;
        bool ok = true;
        auto arrive = [&]() {
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            mbar_arrive(saddr(&c.afull[pending]));
            pending = -1;
        };
        for (int64_t w = blockIdx.x; ok && w < a.nwork; w += gridDim.x, ++n) {
            const HItem it = hitem(a, w);
            for (int p = 0; p < planes; ++p) {
                const uint32_t ready = saddr(&c.aempty[p]), parity = (n & 1) ^ 1;
                if (pending >= 0 && !mbar_try(ready, parity)) {
                    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
                    arrive();
                }
                if (!wait_bar(ready, parity, c.abort)) {
                    fail(c.abort, status, 6);
                    ok = false;
                    break;
                }
                const int z = it.z0 + p - 1;
                for (int r = 0; r < rows; ++r) {
                    const int y = it.y0 + r - 1;
                    const bool in = z >= 0 && z < a.Z && y >= 0 && y < a.Y;
                    const __nv_bfloat16 *src =
                        x + ((((int64_t)it.b * a.Z + (in ? z : 0)) * a.Y + (in ? y : 0)) * a.X + cell0) * CK + g * 8;
                    const uint32_t dst = saddr(sA) + (uint32_t)(((p * rows + r) * P + 1 + cell0) * 16) + g * a.lbo;
                    const uint32_t bytes = in ? 16 : 0;
#pragma unroll 4
                    for (int i = 0; i < a.X - cell0; i += STEP)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst + i * 16),
                                     "l"(src + i * CK), "r"(bytes)
                                     : "memory");
                }
                asm volatile("cp.async.commit_group;\n" ::: "memory");
                if (pending >= 0) {
                    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
                    arrive();
                }
                pending = p;
            }
        }
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        if (pending >= 0) arrive();
    } else if (warp == 4) {
        if (elect_one()) {
            uint32_t it = 0;
            Ring r;
            bool ok = true;
            for (int64_t w = blockIdx.x; ok && w < a.nwork; w += gridDim.x) {
                const int n0 = hitem(a, w).n0;
                for (int tap = 0; tap < 27; tap += a.tps, r.next(S)) {
                    if (!wait_bar(saddr(&c.empty[r.s]), r.round ^ 1, c.abort)) {
                        fail(c.abort, status, 1);
                        ok = false;
                        break;
                    }
                    const uint32_t fb = saddr(&c.full[r.s]);
                    mbar_expect_tx(fb, a.b_bytes);
                    tma3(saddr(sB + (size_t)r.s * a.b_bytes), &wmap, 0, n0, tap, fb);
                    ++it;
                }
            }
            for (uint32_t j = it > (uint32_t)S ? it - S : 0; j < it; ++j)
                if (!wait_bar(saddr(&c.full[j % S]), (j / S) & 1, nullptr)) atomicCAS(status, 0, 3);
        }
    } else if (warp == 5) {
        if (elect_one()) {
            switch (a.ntiles) {
            case 1: halo_issue<1, CK>(a, c, sA, sB, tmem, status); break;
            case 2: halo_issue<2, CK>(a, c, sA, sB, tmem, status); break;
            case 3: halo_issue<3, CK>(a, c, sA, sB, tmem, status); break;
            case 4: halo_issue<4, CK>(a, c, sA, sB, tmem, status); break;
            case 5: halo_issue<5, CK>(a, c, sA, sB, tmem, status); break;
            case 6: halo_issue<6, CK>(a, c, sA, sB, tmem, status); break;
            case 7: halo_issue<7, CK>(a, c, sA, sB, tmem, status); break;
            default: halo_issue<8, CK>(a, c, sA, sB, tmem, status); break;
            }
            commit(saddr(c.drain));
            if (!wait_bar(saddr(c.drain), 0, nullptr)) atomicCAS(status, 0, 4);
        }
        __syncwarp();
    } else {
        const int quad = warp & 3, row = quad * 32 + lane;
        uint32_t n = 0;
        for (int64_t w = blockIdx.x; w < a.nwork; w += gridDim.x, ++n) {
            const uint32_t set = a.sets == 2 ? n & 1 : 0, use = a.sets == 2 ? n >> 1 : n;
            if (!wait_bar(saddr(&c.accf[set]), use & 1, c.abort)) {
                fail(c.abort, status, 5);
                break;
            }
            tc_after();
            const HItem it = hitem(a, w);
            const uint32_t base = tmem + ((uint32_t)(quad * 32) << 16) + set * (uint32_t)(a.ntiles * a.ntile);
            for (int t = 0; t < a.ntiles; ++t) {
                const int zo = t / a.ptiles, j = (t % a.ptiles) * a.tstep + row, ry = j / P, rx = j - ry * P;
                const int z = it.z0 + zo, y = it.y0 + ry;
                const bool valid = rx < a.X && ry < a.sy && z < a.Z && y < a.Y;
                TO *dst = out + ((((int64_t)it.b * a.Z + (valid ? z : 0)) * a.Y + (valid ? y : 0)) * a.X + (valid ? rx : 0)) * a.ldo +
                          a.ooff + it.n0;
                for (int cc = 0; cc < a.ntile; cc += 16) {
                    float v[16];
                    tmem_ld16(base + (uint32_t)(t * a.ntile + cc), v);
                    if (valid) store16(dst + cc, v);
                }
            }
            tc_before();
            mbar_arrive(saddr(&c.acce[set]));
        }
    }
    tc_before();
    __syncthreads();
    tc_after();
    if (warp == 5) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(a.tmem_cols) : "memory");
    }
}

// ---------------------------------------------------------------------------
// weight gradient
// ---------------------------------------------------------------------------
struct WItem {
    int mt, nt;
    int64_t c0, c1;
};

__device__ __forceinline__ WItem witem(const WgradArgs &a, int64_t w)
{
    WItem it;
    const int ks = (int)(w % a.ksplit);
    const int64_t r = w / a.ksplit;
    it.nt = (int)(r % a.nntiles);
    it.mt = (int)(r / a.nntiles);
    it.c0 = a.nchunks * ks / a.ksplit;
    it.c1 = a.nchunks * (ks + 1) / a.ksplit;
    return it;
}

// W: channels per copied row.  The copies go at a row every 4 to 6 cycles
// whether it has 64 or 128 bytes, and the kernel waits for them, so channel
// counts that are multiples of 64 take 128-byte rows (64 -> 64 channels at
// 64x32x32, batch 8: 461 against 394 us).
template <int W>
__global__ void __launch_bounds__(NT, 1) k_wgrad_umma(const __grid_constant__ CUtensorMap xmap,
                                                      const __grid_constant__ CUtensorMap gmap, const WgradArgs a,
                                                      float *__restrict__ g, int *status)
{
    extern __shared__ unsigned char raw[];
    unsigned char *sm = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~uintptr_t(1023));
    const int S = a.stages;
    unsigned char *sA = sm;
    unsigned char *sB = sm + (size_t)S * a.a_bytes;
    const Ctl c = ctl_at(sB + (size_t)S * a.b_bytes, S);
    const int warp = (int)uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    ctl_init(c, S, a.tmem_cols);
    const uint32_t tmem = uniform(*c.tslot);
    constexpr uint32_t ATOM = 128 * W * 2;         // 128 cells x W channels

    if (warp == 0) {
        if (elect_one()) {
            uint32_t it = 0;
            Ring r;
            bool ok = true;
            for (int64_t w = blockIdx.x; ok && w < a.nwork; w += gridDim.x) {
                const WItem wi = witem(a, w);
                for (int64_t ch = wi.c0; ch < wi.c1; ++ch) {
                    const Box o = box_origin(ch, a.tx, a.ty, a.tz, a.bx, a.by, a.bz, a.bb);
                    const uint32_t s = r.s;
                    if (!wait_bar(saddr(&c.empty[s]), r.round ^ 1, c.abort)) {
                        fail(c.abort, status, 1);
                        ok = false;
                        break;
                    }
                    const uint32_t fb = saddr(&c.full[s]);
                    mbar_expect_tx(fb, a.a_bytes + a.b_bytes);
                    for (int at = 0; at < 128 / W; ++at) {
                        const int ga = wi.mt * (128 / W) + at;
                        // rows past 27 * cin load a valid tap and are discarded
                        const int tap = min(ga / a.cin_blocks, 26), cb = ga / a.cin_blocks > 26 ? 0 : ga % a.cin_blocks;
                        const int dz = tap / 9, dy = (tap / 3) % 3, dx = tap % 3;
                        tma5(saddr(sA + (size_t)s * a.a_bytes + at * ATOM), &xmap, cb * W, o.x0 + dx - 1,
                             o.y0 + dy - 1, o.z0 + dz - 1, o.b0, fb);
                    }
                    for (int j = 0; j < a.ntile / W; ++j)
                        tma5(saddr(sB + (size_t)s * a.b_bytes + j * ATOM), &gmap, wi.nt * a.ntile + j * W, o.x0, o.y0,
                             o.z0, o.b0, fb);
                    ++it;
                    r.next(S);
                }
            }
            drain_loads(c, it, S, status);
        }
    } else if (warp == 1) {
        if (elect_one()) {
            uint32_t tc = 0;
            Ring r;
            bool ok = true;
            for (int64_t w = blockIdx.x; ok && w < a.nwork; w += gridDim.x) {
                const WItem wi = witem(a, w);
                if (wi.c1 <= wi.c0) continue;
                const uint32_t acc = tc & 1;
                if (!wait_bar(saddr(&c.acce[acc]), ((tc >> 1) & 1) ^ 1, c.abort)) {
                    fail(c.abort, status, 2);
                    break;
                }
                tc_after();
                const uint32_t d = tmem + acc * (uint32_t)a.ntile;
                for (int64_t ch = wi.c0; ch < wi.c1; ++ch, r.next(S)) {
                    const uint32_t s = r.s;
                    if (!wait_bar(saddr(&c.full[s]), r.round, c.abort)) {
                        fail(c.abort, status, 2);
                        ok = false;
                        break;
                    }
                    const uint64_t ad = desc_mn<W>(saddr(sA + (size_t)s * a.a_bytes), ATOM),
                                   bd = desc_mn<W>(saddr(sB + (size_t)s * a.b_bytes), ATOM);
#pragma unroll
                    for (int k = 0; k < 8; ++k)                // 16 cells (two 8-row groups) per product
                        umma(d, ad + 2 * W * k, bd + 2 * W * k, a.idesc, (ch > wi.c0 || k > 0) ? 1u : 0u);
                    commit(saddr(&c.empty[s]));
                }
                if (ok) commit(saddr(&c.accf[acc]));
                ++tc;
            }
            drain_mma(c, status);
        }
        __syncwarp();
    } else {
        const int quad = warp & 3;
        const int row = quad * 32 + lane;
        uint32_t tc = 0;
        for (int64_t w = blockIdx.x; w < a.nwork; w += gridDim.x) {
            const WItem wi = witem(a, w);
            if (wi.c1 <= wi.c0) continue;
            const uint32_t acc = tc & 1;
            if (!wait_bar(saddr(&c.accf[acc]), (tc >> 1) & 1, c.abort)) {
                fail(c.abort, status, 5);
                break;
            }
            tc_after();
            const int m = wi.mt * 128 + row;
            float *dst = g + (int64_t)(m < a.m_total ? m : 0) * a.ldg + wi.nt * a.ntile;
            const uint32_t base = tmem + ((uint32_t)(quad * 32) << 16) + acc * (uint32_t)a.ntile;
            for (int cc = 0; cc < a.ntile; cc += 16) {
                float v[16];
                tmem_ld16(base + cc, v);
                if (m < a.m_total) {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        atomicAdd(reinterpret_cast<float4 *>(dst + cc) + q,
                                  make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]));
                }
            }
            tc_before();
            mbar_arrive(saddr(&c.acce[acc]));
            ++tc;
        }
    }
    ctl_finish(c, tmem, a.tmem_cols);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        cudaDriverEntryPointQueryResult q;
        void *p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        else
            cudaGetLastError();
    }
    return fn;
}

bool encode(unsigned char *dst, int rank, const void *base, const cuuint64_t *dims, const cuuint64_t *strides,
            const cuuint32_t *box, CUtensorMapSwizzle sw)
{
    static_assert(sizeof(CUtensorMap) == 128, "tensor map size");
    PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
    if (!fn || (reinterpret_cast<uintptr_t>(base) & 15u)) return false;
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    CUtensorMap m;
    const CUresult r = fn(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void *>(base), dims, strides, box,
                          estr, CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return false;
    std::memcpy(dst, &m, sizeof m);
    return true;
}

bool pow2(int v) { return v > 0 && (v & (v - 1)) == 0; }

// A tile of 128 cells: whole rows of x first, then rows of y, planes of z,
// samples (grids with power-of-two sides).
void box_for(int X, int Y, int Z, int &bx, int &by, int &bz, int &bb)
{
    bx = std::min(X, 128);
    by = std::min(Y, 128 / bx);
    bz = std::min(Z, 128 / (bx * by));
    bb = 128 / (bx * by * bz);
}

int pick_ntile(int N)
{
    for (int t = std::min(N, 256); t >= 32; t -= 32)
        if (N % t == 0) return t;
    return 0;
}

uint32_t tmem_cols_for(int ntile)
{
    uint32_t c = 32;
    while (c < 2u * (uint32_t)ntile) c <<= 1;
    return c;
}

// kind::f16 instruction descriptor: FP32 accumulator, BF16 A and B, M = 128.
uint32_t idesc_for(int ntile, bool a_mn, bool b_mn)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) |
           ((uint32_t)(ntile >> 3) << 17) | ((128u >> 4) << 24);
}

size_t ctl_bytes(int S) { return (size_t)(2 * S + 5) * 8 + 16; }

}  // namespace

static bool halo_plan(ConvPlan &p, const void *act, int lda, int k, int X, int Y, int Z, int B, const void *wt, int N, int sms);

bool conv_plan(ConvPlan &p, const void *act, int lda, int k, int X, int Y, int Z, int B, const void *w, int N,
               int ntaps, int ldo, int ooff, int sms, const char **err, bool split)
{
    auto bad = [&](const char *m) {
        if (err) *err = m;
        return false;
    };
    if (!pow2(X) || !pow2(Y) || !pow2(Z) || B < 1) return bad("conv: grid sides must be powers of two");
    if (k < 32 || k % 32 || lda < k || lda % 8) return bad("conv: input channels must be a multiple of 32");
    if (N < 32 || N % 32 || ooff % 16 || ldo % 8 || ldo < ooff + N) return bad("conv: output channels");
    if (ntaps != 1 && ntaps != 27) return bad("conv: taps must be 1 or 27");
    ConvArgs &a = p.a;
    std::memset(&a, 0, sizeof a);
    p.ck = (k % 64 == 0) ? 64 : 32;
    a.X = X; a.Y = Y; a.Z = Z; a.B = B;
    box_for(X, Y, Z, a.bx, a.by, a.bz, a.bb);
    a.tx = X / a.bx; a.ty = Y / a.by; a.tz = Z / a.bz; a.tb = (B + a.bb - 1) / a.bb;
    a.ntaps = ntaps;
    a.kchunks = k / p.ck;
    a.ntile = pick_ntile(N);
    const int64_t cell_tiles = (int64_t)a.tx * a.ty * a.tz * a.tb;
    const int nk = ntaps * a.kchunks;
    // A few cell tiles leave most SMs idle behind one long chain of products:
    // narrower channel tiles, and (where the caller adds the parts up) slices
    // of the taps and chunks, at least 8 of them each.  512 channels from 256
    // at 8x4x4, batch 2 (2 cell tiles): 44 us on 4 SMs, 9 x 16 items 8.9 us and
    // 3.7 us for the sum of the parts.
    a.ksplit = 1;
    if (split && cell_tiles * (N / a.ntile) * 2 <= sms) {
        while (a.ntile > 64 && a.ntile % 64 == 0 && cell_tiles * (N / a.ntile) * 8 < sms) a.ntile /= 2;
        a.ksplit = (int)std::max<int64_t>(1, std::min<int64_t>(nk / 8, sms / (cell_tiles * (N / a.ntile))));
    }
    a.split_stride = (int64_t)X * Y * Z * B * ldo;
    a.nntiles = N / a.ntile;
    a.ldo = ldo; a.ooff = ooff;
    a.a_bytes = 128u * p.ck * 2;
    a.b_bytes = (uint32_t)a.ntile * p.ck * 2;
    a.stages = (int)std::min<size_t>(8, (SMEM_MAX - 2048 - ctl_bytes(8)) / (a.a_bytes + a.b_bytes));
    if (a.stages < 2) return bad("conv: tile does not fit in shared memory");
    a.nwork = cell_tiles * a.nntiles * a.ksplit;
    a.idesc = idesc_for(a.ntile, false, false);
    a.tmem_cols = tmem_cols_for(a.ntile);
    p.smem = std::max(SMEM_ONE_CTA, 1024 + (size_t)a.stages * (a.a_bytes + a.b_bytes) + ctl_bytes(a.stages));
    p.grid = (int)std::min<int64_t>(a.nwork, std::max(1, sms));
    const CUtensorMapSwizzle sw = p.ck == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B;
    const cuuint64_t adims[5] = {(cuuint64_t)lda, (cuuint64_t)X, (cuuint64_t)Y, (cuuint64_t)Z, (cuuint64_t)B};
    const cuuint64_t astr[4] = {(cuuint64_t)lda * 2, (cuuint64_t)lda * 2 * X, (cuuint64_t)lda * 2 * X * Y,
                                (cuuint64_t)lda * 2 * X * Y * Z};
    const cuuint32_t abox[5] = {(cuuint32_t)p.ck, (cuuint32_t)a.bx, (cuuint32_t)a.by, (cuuint32_t)a.bz,
                                (cuuint32_t)a.bb};
    if (!encode(p.amap, 5, act, adims, astr, abox, sw)) return bad("conv: activation tensor map rejected");
    const cuuint64_t wdims[3] = {(cuuint64_t)k, (cuuint64_t)N, (cuuint64_t)ntaps};
    const cuuint64_t wstr[2] = {(cuuint64_t)k * 2, (cuuint64_t)k * 2 * N};
    const cuuint32_t wbox[3] = {(cuuint32_t)p.ck, (cuuint32_t)a.ntile, 1};
    if (!encode(p.wmap, 3, w, wdims, wstr, wbox, sw)) return bad("conv: weight tensor map rejected");
    p.halo = false;
    if (ntaps == 27 && a.ksplit == 1) halo_plan(p, act, lda, k, X, Y, Z, B, w, N, sms);
    return true;
}

// The halo kernel's block: rows and planes that need the fewest cycles per
// cell, from the products (an M = 128 tile reads its A rows at 128 bytes a
// cycle: 32 + N / 4 cycles, or N / 2 where the products themselves take
// longer) and the bytes fetched (about 50 a cycle on one SM, partly behind the
// products); taken where that is at most 0.8 of the shifted copies' cost (27
// taps of cells and weights at the 16.6 bytes a cycle and SM that all SMs
// together reach).  lda = k: the block's cells are whole runs of channels.
static bool halo_plan(ConvPlan &p, const void *act, int lda, int k, int X, int Y, int Z, int B, const void *wt, int N, int sms)
{
    if (lda != k || (k != 32 && k != 64) || X < 16 || X > 128 || (reinterpret_cast<uintptr_t>(act) & 15)) return false;
    const ConvArgs &o = p.a;
    HaloArgs best{};
    double best_cost = 1e300;
    const int P = X + 2;
    for (int bz = 1; bz <= std::min(4, Z); ++bz)
        for (int sy = 1; sy <= Y; ++sy) {
            HaloArgs a{};
            a.bz = bz;
            a.sy = sy;
            a.tstep = X == 128 ? P : 128;
            a.ptiles = X == 128 ? sy : (sy * P - 2 + 127) / 128;
            a.ntiles = bz * a.ptiles;
            if (a.ntiles * o.ntile > 512 || a.ntiles > HALO_TILES) continue;
            a.sets = 2 * a.ntiles * o.ntile <= 512 ? 2 : 1;
            const int cells = (bz + 2) * (sy + 2) * P + 130;           // and what the last tile reads past them
            a.lbo = (uint32_t)cells * 16;
            a.a_bytes = a.lbo * (uint32_t)(k / 8);
            a.tap_bytes = o.b_bytes;
            const size_t room = SMEM_MAX - 1024 - 512;
            a.tps = a.a_bytes + 9 * (size_t)a.tap_bytes <= room ? 3 : 1;     // taps per stage of weights
            a.b_bytes = (uint32_t)a.tps * a.tap_bytes;
            if (a.a_bytes + 3 * (size_t)a.b_bytes > room) continue;
            a.stages = (int)std::min<size_t>(8, (room - a.a_bytes) / a.b_bytes);
            a.ty = (Y + sy - 1) / sy;
            a.tz = (Z + bz - 1) / bz;
            a.nwork = (int64_t)B * a.tz * a.ty * o.nntiles;
            const double mma = (double)a.ntiles * 27 * (k / 16) * std::max(o.ntile / 2.0, 32.0 + o.ntile / 4.0);
            const double load = ((double)cells * k * 2 + 27.0 * k * o.ntile * 2) / 50.0;
            const double waves = std::ceil((double)a.nwork / std::max(1, sms));
            const double cost = waves * (mma + 0.6 * load);
            if (cost < best_cost) {
                best_cost = cost;
                best = a;
            }
        }
    const double copies = std::ceil((double)o.nwork / std::max(1, sms)) * 27.0 * (256.0 * k + 2.0 * o.ntile * k) / 16.6;
    if (best_cost > 0.8 * copies) return false;
    HaloArgs &h = p.h;
    h = best;
    h.X = X; h.Y = Y; h.Z = Z; h.B = B;
    h.C = k;
    h.ntile = o.ntile; h.nntiles = o.nntiles;
    h.ldo = o.ldo; h.ooff = o.ooff;
    h.idesc = o.idesc;
    h.tmem_cols = 32;
    while (h.tmem_cols < (uint32_t)(h.sets * h.ntiles * h.ntile)) h.tmem_cols <<= 1;
    const cuuint64_t wdims[3] = {(cuuint64_t)k, (cuuint64_t)N, 27};
    const cuuint64_t wstr[2] = {(cuuint64_t)k * 2, (cuuint64_t)k * 2 * N};
    const cuuint32_t wbox[3] = {(cuuint32_t)k, (cuuint32_t)h.ntile, (cuuint32_t)h.tps};
    if (!encode(p.wmap, 3, wt, wdims, wstr, wbox, k == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B)) return false;
    p.act = act;
    p.halo = true;
    p.smem = std::max(SMEM_ONE_CTA, 1024 + (size_t)h.stages * h.b_bytes + h.a_bytes + (size_t)(2 * HPL + 5 + 2 * h.stages) * 8 + 16);
    p.grid = (int)std::min<int64_t>(h.nwork, std::max(1, sms));
    return true;
}

template <int CK>
static void launch_halo(const ConvPlan &p, const CUtensorMap &wm, void *out, bool out_f32, int *status, cudaStream_t s)
{
    const __nv_bfloat16 *x = static_cast<const __nv_bfloat16 *>(p.act);
    if (out_f32) k_conv_halo<CK, float><<<p.grid, HT, p.smem, s>>>(x, wm, p.h, static_cast<float *>(out), status);
    else k_conv_halo<CK, __nv_bfloat16><<<p.grid, HT, p.smem, s>>>(x, wm, p.h, static_cast<__nv_bfloat16 *>(out), status);
}

// out = sum of the parts, in their order
__global__ void __launch_bounds__(256) k_sum_split(const float4 *__restrict__ part, int parts, int64_t n4,
                                                   float4 *__restrict__ out)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (int64_t)gridDim.x * blockDim.x) {
        float4 s = part[i];
        for (int p = 1; p < parts; ++p) {
            const float4 v = part[p * n4 + i];
            s.x += v.x;
            s.y += v.y;
            s.z += v.z;
            s.w += v.w;
        }
        out[i] = s;
    }
}

void conv_sum(const ConvPlan &p, const float *part, float *out, cudaStream_t s)
{
    const int64_t n4 = p.a.split_stride / 4;
    k_sum_split<<<(unsigned)std::min<int64_t>((n4 + 255) / 256, 2048), 256, 0, s>>>(
        reinterpret_cast<const float4 *>(part), p.a.ksplit, n4, reinterpret_cast<float4 *>(out));
}

void conv_launch(const ConvPlan &p, void *out, bool out_f32, int *status, cudaStream_t s)
{
    CUtensorMap am, wm;
    std::memcpy(&am, p.amap, sizeof am);
    std::memcpy(&wm, p.wmap, sizeof wm);
    if (p.halo) {
        if (p.ck == 64) launch_halo<64>(p, wm, out, out_f32, status, s);
        else launch_halo<32>(p, wm, out, out_f32, status, s);
        return;
    }
    if (p.ck == 64) {
        if (out_f32)
            k_conv_umma<64, float><<<p.grid, NT, p.smem, s>>>(am, wm, p.a, static_cast<float *>(out), status);
        else
            k_conv_umma<64, __nv_bfloat16><<<p.grid, NT, p.smem, s>>>(am, wm, p.a, static_cast<__nv_bfloat16 *>(out),
                                                                      status);
    } else {
        if (out_f32)
            k_conv_umma<32, float><<<p.grid, NT, p.smem, s>>>(am, wm, p.a, static_cast<float *>(out), status);
        else
            k_conv_umma<32, __nv_bfloat16><<<p.grid, NT, p.smem, s>>>(am, wm, p.a, static_cast<__nv_bfloat16 *>(out),
                                                                      status);
    }
}

bool wgrad_plan(WgradPlan &p, const void *x, int ldx, int cin, const void *gz, int ldgz, int N, int X, int Y, int Z,
                int B, int sms, const char **err)
{
    auto bad = [&](const char *m) {
        if (err) *err = m;
        return false;
    };
    if (!pow2(X) || !pow2(Y) || !pow2(Z) || B < 1) return bad("wgrad: grid sides must be powers of two");
    if (cin < 32 || cin % 32 || ldx < cin || ldx % 8) return bad("wgrad: input channels must be a multiple of 32");
    if (N < 32 || N % 32 || ldgz < N || ldgz % 8) return bad("wgrad: output channels must be a multiple of 32");
    WgradArgs &a = p.a;
    std::memset(&a, 0, sizeof a);
    a.X = X; a.Y = Y; a.Z = Z; a.B = B;
    box_for(X, Y, Z, a.bx, a.by, a.bz, a.bb);
    a.tx = X / a.bx; a.ty = Y / a.by; a.tz = Z / a.bz; a.tb = (B + a.bb - 1) / a.bb;
    const int W = cin % 64 == 0 && N % 64 == 0 ? 64 : 32;
    p.w = W;
    a.cin_blocks = cin / W;
    a.m_total = 27 * cin;
    a.mtiles = (a.m_total + 127) / 128;
    a.ntile = pick_ntile(N);
    while (a.ntile % W || N % a.ntile) a.ntile -= 32;
    a.nntiles = N / a.ntile;
    a.nchunks = (int64_t)a.tx * a.ty * a.tz * a.tb;
    const int64_t items = (int64_t)a.mtiles * a.nntiles;
    int64_t ks = (2 * (int64_t)std::max(1, sms) + items - 1) / items;
    ks = std::min<int64_t>(ks, std::max<int64_t>(1, a.nchunks / 4));
    a.ksplit = (int)std::max<int64_t>(1, ks);
    a.nwork = items * a.ksplit;
    a.a_bytes = 128u * 128 * 2;
    a.b_bytes = (uint32_t)a.ntile * 128 * 2;
    a.stages = (int)std::min<size_t>(6, (SMEM_MAX - 2048 - ctl_bytes(6)) / (a.a_bytes + a.b_bytes));
    if (a.stages < 2) return bad("wgrad: tile does not fit in shared memory");
    a.idesc = idesc_for(a.ntile, true, true);
    a.tmem_cols = tmem_cols_for(a.ntile);
    a.ldg = N;
    p.smem = std::max(SMEM_ONE_CTA, 1024 + (size_t)a.stages * (a.a_bytes + a.b_bytes) + ctl_bytes(a.stages));
    p.grid = (int)std::min<int64_t>(a.nwork, std::max(1, sms));
    const CUtensorMapSwizzle sw = W == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B;
    const cuuint32_t box[5] = {(cuuint32_t)W, (cuuint32_t)a.bx, (cuuint32_t)a.by, (cuuint32_t)a.bz, (cuuint32_t)a.bb};
    const cuuint64_t xd[5] = {(cuuint64_t)ldx, (cuuint64_t)X, (cuuint64_t)Y, (cuuint64_t)Z, (cuuint64_t)B};
    const cuuint64_t xs[4] = {(cuuint64_t)ldx * 2, (cuuint64_t)ldx * 2 * X, (cuuint64_t)ldx * 2 * X * Y,
                              (cuuint64_t)ldx * 2 * X * Y * Z};
    if (!encode(p.xmap, 5, x, xd, xs, box, sw)) return bad("wgrad: input tensor map rejected");
    const cuuint64_t gd[5] = {(cuuint64_t)ldgz, (cuuint64_t)X, (cuuint64_t)Y, (cuuint64_t)Z, (cuuint64_t)B};
    const cuuint64_t gs[4] = {(cuuint64_t)ldgz * 2, (cuuint64_t)ldgz * 2 * X, (cuuint64_t)ldgz * 2 * X * Y,
                              (cuuint64_t)ldgz * 2 * X * Y * Z};
    if (!encode(p.gmap, 5, gz, gd, gs, box, sw)) return bad("wgrad: gradient tensor map rejected");
    return true;
}

void wgrad_launch(const WgradPlan &p, float *g, int *status, cudaStream_t s)
{
    CUtensorMap xm, gm;
    std::memcpy(&xm, p.xmap, sizeof xm);
    std::memcpy(&gm, p.gmap, sizeof gm);
    if (p.w == 64) k_wgrad_umma<64><<<p.grid, NT, p.smem, s>>>(xm, gm, p.a, g, status);
    else k_wgrad_umma<32><<<p.grid, NT, p.smem, s>>>(xm, gm, p.a, g, status);
}

bool gemm_set_attrs()
{
    static int done = 0;
    if (done) return done > 0;
    const int v = (int)SMEM_MAX;
    const auto a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    const bool ok = cudaFuncSetAttribute(k_conv_umma<64, float>, a, v) == cudaSuccess &&
                    cudaFuncSetAttribute(k_conv_umma<64, __nv_bfloat16>, a, v) == cudaSuccess &&
                    cudaFuncSetAttribute(k_conv_umma<32, float>, a, v) == cudaSuccess &&
                    cudaFuncSetAttribute(k_conv_umma<32, __nv_bfloat16>, a, v) == cudaSuccess &&
                    cudaFuncSetAttribute(k_conv_halo<64, float>, a, v) == cudaSuccess &&
                    cudaFuncSetAttribute(k_conv_halo<64, __nv_bfloat16>, a, v) == cudaSuccess &&
                    cudaFuncSetAttribute(k_conv_halo<32, float>, a, v) == cudaSuccess &&
                    cudaFuncSetAttribute(k_conv_halo<32, __nv_bfloat16>, a, v) == cudaSuccess &&
                    cudaFuncSetAttribute(k_wgrad_umma<32>, a, v) == cudaSuccess &&
                    cudaFuncSetAttribute(k_wgrad_umma<64>, a, v) == cudaSuccess;
    done = ok ? 1 : -1;
    return ok;
}

}  // namespace unet
