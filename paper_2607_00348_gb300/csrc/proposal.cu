// Learned period proposal: a small 1D CNN over the time-binned light curve
// that predicts, per log-spaced region of trial periods, the largest signal
// residue SR(P) the TLS search finds there (the paper has no such stage; it
// is trained on spectra that the search itself produces).
//
// Network (fixed): input [B][4096][1]; six 'same' convolutions (taps 7, 5,
// 5, 5, 5, 5, dilated 1, 2, 2, 4, 4, 8 bins of their own input; 64
// channels) each followed by ReLU and max-pooling by 2; linear head 4096 ->
// 128 regions; logistic loss with soft targets; Adam.  The dilations give
// a last-layer unit a receptive field of about 1530 input bins (taps and
// pooling windows; more than a third of the curve) instead of about 320.
//
// Every contraction (convolution forward, data and weight gradients, head
// forward and its two gradients) runs on the BF16 tensor cores (mma.sync
// m16n8k16, FP32 accumulation).  A convolution is an implicit GEMM: a tile of
// 128 positions of one curve and its halo is staged once in shared memory
// (128-byte rows, 16-byte chunks swizzled), and tap k reads the same tile
// k dilation rows further down, so no im2col matrix exists anywhere.  The
// gradient of a pre-activation is never stored either: the tiles of the
// gradient kernels are made from the pooled gradient, the pooled value and
// the pooling choice while they are staged.  Activations are BF16
// [batch][length][channel]; gradients and master parameters are FP32.
// The products of an output are added tap by tap, channels ascending, in
// chains of k16 steps, in the forward pass and the data gradient.
// Measured: forward pass of 256 curves 0.18 ms (2.09 ms with one 64 x 64 tile
// GEMM that gathered its operands element by element), of one curve 41 us
// (607 us), gradient of 128 curves 0.55 ms (11.9 ms).  The first two
// convolutions run at about 300 TFLOP/s, half of what mma.sync reaches from
// registers; the rest is bound by their latency.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "gtls_internal.h"

namespace {

using gtls::set_error;
using bf16 = __nv_bfloat16;

#define PROP_CUDA(call)                                                                         \
    do {                                                                                        \
        cudaError_t e_ = (call);                                                                \
        if (e_ != cudaSuccess)                                                                  \
            return set_error(e_ == cudaErrorMemoryAllocation ? GTLS_ERR_OOM : GTLS_ERR_CUDA,    \
                             std::string(#call) + ": " + cudaGetErrorString(e_));               \
    } while (0)

#define PROP_TRY(x)                   \
    do {                              \
        gtls_status s_ = (x);         \
        if (s_ != GTLS_OK) return s_; \
    } while (0)

constexpr int kBins = 4096;
constexpr int kCh = 64;
constexpr int kConv = 6;
constexpr int kReg = 128;
constexpr int kFeat = (kBins >> kConv) * kCh;
constexpr int kTaps[kConv] = {7, 5, 5, 5, 5, 5};
constexpr int kDil[kConv] = {1, 2, 2, 4, 4, 8};   // tap spacing of each convolution (its input's bins)
constexpr double kRegionLo = 0.5, kRegionHi = 1024.0;   // days: regions split this range evenly in log P

// offsets of the flat parameter vector (order: w0 b0 ... w5 b5 wh bh)
struct Layout {
    int64_t w[kConv], b[kConv], wh, bh, total;
    Layout()
    {
        int64_t pos = 0;
        int cin = 1;
        for (int i = 0; i < kConv; ++i) {
            w[i] = pos;
            pos += (int64_t)kCh * kTaps[i] * cin;
            b[i] = pos;
            pos += kCh;
            cin = kCh;
        }
        wh = pos;
        pos += (int64_t)kReg * kFeat;
        bh = pos;
        pos += kReg;
        total = pos;
    }
};

// ---------------------------------------------------------------------------
// tensor-core building blocks
// ---------------------------------------------------------------------------

__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

__device__ __forceinline__ void ldsm2t(uint32_t& r0, uint32_t& r1, uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(addr));
}

// 16 bytes global -> shared, zeros when !in
__device__ __forceinline__ void copy16(uint32_t dst, const void* src, bool in)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16 : 0) : "memory");
}

__device__ __forceinline__ void copies_done()
{
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
}

__device__ __forceinline__ uint32_t smem_addr(const void* p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Byte offset of 16-byte chunk c of row r in a tile of 128-byte rows: the
// eight rows of one ldmatrix phase fall into eight different bank groups.
__device__ __forceinline__ uint32_t at128(int r, int c) { return (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4)); }

constexpr int kRows = 128;                     // positions per convolution tile
constexpr int kMaxHalo = 16;                   // rows before and after it (2 x the largest dilation)
constexpr int kConvTaps = 5;                   // taps of convolutions 1..5
constexpr int kWBytes = kConvTaps * kCh * 128; // their staged weights
constexpr int kABytes = (kRows + 2 * kMaxHalo) * 128;

// Where the gradient of a pre-activation comes from: the gradient of the
// pooled output (FP32), the pooled output and which row of a pair won.
struct PoolGrad {
    const float* grad;
    const bf16* pooled;
    const uint8_t* arg;
};

// Rows [l0, l0 + rows) (l0, rows even) of the pre-activation gradient of one
// curve of L positions, made from its pooled gradient (to the winning row of
// each pair where the pooled value is positive, zero elsewhere), into a tile
// of 128-byte rows; rows outside [0, L) are zero.  `first`: the curve's first
// pooled position.
__device__ __forceinline__ void stage_pool_grad(unsigned char* tile, const PoolGrad& pg, int64_t first, int l0, int rows,
                                                int L)
{
    for (int e = threadIdx.x; e < rows / 2 * 8; e += blockDim.x) {
        const int q = e >> 3, c = e & 7;
        const int pos = (l0 >> 1) + q;
        uint4 lo = make_uint4(0, 0, 0, 0), hi = lo;
        if (pos >= 0 && pos < L / 2) {
            const int64_t at = (first + pos) * kCh + 8 * c;
            const float4 g0 = __ldg(reinterpret_cast<const float4*>(pg.grad + at));
            const float4 g1 = __ldg(reinterpret_cast<const float4*>(pg.grad + at) + 1);
            const uint4 pv = __ldg(reinterpret_cast<const uint4*>(pg.pooled + at));
            const uint2 av = __ldg(reinterpret_cast<const uint2*>(pg.arg + at));
            const float g[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
            const uint32_t p[4] = {pv.x, pv.y, pv.z, pv.w};
            uint32_t a[4], b[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                uint32_t even = 0, odd = 0;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint32_t pb = h ? p[u] >> 16 : p[u] & 0xffffu;
                    // pooled > 0: the pooled value is a ReLU's output
                    const float v = pb != 0 && pb <= 0x7f80u ? g[2 * u + h] : 0.0f;
                    const uint32_t bits = (uint32_t)__bfloat16_as_ushort(__float2bfloat16(v)) << (16 * h);
                    const uint32_t won = (((u < 2 ? av.x : av.y) >> (8 * ((2 * u + h) & 3))) & 1u);
                    if (won) odd |= bits;
                    else even |= bits;
                }
                a[u] = even;
                b[u] = odd;
            }
            lo = make_uint4(a[0], a[1], a[2], a[3]);
            hi = make_uint4(b[0], b[1], b[2], b[3]);
        }
        *reinterpret_cast<uint4*>(tile + at128(2 * q, c)) = lo;
        *reinterpret_cast<uint4*>(tile + at128(2 * q + 1, c)) = hi;
    }
}

// Rows [l0, l0 + rows) of one curve's activations (L x 64, zero outside).
__device__ __forceinline__ void stage_rows(uint32_t tile, const bf16* x, int l0, int rows, int L)
{
    for (int e = threadIdx.x; e < rows * 8; e += blockDim.x) {
        const int r = e >> 3, c = e & 7, l = l0 + r;
        const bool in = l >= 0 && l < L;
        copy16(tile + at128(r, c), x + (int64_t)(in ? l : 0) * kCh + 8 * c, in);
    }
}

// Bias, ReLU and max-pool of row pairs of a warp's (16 i + g, 8 j + 2 t)
// accumulators into the staged output tile (pooled rows of 128 bytes, and 64
// bytes of pooling choices when kArg); rows 2q and 2q + 1 sit in lanes g, g ^ 1.
template <bool kArg>
__device__ __forceinline__ void pool_tile(float (&acc)[2][8][4], const float* __restrict__ bias, int row0, int lane,
                                          bf16* pool, uint8_t* arg)
{
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const float2 bv = __ldg(reinterpret_cast<const float2*>(bias + 8 * j + 2 * t));
#pragma unroll
        for (int i = 0; i < 2; ++i) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float v0 = fmaxf(acc[i][j][2 * h] + bv.x, 0.0f), v1 = fmaxf(acc[i][j][2 * h + 1] + bv.y, 0.0f);
                const float o0 = __shfl_xor_sync(0xffffffffu, v0, 4), o1 = __shfl_xor_sync(0xffffffffu, v1, 4);
                if ((g & 1) != 0) continue;
                const int q = (row0 + 16 * i + g + 8 * h) >> 1, col = 8 * j + 2 * t;
                const bool w0 = o0 > v0, w1 = o1 > v1;   // the first of equal values wins
                *reinterpret_cast<__nv_bfloat162*>(pool + q * kCh + col) =
                    __nv_bfloat162(__float2bfloat16(w0 ? o0 : v0), __float2bfloat16(w1 ? o1 : v1));
                if (kArg) *reinterpret_cast<uint16_t*>(arg + q * kCh + col) = (uint16_t)((w0 ? 1 : 0) | (w1 ? 256 : 0));
            }
        }
    }
}

// The staged output tile to global memory (64 pooled rows, contiguous).
template <bool kArg>
__device__ __forceinline__ void store_pool_tile(const bf16* pool, const uint8_t* arg, bf16* out, uint8_t* arg_out)
{
    for (int e = threadIdx.x; e < kRows / 2 * kCh / 8; e += blockDim.x)
        reinterpret_cast<uint4*>(out)[e] = reinterpret_cast<const uint4*>(pool)[e];
    if (kArg)
        for (int e = threadIdx.x; e < kRows / 2 * kCh / 16; e += blockDim.x)
            reinterpret_cast<uint4*>(arg_out)[e] = reinterpret_cast<const uint4*>(arg)[e];
}

// ---------------------------------------------------------------------------
// convolution 0 (one input channel, 7 taps): the taps are one zero-padded k16
// step; the FP32 input is rounded here (and kept for the backward pass).
// Bound by the stores of its pooled output: 256 curves 32 us (67 MB)
// ---------------------------------------------------------------------------

template <bool kTrain>
__global__ void __launch_bounds__(128) k_conv0(const float* __restrict__ x, const bf16* __restrict__ w,
                                               const float* __restrict__ bias, bf16* __restrict__ xb,
                                               bf16* __restrict__ out, uint8_t* __restrict__ arg_out, int tiles)
{
    __shared__ bf16 xs[kRows + 16];
    __shared__ __align__(16) bf16 pool[kRows / 2 * kCh];
    __shared__ __align__(16) uint8_t arg[kTrain ? kRows / 2 * kCh : 16];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, t = lane & 3;
    const uint32_t last = t == 3 ? 0x0000ffffu : 0xffffffffu;   // taps 0..6 of the eight
    uint32_t b[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const bf16* r = w + (8 * j + g) * 7 + 2 * t;
        b[j] = (uint32_t)__bfloat16_as_ushort(r[0]) |
               (t < 3 ? (uint32_t)__bfloat16_as_ushort(r[1]) << 16 : 0u);
    }
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int64_t row0 = (int64_t)tile * kRows;
        const int l0 = (int)(row0 % kBins);
        for (int e = threadIdx.x; e < kRows + 8; e += blockDim.x) {
            const int l = l0 + e - 3;
            const bf16 v = __float2bfloat16(l >= 0 && l < kBins ? x[row0 + e - 3] : 0.0f);
            xs[e] = v;
            if (kTrain && e >= 3 && e < kRows + 3) xb[row0 + e - 3] = v;
        }
        __syncthreads();
        float acc[2][8][4];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            uint32_t a[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const bf16* r = xs + warp * 32 + 16 * i + 8 * h + g + 2 * t;
                a[h] = ((uint32_t)__bfloat16_as_ushort(r[0]) | (uint32_t)__bfloat16_as_ushort(r[1]) << 16) & last;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
#pragma unroll
                for (int u = 0; u < 4; ++u) acc[i][j][u] = 0.0f;
                mma_bf16(acc[i][j], a, b[j], 0u);
            }
        }
        pool_tile<kTrain>(acc, bias, warp * 32, lane, pool, arg);
        __syncthreads();
        store_pool_tile<kTrain>(pool, arg, out + row0 / 2 * kCh, kTrain ? arg_out + row0 / 2 * kCh : nullptr);
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// convolutions 1..5, and their data gradient (kBack: the 'same' convolution
// of the pre-activation gradient with the flipped taps; the transposed
// weights are read through ldmatrix.trans from the same staged weights).
// Four warps of 32 rows x 64 columns; the weights stay staged over a CTA's
// tiles, and three CTAs of an SM overlap their staging and their products.
// ---------------------------------------------------------------------------

struct ConvArgs {
    const bf16* x;            // activations in (!kBack)
    PoolGrad pg;              // pre-activation gradient in (kBack)
    const bf16* w;            // [64][5][64]
    const float* bias;
    bf16* pooled;             // out (!kBack)
    uint8_t* arg;
    float* dx;                // out (kBack)
    int L, dil, tiles;
};

template <bool kBack, bool kArg>
__global__ void __launch_bounds__(128, 3) k_conv(const __grid_constant__ ConvArgs c)
{
    extern __shared__ __align__(128) unsigned char conv_smem[];
    unsigned char* const ws = conv_smem;
    unsigned char* const as = conv_smem + kWBytes;
    const uint32_t ws_a = smem_addr(ws), as_a = smem_addr(as);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, t = lane & 3, m8 = lane >> 3, r8 = lane & 7;
    for (int e = threadIdx.x; e < kConvTaps * kCh * 8; e += blockDim.x) {
        const int tap = e / (kCh * 8), co = (e >> 3) % kCh, ch = e & 7;
        copy16(ws_a + tap * kCh * 128 + at128(co, ch), c.w + (co * kConvTaps + tap) * kCh + 8 * ch, true);
    }
    const int halo = 2 * c.dil, rows = kRows + 2 * halo;
    const int per = c.L / kRows;
    for (int tile = blockIdx.x; tile < c.tiles; tile += gridDim.x) {
        const int seq = tile / per, l0 = (tile - seq * per) * kRows;
        if (kBack) stage_pool_grad(as, c.pg, (int64_t)seq * (c.L / 2), l0 - halo, rows, c.L);
        else stage_rows(as_a, c.x + (int64_t)seq * c.L * kCh, l0 - halo, rows, c.L);
        copies_done();
        __syncthreads();
        float acc[2][8][4];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j)
#pragma unroll
                for (int u = 0; u < 4; ++u) acc[i][j][u] = 0.0f;
        for (int tap = 0; tap < kConvTaps; ++tap) {
            const int base = warp * 32 + tap * c.dil + (lane & 15);
            const uint32_t wt = ws_a + (kBack ? kConvTaps - 1 - tap : tap) * kCh * 128;
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
                uint32_t a[2][4];
#pragma unroll
                for (int i = 0; i < 2; ++i) ldsm4(a[i], as_a + at128(base + 16 * i, 2 * ks + (lane >> 4)));
#pragma unroll
                for (int jp = 0; jp < 4; ++jp) {
                    uint32_t b[4];
                    if (kBack) ldsm4t(b, wt + at128(16 * ks + 8 * (m8 & 1) + r8, 2 * jp + (m8 >> 1)));
                    else ldsm4(b, wt + at128(16 * jp + 8 * (m8 >> 1) + r8, 2 * ks + (m8 & 1)));
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        mma_bf16(acc[i][2 * jp], a[i], b[0], b[1]);
                        mma_bf16(acc[i][2 * jp + 1], a[i], b[2], b[3]);
                    }
                }
            }
        }
        __syncthreads();   // the tile is read: its space takes the output
        if (kBack) {
            float* const out = c.dx + ((int64_t)seq * c.L + l0 + warp * 32) * kCh;
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j)
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        *reinterpret_cast<float2*>(out + (16 * i + g + 8 * h) * kCh + 8 * j + 2 * t) =
                            make_float2(acc[i][j][2 * h], acc[i][j][2 * h + 1]);
        } else {
            bf16* const pool = reinterpret_cast<bf16*>(as);
            uint8_t* const arg = as + kRows / 2 * 128;
            pool_tile<kArg>(acc, c.bias, warp * 32, lane, pool, arg);
            __syncthreads();
            const int64_t q0 = ((int64_t)seq * c.L + l0) / 2 * kCh;
            store_pool_tile<kArg>(pool, arg, c.pooled + q0, kArg ? c.arg + q0 : nullptr);
            __syncthreads();
        }
    }
}

// Weight and bias gradient of convolutions 1..5: dW[co][tap][ci] = sum over
// positions of dpre[l][co] x[l + (tap - 2) dil][ci].  Both operands are read
// transposed from tiles of positions; a CTA keeps all 64 x 320 sums in
// registers over its tiles (warp w: input channels 8 w .. 8 w + 7 of every
// tap) and adds them to the gradient once.
__global__ void __launch_bounds__(256, 1) k_conv_dw(const __grid_constant__ ConvArgs c, float* __restrict__ dw,
                                                    float* __restrict__ db)
{
    extern __shared__ __align__(128) unsigned char conv_smem[];
    unsigned char* const ds = conv_smem;               // dpre: 128 rows
    unsigned char* const xs = conv_smem + kRows * 128; // x: 128 rows and the halo
    const uint32_t ds_a = smem_addr(ds), xs_a = smem_addr(xs);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, t = lane & 3, m8 = lane >> 3, r8 = lane & 7;
    const int halo = 2 * c.dil, per = c.L / kRows;
    float acc[kConvTaps][4][4];
#pragma unroll
    for (int tap = 0; tap < kConvTaps; ++tap)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int u = 0; u < 4; ++u) acc[tap][i][u] = 0.0f;
    float colsum = 0.0f;
    for (int tile = blockIdx.x; tile < c.tiles; tile += gridDim.x) {
        const int seq = tile / per, l0 = (tile - seq * per) * kRows;
        stage_rows(xs_a, c.x + (int64_t)seq * c.L * kCh, l0 - halo, kRows + 2 * halo, c.L);
        stage_pool_grad(ds, c.pg, (int64_t)seq * (c.L / 2), l0, kRows, c.L);
        copies_done();
        __syncthreads();
        for (int k0 = 0; k0 < kRows; k0 += 16) {
            uint32_t a[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                ldsm4t(a[i], ds_a + at128(k0 + 8 * (m8 >> 1) + r8, 2 * i + (m8 & 1)));
#pragma unroll
            for (int tap = 0; tap < kConvTaps; ++tap) {
                uint32_t b0, b1;
                ldsm2t(b0, b1, xs_a + at128(k0 + tap * c.dil + 8 * (m8 & 1) + r8, warp));
#pragma unroll
                for (int i = 0; i < 4; ++i) mma_bf16(acc[tap][i], a[i], b0, b1);
            }
        }
        {
            const int col = threadIdx.x & 63, r0 = (threadIdx.x >> 6) * 32;
#pragma unroll 8
            for (int r = r0; r < r0 + 32; ++r)
                colsum += __bfloat162float(*reinterpret_cast<const bf16*>(ds + at128(r, col >> 3) + 2 * (col & 7)));
        }
        __syncthreads();
    }
#pragma unroll
    for (int tap = 0; tap < kConvTaps; ++tap)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                atomicAdd(reinterpret_cast<float2*>(dw + ((16 * i + g + 8 * h) * kConvTaps + tap) * kCh + 8 * warp + 2 * t),
                          make_float2(acc[tap][i][2 * h], acc[tap][i][2 * h + 1]));
    atomicAdd(db + (threadIdx.x & 63), colsum);
}

// The same for convolution 0 (one input channel, 7 taps): the warps split the
// positions of a tile.
__global__ void __launch_bounds__(256) k_conv0_dw(const bf16* __restrict__ x, const PoolGrad pg, float* __restrict__ dw,
                                                  float* __restrict__ db, int tiles)
{
    __shared__ __align__(128) unsigned char ds[kRows * 128];
    __shared__ bf16 xs[kRows + 16];
    __shared__ float sum[kCh * 8];
    const uint32_t ds_a = smem_addr(ds);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, t = lane & 3, m8 = lane >> 3, r8 = lane & 7;
    for (int e = threadIdx.x; e < kCh * 8; e += blockDim.x) sum[e] = 0.0f;
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[i][u] = 0.0f;
    float colsum = 0.0f;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int64_t row0 = (int64_t)tile * kRows;
        const int l0 = (int)(row0 % kBins);
        stage_pool_grad(ds, pg, row0 / kBins * (kBins / 2), l0, kRows, kBins);
        for (int e = threadIdx.x; e < kRows + 8; e += blockDim.x) {
            const int l = l0 + e - 3;
            xs[e] = l >= 0 && l < kBins ? x[row0 + e - 3] : __float2bfloat16(0.0f);
        }
        __syncthreads();
        const int k0 = warp * 16;
        // positions k0 + 2 t, + 1 (and + 8) and tap g (the eighth column is not used)
        const bf16* r = xs + k0 + 2 * t + g;
        const uint32_t b0 = (uint32_t)__bfloat16_as_ushort(r[0]) | (uint32_t)__bfloat16_as_ushort(r[1]) << 16;
        const uint32_t b1 = (uint32_t)__bfloat16_as_ushort(r[8]) | (uint32_t)__bfloat16_as_ushort(r[9]) << 16;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            uint32_t a[4];
            ldsm4t(a, ds_a + at128(k0 + 8 * (m8 >> 1) + r8, 2 * i + (m8 & 1)));
            mma_bf16(acc[i], a, b0, b1);
        }
        const int col = threadIdx.x & 63, q0 = (threadIdx.x >> 6) * 32;
#pragma unroll 8
        for (int q = q0; q < q0 + 32; ++q)
            colsum += __bfloat162float(*reinterpret_cast<const bf16*>(ds + at128(q, col >> 3) + 2 * (col & 7)));
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int u = 0; u < 4; ++u) atomicAdd(&sum[(16 * i + g + 8 * (u >> 1)) * 8 + 2 * t + (u & 1)], acc[i][u]);
    __syncthreads();
    for (int e = threadIdx.x; e < kCh * 7; e += blockDim.x) atomicAdd(dw + e, sum[e / 7 * 8 + e % 7]);
    atomicAdd(db + (threadIdx.x & 63), colsum);
}

// ---------------------------------------------------------------------------
// head
// ---------------------------------------------------------------------------

// z[row][reg] = bias + sum_f feat[row][f] wh[reg][f]: 16 rows x 16 regions per
// CTA, the features split over its eight warps (a batch of 256 gives 128 CTAs,
// one curve 8).  A lane's 16-byte loads hold the k indices of two k16 steps
// (the same permutation of k on both sides).
__global__ void __launch_bounds__(256) k_head(const bf16* __restrict__ feat, const bf16* __restrict__ wh,
                                              const float* __restrict__ bias, float* __restrict__ z,
                                              float* __restrict__ logits, float* __restrict__ scores, int B)
{
    __shared__ float part[8][16][17];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, t = lane & 3;
    const int row0 = blockIdx.x * 16, n0 = blockIdx.y * 16;
    constexpr int kSpan = kFeat / 8;
    const uint4* fa = reinterpret_cast<const uint4*>(feat + (int64_t)min(row0 + g, B - 1) * kFeat + warp * kSpan) + t;
    const uint4* fb = reinterpret_cast<const uint4*>(feat + (int64_t)min(row0 + g + 8, B - 1) * kFeat + warp * kSpan) + t;
    const uint4* wa = reinterpret_cast<const uint4*>(wh + (int64_t)(n0 + g) * kFeat + warp * kSpan) + t;
    const uint4* wb = reinterpret_cast<const uint4*>(wh + (int64_t)(n0 + g + 8) * kFeat + warp * kSpan) + t;
    float acc[2][4] = {{0.0f, 0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f, 0.0f}};
#pragma unroll 4
    for (int k = 0; k < kSpan / 32; ++k) {
        const uint4 a0 = __ldg(fa + 4 * k), a1 = __ldg(fb + 4 * k), b0 = __ldg(wa + 4 * k), b1 = __ldg(wb + 4 * k);
        const uint32_t lo[4] = {a0.x, a1.x, a0.y, a1.y}, hi[4] = {a0.z, a1.z, a0.w, a1.w};
        mma_bf16(acc[0], lo, b0.x, b0.y);
        mma_bf16(acc[1], lo, b1.x, b1.y);
        mma_bf16(acc[0], hi, b0.z, b0.w);
        mma_bf16(acc[1], hi, b1.z, b1.w);
    }
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int u = 0; u < 4; ++u) part[warp][g + 8 * (u >> 1)][8 * j + 2 * t + (u & 1)] = acc[j][u];
    __syncthreads();
    const int r = threadIdx.x >> 4, n = threadIdx.x & 15;
    if (row0 + r >= B) return;
    float v = 0.0f;
#pragma unroll
    for (int w = 0; w < 8; ++w) v += part[w][r][n];
    v += bias[n0 + n];
    const int64_t o = (int64_t)(row0 + r) * kReg + n0 + n;
    z[o] = v;
    if (logits) logits[o] = v;
    if (scores) scores[o] = 1.0f / (1.0f + expf(-v));
}

// The same sums in one chain of k16 steps per output (training: the gradient
// of the logits is rounded to BF16, where the rounding of the logits would
// show): 16 rows x 32 regions per CTA, a warp 8 regions, 256 features staged
// ahead of the products.
constexpr int kHeadSpan = 256;
constexpr int kHeadBytes = (16 + 32) * kHeadSpan * 2;   // one stage

__global__ void __launch_bounds__(128) k_head_chain(const bf16* __restrict__ feat, const bf16* __restrict__ wh,
                                                    const float* __restrict__ bias, float* __restrict__ z, int B)
{
    __shared__ __align__(128) unsigned char hs[2 * kHeadBytes];
    const uint32_t hs_a = smem_addr(hs);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, t = lane & 3;
    const int row0 = blockIdx.x * 16, n0 = blockIdx.y * 32;
    // a stage: per 64 features, 16 rows of features and 32 of weights
    auto stage = [&](int k, uint32_t to) {
        for (int e = threadIdx.x; e < 48 * (kHeadSpan / 8); e += 128) {
            const int c = e & 7, r = (e >> 3) % 48, sub = e / (8 * 48);
            const int f = k * kHeadSpan + sub * 64 + 8 * c;
            const bool in = r >= 16 || row0 + r < B;
            const bf16* src = r < 16 ? feat + (int64_t)(in ? row0 + r : 0) * kFeat : wh + (int64_t)(n0 + r - 16) * kFeat;
            copy16(to + sub * 48 * 128 + at128(r, c), src + f, in);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    stage(0, hs_a);
    for (int k = 0; k < kFeat / kHeadSpan; ++k) {
        const uint32_t at = hs_a + (k & 1) * kHeadBytes;
        if (k + 1 < kFeat / kHeadSpan) {
            stage(k + 1, hs_a + ((k + 1) & 1) * kHeadBytes);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
#pragma unroll
        for (int ks = 0; ks < kHeadSpan / 16; ks += 2) {
            const uint32_t sub = at + (ks >> 2) * 48 * 128;
            uint32_t a0[4], a1[4], b[4];
            ldsm4(a0, sub + at128(lane & 15, 2 * (ks & 3) + (lane >> 4)));
            ldsm4(a1, sub + at128(lane & 15, 2 * ((ks + 1) & 3) + (lane >> 4)));
            ldsm4(b, sub + at128(16 + 8 * warp + (lane & 7), 2 * (ks & 3) + (lane >> 3)));   // k16 steps ks, ks + 1
            mma_bf16(acc, a0, b[0], b[1]);
            mma_bf16(acc, a1, b[2], b[3]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int r = row0 + g + 8 * (u >> 1), n = n0 + 8 * warp + 2 * t + (u & 1);
        if (r < B) z[(int64_t)r * kReg + n] = acc[u] + bias[n];
    }
}

// dWh[reg][f] = sum_b dz[b][reg] feat[b][f] for 32 features per CTA (warp w:
// regions 16 w ..), and the bias gradient (CTA 0).
__global__ void __launch_bounds__(256) k_head_dw(const bf16* __restrict__ dzb, const float* __restrict__ dz,
                                                 const bf16* __restrict__ feat, float* __restrict__ dw,
                                                 float* __restrict__ db, int B)
{
    __shared__ __align__(128) unsigned char zs[64 * 256];   // 64 rows of 128 regions (two 128-byte halves)
    __shared__ __align__(128) unsigned char fs[64 * 128];   // 64 rows of 32 features (a 128-byte row each, half used)
    const uint32_t zs_a = smem_addr(zs), fs_a = smem_addr(fs);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, t = lane & 3, m8 = lane >> 3, r8 = lane & 7;
    const int f0 = blockIdx.x * 32;
    float acc[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[j][u] = 0.0f;
    for (int b0 = 0; b0 < B; b0 += 64) {
        for (int e = threadIdx.x; e < 64 * 16; e += blockDim.x) {
            const int r = e >> 4, c = e & 15;
            const bool in = b0 + r < B;
            copy16(zs_a + (c >> 3) * 64 * 128 + at128(r, c & 7), dzb + (int64_t)(in ? b0 + r : 0) * kReg + 8 * c, in);
        }
        {
            const int r = threadIdx.x >> 2, c = threadIdx.x & 3;
            const bool in = b0 + r < B;
            copy16(fs_a + at128(r, c), feat + (int64_t)(in ? b0 + r : 0) * kFeat + f0 + 8 * c, in);
        }
        copies_done();
        __syncthreads();
#pragma unroll
        for (int k0 = 0; k0 < 64; k0 += 16) {
            uint32_t a[4];
            ldsm4t(a, zs_a + (warp >> 2) * 64 * 128 + at128(k0 + 8 * (m8 >> 1) + r8, 2 * (warp & 3) + (m8 & 1)));
#pragma unroll
            for (int jp = 0; jp < 2; ++jp) {
                uint32_t b[4];
                ldsm4t(b, fs_a + at128(k0 + 8 * (m8 & 1) + r8, 2 * jp + (m8 >> 1)));
                mma_bf16(acc[2 * jp], a, b[0], b[1]);
                mma_bf16(acc[2 * jp + 1], a, b[2], b[3]);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h)
            *reinterpret_cast<float2*>(dw + (int64_t)(16 * warp + g + 8 * h) * kFeat + f0 + 8 * j + 2 * t) =
                make_float2(acc[j][2 * h], acc[j][2 * h + 1]);
    if (blockIdx.x == 0 && threadIdx.x < kReg) {
        float s = 0.0f;
#pragma unroll 8
        for (int b = 0; b < B; ++b) s += dz[(int64_t)b * kReg + threadIdx.x];
        db[threadIdx.x] = s;
    }
}

// dfeat[b][f] = sum_reg dz[b][reg] wh[reg][f]: 64 rows x 64 features per CTA.
__global__ void __launch_bounds__(128) k_head_dx(const bf16* __restrict__ dzb, const bf16* __restrict__ wh,
                                                 float* __restrict__ dfeat, int B)
{
    __shared__ __align__(128) unsigned char zs[64 * 256];
    __shared__ __align__(128) unsigned char ws[kReg * 128];
    const uint32_t zs_a = smem_addr(zs), ws_a = smem_addr(ws);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, t = lane & 3, m8 = lane >> 3, r8 = lane & 7;
    const int b0 = blockIdx.x * 64, f0 = blockIdx.y * 64;
    for (int e = threadIdx.x; e < 64 * 16; e += blockDim.x) {
        const int r = e >> 4, c = e & 15;
        const bool in = b0 + r < B;
        copy16(zs_a + (c >> 3) * 64 * 128 + at128(r, c & 7), dzb + (int64_t)(in ? b0 + r : 0) * kReg + 8 * c, in);
    }
    for (int e = threadIdx.x; e < kReg * 8; e += blockDim.x)
        copy16(ws_a + at128(e >> 3, e & 7), wh + (int64_t)(e >> 3) * kFeat + f0 + 8 * (e & 7), true);
    copies_done();
    __syncthreads();
    float acc[8][4];
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[j][u] = 0.0f;
#pragma unroll
    for (int ks = 0; ks < kReg / 16; ++ks) {
        uint32_t a[4];
        ldsm4(a, zs_a + (ks >> 2) * 64 * 128 + at128(warp * 16 + (lane & 15), 2 * (ks & 3) + (lane >> 4)));
#pragma unroll
        for (int jp = 0; jp < 4; ++jp) {
            uint32_t b[4];
            ldsm4t(b, ws_a + at128(16 * ks + 8 * (m8 & 1) + r8, 2 * jp + (m8 >> 1)));
            mma_bf16(acc[2 * jp], a, b[0], b[1]);
            mma_bf16(acc[2 * jp + 1], a, b[2], b[3]);
        }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = b0 + warp * 16 + g + 8 * h;
            if (r < B)
                *reinterpret_cast<float2*>(dfeat + (int64_t)r * kFeat + f0 + 8 * j + 2 * t) =
                    make_float2(acc[j][2 * h], acc[j][2 * h + 1]);
        }
}

// ---------------------------------------------------------------------------
// element-wise and reduction kernels
// ---------------------------------------------------------------------------

__global__ void k_to_bf16(const float* __restrict__ x, bf16* __restrict__ y, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = __float2bfloat16(x[i]);
}

// Masked logistic loss with soft targets: loss = sum mask (softplus(z) - t z)
// / sum mask; dz = mask (sigmoid(z) - t) / sum mask (FP32 and BF16).  The FP64
// transcendentals bound it (a warp's FP64 instruction takes an SM 16 cycles: 72
// us at a batch of 128 on 16 SMs), so the elements are spread over all SMs; each sums the mask for itself, and
// the last one to finish adds the blocks' parts (one per thread).
constexpr int kLossBlocks = 128, kLossThreads = 128;
static_assert(kLossBlocks <= kLossThreads, "the last block reads one part per thread");

__device__ __forceinline__ double block_sum_fp64(double v, double* sh)
{
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    const double r = sh[0];
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(kLossThreads) k_loss(const float* __restrict__ z, const float* __restrict__ tgt,
                                               const float* __restrict__ mask, int n, float* __restrict__ dz,
                                               bf16* __restrict__ dzb, double* __restrict__ part,
                                               unsigned int* __restrict__ done, double* __restrict__ loss)
{
    __shared__ double sh[kLossThreads];
    __shared__ bool last;
    // masks of zeros and ones are counted in integers
    int ones = 0;
    double cnt = 0.0;
#pragma unroll 8
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const float m = mask[i];
        if (m == 1.0f) ++ones;
        else if (m != 0.0f) cnt += m;
    }
    const double total = fmax(block_sum_fp64(cnt + ones, sh), 1.0);
    double acc = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const double zi = z[i], m = mask[i], ti = tgt[i];
        const double e = exp(-fabs(zi)), inv = 1.0 / (1.0 + e);
        acc += m * (fmax(zi, 0.0) + log1p(e) - ti * zi);
        const double sg = zi >= 0.0 ? inv : e * inv;
        const float d = (float)(m * (sg - ti) / total);
        dz[i] = d;
        dzb[i] = __float2bfloat16(d);
    }
    acc = block_sum_fp64(acc, sh);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = acc;
        __threadfence();
        last = atomicAdd(done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (last) {   // block-uniform
        __threadfence();
        const double all = block_sum_fp64(threadIdx.x < gridDim.x ? __ldcg(part + threadIdx.x) : 0.0, sh);
        if (threadIdx.x == 0) {
            *loss = all / total;
            *done = 0u;
        }
    }
}

// Adam (Kingma & Ba 2015) on the FP32 master parameters, then their BF16 copy.
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, bf16* __restrict__ pb, int64_t n, float lr, float c1, float c2)
{
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        p[i] = pi;
        pb[i] = __float2bfloat16(pi);
    }
}

// Time binning: bin b of a curve holds its points with
// floor((t - t_min) / (t_max - t_min) * 4096) = b (the last point in the last
// bin); value sum(w r) / sqrt(sum w), r = 1 - y, w = 1/dy^2; empty bins 0.
// Sums in FP64.
//
// The FP64 pipe bounds it: an FP64 instruction of a warp takes an SM 16
// cycles, whether one lane needs it or all.  k_bin_sorted (points in time
// order, as curves come) therefore first finds where every bin starts -- one
// subtraction and one conversion in FP64 per point, the product in FP32, and
// the bin formula itself only where that product is too near a bin's edge --
// and then gives each bin to one thread, which needs two FP64 operations per
// point (1 - y and its sum) and one reciprocal per bin while dy stays the
// same.  kBinCtas CTAs share a curve, each a quarter of the bins.  Curves
// whose points turn out not to be in order, or that have too many of them for
// its 32-bit counts, are flagged and left to k_bin_any (shared-memory atomics).  256 curves of 20,000 to 72,000 points:
// 0.28 ms; 1.9 ms with two divisions and two atomics per point.
constexpr int kBinThreads = 256;
constexpr int kBinRun = 16;      // consecutive points of a thread (k_bin_any)
constexpr int kBinCtas = 4;      // CTAs per curve
constexpr int64_t kBinSortedMax = int64_t(1) << 30;   // points of a curve that k_bin_sorted takes (steps of a few
                                                      // thousand past the last one still fit an int)
constexpr long long kInfKey = 0x7ff0000000000000ll;

// The bin formula.
__device__ __forceinline__ int bin_of(double t, double lo, double span)
{
    if (!(span > 0.0)) return 0;
    const double f = __dmul_rn(__ddiv_rn(__dsub_rn(t, lo), span), (double)kBins);
    return max((int)fmin(floor(f), (double)(kBins - 1)), 0);
}

// The same, by an FP32 product where that is clear of the bins' edges: its
// three roundings are off by at most 4096 * 3 * 2^-24 = 7.4e-4 together.
__device__ __forceinline__ int bin_near(double t, double lo, double span, float per_day)
{
    const float f = (float)__dsub_rn(t, lo) * per_day;
    const float fl = floorf(f), frac = f - fl;
    if (frac > 8e-4f && frac < 1.0f - 8e-4f && f < (float)kBins) return (int)fl;
    return bin_of(t, lo, span);
}

__device__ __forceinline__ long long time_key(double v)
{
    const long long u = __double_as_longlong(v);
    return u < 0 ? u ^ 0x7fffffffffffffffll : u;
}

__device__ __forceinline__ double key_time(long long k)
{
    return __longlong_as_double(k < 0 ? k ^ 0x7fffffffffffffffll : k);
}

__global__ void __launch_bounds__(kBinThreads) k_bin_sorted(const double* __restrict__ t, const double* __restrict__ y,
                                                            const double* __restrict__ dy,
                                                            const int64_t* __restrict__ off, float* __restrict__ x,
                                                            float* __restrict__ mean, float* __restrict__ wsum,
                                                            unsigned int* __restrict__ unsorted)
{
    constexpr int kShare = kBins / kBinCtas;
    __shared__ int start[kShare + 1];
    __shared__ int edge[2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lc = blockIdx.x / kBinCtas, rank = blockIdx.x - lc * kBinCtas;
    const int64_t o = off[lc], points = off[lc + 1] - o;
    if (points > kBinSortedMax) {   // (all CTAs of the curve)
        if (threadIdx.x == 0) unsorted[lc] = 1u;
        return;
    }
    const int n = (int)points;
    t += o;
    y += o;
    dy += o;
    const double lo = t[0], span = __dsub_rn(t[n - 1], lo);
    const float per_day = span > 0.0 ? (float)((double)kBins / span) : 0.0f;
    const int b0 = rank * kShare;
    // first point of bin b0 and of the next CTA's first bin, as if in order
    // (32 probes at a time)
    if (warp < 2) {
        const int want = b0 + warp * kShare;
        int a = 0, b = n;   // the answer lies in [a, b]
        if (want == 0) b = 0;
        if (want == kBins) a = n;
        while (a < b) {
            const int step = (b - a + 31) / 32;
            const int i = a + lane * step;
            const unsigned int below = __ballot_sync(0xffffffffu, i < b && bin_of(t[min(i, n - 1)], lo, span) < want);
            const int c = __popc(below);   // probes below: the answer is past the last of them
            const int na = c == 0 ? a : min(b, a + (c - 1) * step + 1);
            b = c == 0 ? a : min(b, a + c * step);
            a = na;
        }
        if (lane == 0) edge[warp] = a;
    }
    __syncthreads();
    const int p0 = edge[0], p1 = edge[1];
    for (int b = threadIdx.x; b <= kShare; b += kBinThreads) start[b] = p1;
    __syncthreads();
    // where the bins start; whether the points are in order and in these bins
    bool bad = p1 < p0;
    const int per_warp = p1 > p0 ? ((p1 - p0 + kBinThreads - 1) / kBinThreads) * 32 : 0;
    const int w0 = p0 + warp * per_warp, w1 = min(p1, w0 + per_warp);
    int before = w0 > p0 && w0 < w1 ? bin_of(t[w0 - 1], lo, span) - b0 : -1;   // bin of the point before
    double t_before = w0 < w1 ? t[max(w0 - 1, 0)] : 0.0;
#pragma unroll 2
    for (int i0 = w0; i0 < w1; i0 += 32) {
        const int i = i0 + lane;
        const bool on = i < w1;
        const double ti = t[min(i, w1 - 1)];
        const int b = bin_near(ti, lo, span, per_day) - b0;
        int pb = __shfl_up_sync(0xffffffffu, b, 1);
        double pt = __shfl_up_sync(0xffffffffu, ti, 1);
        if (lane == 0) {
            pb = before;
            pt = t_before;
        }
        const long long k = time_key(ti);
        if (on) {
            bad = bad || time_key(pt) > k || k > kInfKey || k < ~kInfKey || b < 0 || b >= kShare;
            if (!bad)
                for (int q = max(pb, -1) + 1; q <= b; ++q) start[q] = i;
        }
        before = __shfl_sync(0xffffffffu, b, 31);
        t_before = __shfl_sync(0xffffffffu, ti, 31);
        // (for k_bin_any.  256 curves of 46,000 points in random order: 612 us here
        // without the way out, as much as k_bin_any takes)
        if (__any_sync(0xffffffffu, bad)) break;
    }
    if (__syncthreads_or(bad)) {
        if (threadIdx.x == 0) unsorted[lc] = 1u;
        return;
    }
    for (int b = threadIdx.x; b < kShare; b += kBinThreads) {
        const int i1 = start[b + 1];
        int i = start[b];
        double sw = 0.0, swr = 0.0, sum = 0.0;
        long long dy_bits = -1;   // (the bits of a NaN, whose w is one too)
        double w = __longlong_as_double(dy_bits);
        int cnt = 0;
#pragma unroll 4
        for (; i < i1; ++i) {
            const double d = dy[i], r = __dsub_rn(1.0, y[i]);
            if (__double_as_longlong(d) != dy_bits) {
                if (cnt > 0) {
                    swr = __dadd_rn(swr, __dmul_rn(w, sum));
                    sw = __dadd_rn(sw, __dmul_rn(w, (double)cnt));
                }
                cnt = 0;
                sum = 0.0;
                dy_bits = __double_as_longlong(d);
                w = __drcp_rn(__dmul_rn(d, d));
            }
            sum = __dadd_rn(sum, r);
            ++cnt;
        }
        if (cnt > 0) {
            swr = __dadd_rn(swr, __dmul_rn(w, sum));
            sw = __dadd_rn(sw, __dmul_rn(w, (double)cnt));
        }
        const int64_t at = (int64_t)lc * kBins + b0 + b;
        x[at] = sw > 0.0 ? (float)(swr * rsqrt(sw)) : 0.0f;
        if (mean) mean[at] = sw > 0.0 ? (float)(swr / sw) : 0.0f;
        if (wsum) wsum[at] = (float)sw;
    }
}

// Any order of the points; curves that are not flagged return at once.  Its
// sums (64 KB) leave an SM three CTAs: 512 threads each wait less for FP64 and
// the atomics than 256 (256 curves of 46,000 points in random order with a dy
// each: 0.78 against 0.88 ms for the call, 0.81 before k_bin_sorted).
constexpr int kAnyThreads = 512;

__global__ void __cluster_dims__(kBinCtas, 1, 1) __launch_bounds__(kAnyThreads, 3)
k_bin_any(const double* __restrict__ t, const double* __restrict__ y, const double* __restrict__ dy,
          const int64_t* __restrict__ off, float* __restrict__ x, float* __restrict__ mean, float* __restrict__ wsum,
          unsigned int* __restrict__ unsorted)
{
    namespace cg = cooperative_groups;
    extern __shared__ double sb[];   // [kBins] sum w r, [kBins] sum w
    __shared__ long long mn[kAnyThreads / 32], mx[kAnyThreads / 32], range[2];
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int lc = blockIdx.x / kBinCtas;
    if (unsorted[lc] == 0u) return;   // the whole cluster
    const int64_t o = off[lc], n = off[lc + 1] - o;
    t += o;
    y += o;
    dy += o;
    // this CTA's points: whole runs
    const int64_t part = ((n + kBinCtas - 1) / kBinCtas + kBinRun - 1) / kBinRun * kBinRun;
    const int64_t p0 = min(n, rank * part), p1 = min(n, p0 + part);
    for (int b = threadIdx.x; b < 2 * kBins; b += blockDim.x) sb[b] = 0.0;
    long long klo = kInfKey, khi = ~kInfKey;   // +inf, -inf
#pragma unroll 4
    for (int64_t i = p0 + threadIdx.x; i < p1; i += blockDim.x) {
        const long long u = __double_as_longlong(t[i]);
        if ((u & 0x7fffffffffffffffll) > kInfKey) continue;   // NaN
        const long long k = u < 0 ? u ^ 0x7fffffffffffffffll : u;
        klo = k < klo ? k : klo;
        khi = k > khi ? k : khi;
    }
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        const long long a = __shfl_xor_sync(0xffffffffu, klo, s), b = __shfl_xor_sync(0xffffffffu, khi, s);
        klo = a < klo ? a : klo;
        khi = b > khi ? b : khi;
    }
    if ((threadIdx.x & 31) == 0) {
        mn[threadIdx.x >> 5] = klo;
        mx[threadIdx.x >> 5] = khi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kAnyThreads / 32; ++w) {
            klo = mn[w] < klo ? mn[w] : klo;
            khi = mx[w] > khi ? mx[w] : khi;
        }
        range[0] = klo;
        range[1] = khi;
    }
    cluster.sync();
    klo = range[0];
    khi = range[1];
    for (int r = 0; r < kBinCtas; ++r) {
        const long long* const other = cluster.map_shared_rank(range, r);
        klo = other[0] < klo ? other[0] : klo;
        khi = other[1] > khi ? other[1] : khi;
    }
    const double lo = key_time(klo), hi = key_time(khi);
    const double span = __dsub_rn(hi, lo);
    long long dy_bits = -1;   // (the bits of a NaN, whose w is one too)
    double w = __longlong_as_double(dy_bits);
    for (int64_t i0 = p0 + (int64_t)threadIdx.x * kBinRun; i0 < p1; i0 += (int64_t)kAnyThreads * kBinRun) {
        const int len = (int)min((int64_t)kBinRun, p1 - i0);
        int bin = -1, cnt = 0;
        double sum = 0.0;
        for (int u = 0; u < len; ++u) {
            const double d = dy[i0 + u];
            const int b = bin_of(t[i0 + u], lo, span);
            const bool other = __double_as_longlong(d) != dy_bits;
            if (b != bin || other) {
                if (cnt > 0) {
                    atomicAdd(&sb[bin], __dmul_rn(w, sum));
                    atomicAdd(&sb[kBins + bin], __dmul_rn(w, (double)cnt));
                }
                cnt = 0;
                sum = 0.0;
                bin = b;
                if (other) {
                    dy_bits = __double_as_longlong(d);
                    w = __drcp_rn(__dmul_rn(d, d));
                }
            }
            sum = __dadd_rn(sum, __dsub_rn(1.0, y[i0 + u]));
            ++cnt;
        }
        if (cnt > 0) {
            atomicAdd(&sb[bin], __dmul_rn(w, sum));
            atomicAdd(&sb[kBins + bin], __dmul_rn(w, (double)cnt));
        }
    }
    cluster.sync();
    constexpr int kShare = kBins / kBinCtas;
    for (int b = rank * kShare + threadIdx.x; b < (rank + 1) * kShare; b += blockDim.x) {
        double sw = 0.0, swr = 0.0;
        for (int r = 0; r < kBinCtas; ++r) {
            const double* const other = cluster.map_shared_rank(sb, r);
            swr += other[b];
            sw += other[kBins + b];
        }
        x[(int64_t)lc * kBins + b] = sw > 0.0 ? (float)(swr / sqrt(sw)) : 0.0f;
        if (mean) mean[(int64_t)lc * kBins + b] = sw > 0.0 ? (float)(swr / sw) : 0.0f;
        if (wsum) wsum[(int64_t)lc * kBins + b] = (float)sw;
    }
    cluster.sync();   // the others' sums are read before a CTA leaves
    if (rank == 0 && threadIdx.x == 0) unsorted[lc] = 0u;
}

int grid_for(int64_t n)
{
    return (int)std::min<int64_t>(4096, std::max<int64_t>(1, (n + 255) / 256));
}

}  // namespace

struct gtls_cnn {
    int device = -1;
    int max_batch = 0;
    Layout lay;
    float* p = nullptr;       // FP32 master parameters
    bf16* pb = nullptr;       // BF16 copy used by the GEMMs
    float* g = nullptr;       // gradients
    float* m = nullptr;       // Adam moments
    float* v = nullptr;
    int64_t step = 0;
    bf16* act[kConv + 1] = {};   // act[0] input, act[i+1] pooled output of conv i
    uint8_t* arg[kConv] = {};
    float* z = nullptr;
    float* dz = nullptr;
    bf16* dz_b = nullptr;
    float* da[2] = {};        // FP32 gradient of a pooled output (ping-pong)
    double* loss = nullptr;   // [0] loss, [1 ..] the loss blocks' parts
    unsigned int* loss_done = nullptr;
    unsigned int* unsorted = nullptr;   // per curve of a binning call: points out of time order
    int n_sm = 0;
    int64_t* off = nullptr;   // binning offsets (max_batch + 1)
    std::vector<void*> allocs;
};

namespace {

template <class T>
gtls_status cnn_alloc(gtls_cnn* c, T** ptr, int64_t count)
{
    void* q = nullptr;
    const cudaError_t e = cudaMalloc(&q, std::max<int64_t>(count, 1) * sizeof(T));
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return set_error(GTLS_ERR_OOM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
    }
    c->allocs.push_back(q);
    *ptr = static_cast<T*>(q);
    return GTLS_OK;
}

int conv_len(int i) { return kBins >> i; }      // input length of conv i

// Logits into c->z (and the caller's arrays).  `train`: the input and the
// pooling choices are kept for the backward pass.
gtls_status cnn_forward(gtls_cnn* c, const float* x, int B, bool train, float* logits, float* scores, cudaStream_t st)
{
    const int tiles0 = B * (kBins / kRows), grid0 = std::min(tiles0, c->n_sm * 12);
    const bf16* w0 = c->pb + c->lay.w[0];
    const float* b0 = c->p + c->lay.b[0];
    if (train) k_conv0<true><<<grid0, 128, 0, st>>>(x, w0, b0, c->act[0], c->act[1], c->arg[0], tiles0);
    else k_conv0<false><<<grid0, 128, 0, st>>>(x, w0, b0, c->act[0], c->act[1], c->arg[0], tiles0);
    PROP_CUDA(cudaGetLastError());
    for (int i = 1; i < kConv; ++i) {
        ConvArgs a{};
        a.x = c->act[i];
        a.w = c->pb + c->lay.w[i];
        a.bias = c->p + c->lay.b[i];
        a.pooled = c->act[i + 1];
        a.arg = c->arg[i];
        a.L = conv_len(i);
        a.dil = kDil[i];
        a.tiles = B * (a.L / kRows);
        const int grid = std::min(a.tiles, c->n_sm * 3);
        if (train) k_conv<false, true><<<grid, 128, kWBytes + kABytes, st>>>(a);
        else k_conv<false, false><<<grid, 128, kWBytes + kABytes, st>>>(a);
        PROP_CUDA(cudaGetLastError());
    }
    if (train)
        k_head_chain<<<dim3((unsigned)((B + 15) / 16), kReg / 32), 128, 0, st>>>(c->act[kConv], c->pb + c->lay.wh,
                                                                                c->p + c->lay.bh, c->z, B);
    else
        k_head<<<dim3((unsigned)((B + 15) / 16), kReg / 16), 256, 0, st>>>(c->act[kConv], c->pb + c->lay.wh,
                                                                       c->p + c->lay.bh, c->z, logits, scores, B);
    PROP_CUDA(cudaGetLastError());
    return GTLS_OK;
}

gtls_status cnn_backward(gtls_cnn* c, const float* tgt, const float* mask, int B, cudaStream_t st)
{
    const int nz = B * kReg;
    k_loss<<<kLossBlocks, kLossThreads, 0, st>>>(c->z, tgt, mask, nz, c->dz, c->dz_b, c->loss + 1, c->loss_done, c->loss);
    PROP_CUDA(cudaGetLastError());
    // the convolutions' gradients are added up by many blocks
    PROP_CUDA(cudaMemsetAsync(c->g, 0, c->lay.wh * sizeof(float), st));
    k_head_dw<<<kFeat / 32, 256, 0, st>>>(c->dz_b, c->dz, c->act[kConv], c->g + c->lay.wh, c->g + c->lay.bh, B);
    PROP_CUDA(cudaGetLastError());
    k_head_dx<<<dim3((unsigned)((B + 63) / 64), kFeat / 64), 128, 0, st>>>(c->dz_b, c->pb + c->lay.wh, c->da[0], B);
    PROP_CUDA(cudaGetLastError());
    int cur = 0;
    for (int i = kConv - 1; i >= 0; --i) {
        const PoolGrad pg{c->da[cur], c->act[i + 1], c->arg[i]};
        const int tiles = B * (conv_len(i) / kRows);
        if (i == 0) {
            k_conv0_dw<<<std::min(tiles, c->n_sm * 6), 256, 0, st>>>(c->act[0], pg, c->g + c->lay.w[0],
                                                                     c->g + c->lay.b[0], tiles);
            PROP_CUDA(cudaGetLastError());
            break;
        }
        ConvArgs a{};
        a.x = c->act[i];
        a.pg = pg;
        a.w = c->pb + c->lay.w[i];
        a.dx = c->da[cur ^ 1];
        a.L = conv_len(i);
        a.dil = kDil[i];
        a.tiles = tiles;
        k_conv_dw<<<std::min(tiles, c->n_sm), 256, kRows * 128 + kABytes, st>>>(a, c->g + c->lay.w[i],
                                                                               c->g + c->lay.b[i]);
        PROP_CUDA(cudaGetLastError());
        k_conv<true, false><<<std::min(tiles, c->n_sm * 3), 128, kWBytes + kABytes, st>>>(a);
        PROP_CUDA(cudaGetLastError());
        cur ^= 1;
    }
    return GTLS_OK;
}

gtls_status check_batch(const gtls_cnn* c, int B)
{
    if (!c) return set_error(GTLS_ERR_INVALID_ARG, "null network");
    if (B < 1 || B > c->max_batch)
        return set_error(GTLS_ERR_INVALID_ARG, "batch must be in [1, max_batch]");
    int dev = -1;
    PROP_CUDA(cudaGetDevice(&dev));
    if (dev != c->device) return set_error(GTLS_ERR_INVALID_ARG, "current device differs from the network's");
    return GTLS_OK;
}

}  // namespace

extern "C" {

int64_t gtls_cnn_param_count(void)
{
    return Layout().total;
}

gtls_status gtls_cnn_create(int32_t max_batch, const float* params, gtls_cnn** out)
{
    if (!out) return set_error(GTLS_ERR_INVALID_ARG, "null pointer argument");
    *out = nullptr;
    if (max_batch < 1 || max_batch > 4096) return set_error(GTLS_ERR_INVALID_ARG, "max_batch must be in [1, 4096]");
    gtls_cnn* c = new (std::nothrow) gtls_cnn();
    if (!c) return set_error(GTLS_ERR_OOM, "host allocation of the network failed");
    auto bail = [&](gtls_status s) {
        for (void* q : c->allocs) cudaFree(q);
        delete c;
        return s;
    };
    cudaError_t e = cudaGetDevice(&c->device);
    if (e != cudaSuccess) return bail(set_error(GTLS_ERR_CUDA, cudaGetErrorString(e)));
    c->max_batch = max_batch;
    const int64_t np = c->lay.total, B = max_batch;
    gtls_status s = GTLS_OK;
    auto A = [&](auto** ptr, int64_t cnt) {
        if (s == GTLS_OK) s = cnn_alloc(c, ptr, cnt);
    };
    A(&c->p, np);
    A(&c->pb, np);
    A(&c->g, np);
    A(&c->m, np);
    A(&c->v, np);
    A(&c->act[0], B * kBins);
    for (int i = 0; i < kConv; ++i) {
        A(&c->act[i + 1], B * (conv_len(i) / 2) * kCh);
        A(&c->arg[i], B * (conv_len(i) / 2) * kCh);
    }
    A(&c->z, B * kReg);
    A(&c->dz, B * kReg);
    A(&c->dz_b, B * kReg);
    A(&c->da[0], B * (kBins / 2) * kCh);
    A(&c->da[1], B * (kBins / 2) * kCh);
    A(&c->loss, 1 + kLossBlocks);
    A(&c->loss_done, 1);
    A(&c->off, B + 1);
    A(&c->unsorted, B);
    if (s != GTLS_OK) return bail(s);
    std::vector<float> h(np, 0.0f);
    if (params) std::memcpy(h.data(), params, np * sizeof(float));
    if ((e = cudaMemcpy(c->p, h.data(), np * sizeof(float), cudaMemcpyHostToDevice)) != cudaSuccess ||
        (e = cudaMemset(c->m, 0, np * sizeof(float))) != cudaSuccess ||
        (e = cudaMemset(c->v, 0, np * sizeof(float))) != cudaSuccess ||
        (e = cudaMemset(c->loss_done, 0, sizeof(unsigned int))) != cudaSuccess ||
        (e = cudaMemset(c->unsorted, 0, B * sizeof(unsigned int))) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&c->n_sm, cudaDevAttrMultiProcessorCount, c->device)) != cudaSuccess)
        return bail(set_error(GTLS_ERR_CUDA, cudaGetErrorString(e)));
    for (const void* fn : {(const void*)k_conv<false, false>, (const void*)k_conv<false, true>,
                           (const void*)k_conv<true, false>, (const void*)k_conv_dw})
        if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kWBytes + kABytes)) != cudaSuccess)
            return bail(set_error(GTLS_ERR_CUDA, cudaGetErrorString(e)));
    k_to_bf16<<<grid_for(np), 256>>>(c->p, c->pb, np);
    if ((e = cudaDeviceSynchronize()) != cudaSuccess) return bail(set_error(GTLS_ERR_CUDA, cudaGetErrorString(e)));
    if ((e = cudaFuncSetAttribute(k_bin_any, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  2 * kBins * (int)sizeof(double))) != cudaSuccess)
        return bail(set_error(GTLS_ERR_CUDA, cudaGetErrorString(e)));
    *out = c;
    return GTLS_OK;
}

gtls_status gtls_cnn_get_params(const gtls_cnn* c, float* params)
{
    if (!c || !params) return set_error(GTLS_ERR_INVALID_ARG, "null pointer argument");
    PROP_CUDA(cudaMemcpy(params, c->p, c->lay.total * sizeof(float), cudaMemcpyDeviceToHost));
    return GTLS_OK;
}

gtls_status gtls_cnn_set_params(gtls_cnn* c, const float* params)
{
    if (!c || !params) return set_error(GTLS_ERR_INVALID_ARG, "null pointer argument");
    PROP_CUDA(cudaMemcpy(c->p, params, c->lay.total * sizeof(float), cudaMemcpyHostToDevice));
    k_to_bf16<<<grid_for(c->lay.total), 256>>>(c->p, c->pb, c->lay.total);
    PROP_CUDA(cudaGetLastError());
    PROP_CUDA(cudaMemset(c->m, 0, c->lay.total * sizeof(float)));
    PROP_CUDA(cudaMemset(c->v, 0, c->lay.total * sizeof(float)));
    PROP_CUDA(cudaDeviceSynchronize());
    c->step = 0;
    return GTLS_OK;
}

gtls_status gtls_cnn_bin(gtls_cnn* c, const double* t, const double* y, const double* dy,
                         const int64_t* offsets, int64_t n_lc, float* x, float* mean, float* wsum,
                         void* stream)
{
    PROP_TRY(check_batch(c, (int)std::min<int64_t>(n_lc, 1 << 30)));
    if (!t || !y || !dy || !offsets || !x) return set_error(GTLS_ERR_INVALID_ARG, "null pointer argument");
    const int64_t o0 = offsets[0];
    std::vector<int64_t> off(n_lc + 1);
    for (int64_t i = 0; i <= n_lc; ++i) off[i] = offsets[i] - o0;
    for (int64_t i = 0; i < n_lc; ++i)
        if (off[i + 1] - off[i] < 1) return set_error(GTLS_ERR_INVALID_ARG, "every light curve needs a point");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    PROP_CUDA(cudaMemcpyAsync(c->off, off.data(), off.size() * sizeof(int64_t), cudaMemcpyHostToDevice, st));
    const unsigned int ctas = (unsigned)n_lc * kBinCtas;
    k_bin_sorted<<<ctas, kBinThreads, 0, st>>>(t + o0, y + o0, dy + o0, c->off, x, mean, wsum, c->unsorted);
    PROP_CUDA(cudaGetLastError());
    k_bin_any<<<ctas, kAnyThreads, 2 * kBins * sizeof(double), st>>>(t + o0, y + o0, dy + o0, c->off, x, mean, wsum,
                                                                     c->unsorted);
    PROP_CUDA(cudaGetLastError());
    PROP_CUDA(cudaStreamSynchronize(st));   // the offsets live in host memory of this call
    return GTLS_OK;
}

gtls_status gtls_cnn_forward(gtls_cnn* c, const float* x, int32_t batch, float* logits, float* scores,
                             void* stream)
{
    PROP_TRY(check_batch(c, batch));
    if (!x) return set_error(GTLS_ERR_INVALID_ARG, "null input");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    PROP_TRY(cnn_forward(c, x, batch, false, logits, scores, st));
    return GTLS_OK;
}

gtls_status gtls_cnn_gradient(gtls_cnn* c, const float* x, const float* target, const float* mask,
                              int32_t batch, float* grad, double* loss, void* stream)
{
    PROP_TRY(check_batch(c, batch));
    if (!x || !target || !mask) return set_error(GTLS_ERR_INVALID_ARG, "null pointer argument");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    PROP_TRY(cnn_forward(c, x, batch, true, nullptr, nullptr, st));
    PROP_TRY(cnn_backward(c, target, mask, batch, st));
    if (grad) PROP_CUDA(cudaMemcpyAsync(grad, c->g, c->lay.total * sizeof(float), cudaMemcpyDeviceToHost, st));
    if (loss) PROP_CUDA(cudaMemcpyAsync(loss, c->loss, sizeof(double), cudaMemcpyDeviceToHost, st));
    PROP_CUDA(cudaStreamSynchronize(st));
    return GTLS_OK;
}

gtls_status gtls_cnn_train_step(gtls_cnn* c, const float* x, const float* target, const float* mask,
                                int32_t batch, float lr, double* loss, void* stream)
{
    PROP_TRY(check_batch(c, batch));
    if (!x || !target || !mask) return set_error(GTLS_ERR_INVALID_ARG, "null pointer argument");
    if (!(lr > 0.0f)) return set_error(GTLS_ERR_INVALID_ARG, "lr must be > 0");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    PROP_TRY(cnn_forward(c, x, batch, true, nullptr, nullptr, st));
    PROP_TRY(cnn_backward(c, target, mask, batch, st));
    c->step += 1;
    const float c1 = 1.0f - (float)std::pow(0.9, (double)c->step);
    const float c2 = 1.0f - (float)std::pow(0.999, (double)c->step);
    k_adam<<<grid_for(c->lay.total), 256, 0, st>>>(c->p, c->g, c->m, c->v, c->pb, c->lay.total, lr, c1, c2);
    PROP_CUDA(cudaGetLastError());
    if (loss) {
        PROP_CUDA(cudaMemcpyAsync(loss, c->loss, sizeof(double), cudaMemcpyDeviceToHost, st));
        PROP_CUDA(cudaStreamSynchronize(st));
    }
    return GTLS_OK;
}

gtls_status gtls_region_targets(const double* periods, const double* sr, int64_t n_periods, float* target,
                                float* mask)
{
    if (!periods || !sr || !target || !mask || n_periods < 0)
        return set_error(GTLS_ERR_INVALID_ARG, "null pointer argument");
    const double scale = kReg / std::log(kRegionHi / kRegionLo);
    std::fill(target, target + kReg, 0.0f);
    std::fill(mask, mask + kReg, 0.0f);
    std::vector<double> best(kReg, 0.0);
    for (int64_t i = 0; i < n_periods; ++i) {
        const int64_t r = (int64_t)std::floor(scale * std::log(periods[i] / kRegionLo));
        if (r < 0 || r >= kReg) continue;
        best[r] = std::max(best[r], sr[i]);
        mask[r] = 1.0f;
    }
    for (int r = 0; r < kReg; ++r) target[r] = (float)best[r];
    return GTLS_OK;
}

gtls_status gtls_proposal_periods(const double* periods, int64_t n_periods, const float* scores, double frac,
                                  int64_t* idx, int64_t* n_idx)
{
    if (!periods || !scores || !idx || !n_idx || n_periods < 0)
        return set_error(GTLS_ERR_INVALID_ARG, "null pointer argument");
    if (!(frac > 0.0 && frac <= 1.0)) return set_error(GTLS_ERR_INVALID_ARG, "frac must be in (0, 1]");
    const double scale = kReg / std::log(kRegionHi / kRegionLo);
    std::vector<int> reg(n_periods);
    std::vector<char> valid(kReg, 0);
    for (int64_t i = 0; i < n_periods; ++i) {
        const int64_t r = (int64_t)std::floor(scale * std::log(periods[i] / kRegionLo));
        reg[i] = (r < 0 || r >= kReg) ? -1 : (int)r;
        if (reg[i] >= 0) valid[reg[i]] = 1;
    }
    std::vector<int> cand;
    for (int r = 0; r < kReg; ++r)
        if (valid[r]) cand.push_back(r);
    const int k = std::max(1, (int)std::ceil(frac * (double)cand.size()));
    std::stable_sort(cand.begin(), cand.end(), [&](int a, int b) { return scores[a] > scores[b]; });
    std::vector<char> keep(kReg, 0);
    for (int i = 0; i < k && i < (int)cand.size(); ++i) keep[cand[i]] = 1;
    int64_t n = 0;
    for (int64_t i = 0; i < n_periods; ++i)
        if (reg[i] >= 0 && keep[reg[i]]) idx[n++] = i;
    *n_idx = n;
    return GTLS_OK;
}

void gtls_cnn_destroy(gtls_cnn* c)
{
    if (!c) return;
    int cur = -1;
    const bool sw = cudaGetDevice(&cur) == cudaSuccess && cur != c->device && c->device >= 0;
    if (sw) cudaSetDevice(c->device);
    for (void* q : c->allocs) cudaFree(q);
    if (sw) cudaSetDevice(cur);
    delete c;
}

}  // extern "C"
