// 3x3 convolution layers of the warm-start network (no paper counterpart):
// stride 1, zero padding, NHWC, BF16 activations and weights, FP32
// accumulation, taps dil apart (offsets -d, 0, d).
//
//   32 -> 32 channels, forward and input gradient: implicit GEMM on the
//     fifth-generation tensor cores (conv32_tc05_kernel: tcgen05.mma, BF16 in,
//     FP32 accumulators in tensor memory, read back with tcgen05.ld).
//   32 -> 32 channels, weight gradient: a tcgen05 GEMM over the pixels
//     (conv32_wgrad_tc05_kernel).
//   1 -> 32 and 32 -> 1: CUDA cores, four lanes per pixel with eight channels
//     each (edge_*_kernel).
//
// The single layers (sp_conv3x3_*) take and give FP32 gradients; the whole
// network (sp_convnet_fwd, sp_convnet_bwd) keeps its gradients in BF16, as
// autograd does between BF16 activations, with the ReLU masks folded into the
// kernels that produce them.
#include <cuda_bf16.h>

#include <cstdint>
#include <string>

#include "common.cuh"
#include "../../include/warmstart_conv.h"

namespace spx {
namespace {

typedef __nv_bfloat16 bf16;

constexpr int kC = 32;              // channels of the inner layers
constexpr int kMaxDil = 16;         // largest dilation of the taps

// ------------------------------------------------------------------ edge layers
// Four lanes hold a pixel's 32 channels, eight each (an octet: 16 bytes of
// BF16); a warp takes eight consecutive pixels of an image row at a time.  What
// an octet needs of the nine taps (weights, or partial weight gradients) stays
// in 72 registers.  All three kernels are bound by memory: 64 bytes per pixel
// once, against 288 FMAs per pixel (8 x 256 x 256 pixels: 5 us of HBM, 4 us of
// FMA issue).  One thread per pixel or per output instead (2-byte loads, 64
// bytes apart, or a block per 16 rows) took 54 to 267 us forward and 0.72 and
// 1.81 ms for the two weight gradients at that size.
constexpr int kEdgeThreads = 256;

struct EdgeArgs {
    int B, H, W, dil;
    int sign;   // tap (ky, kx) looks at (h + sign (ky - 1) d, w + sign (kx - 1) d)
};

__device__ __forceinline__ void unpack8(uint4 v, float (&f)[8])
{
    const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        f[2 * k] = __uint_as_float(u[k] << 16);
        f[2 * k + 1] = __uint_as_float(u[k] & 0xffff0000u);
    }
}

__device__ __forceinline__ uint4 pack8(const float (&f)[8])
{
    uint32_t u[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const __nv_bfloat162 t = __floats2bfloat162_rn(f[2 * k], f[2 * k + 1]);
        u[k] = *reinterpret_cast<const uint32_t *>(&t);
    }
    return make_uint4(u[0], u[1], u[2], u[3]);
}

// Eight consecutive channels as floats; vec: the address is a multiple of 16
// bytes (else element by element).
__device__ __forceinline__ void load8(const bf16 *p, bool vec, float (&f)[8])
{
    if (vec) {
        unpack8(*reinterpret_cast<const uint4 *>(p), f);
    } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) f[k] = __bfloat162float(p[k]);
    }
}
__device__ __forceinline__ void load8(const float *p, bool vec, float (&f)[8])
{
    if (vec) {
        const float4 a = reinterpret_cast<const float4 *>(p)[0], b = reinterpret_cast<const float4 *>(p)[1];
        f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w;
        f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
    } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) f[k] = p[k];
    }
}

__device__ __forceinline__ float as_float(bf16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float as_float(float v) { return v; }
__device__ __forceinline__ float round_bf16(float v) { return __bfloat162float(__float2bfloat16(v)); }

// The ReLU's mask: a factor of 0 or 1 on the BF16 gradients of the network
// (non-finite values stay non-finite), a selection on the FP32 results.
template <typename OUT>
__device__ __forceinline__ float masked(float v, bool on)
{
    if constexpr (sizeof(OUT) == 2) return __fmul_rn(v, on ? 1.f : 0.f);
    return on ? v : 0.f;
}

// This warp's pixel groups: group k is row k / gw (over B H), columns
// 8 (k % gw) .. + 7.  Calls f(row, h, w, in) with the lane's pixel.
template <typename F>
__device__ __forceinline__ void for_pixels(const EdgeArgs &a, F f)
{
    // the position is carried along: no division per group
    const unsigned gw = (unsigned)(a.W + 7) / 8, step = gridDim.x * (kEdgeThreads / 32);
    const unsigned first = blockIdx.x * (kEdgeThreads / 32) + (threadIdx.x >> 5);
    const unsigned srow = step / gw, sg = step - srow * gw, sh = srow % (unsigned)a.H;
    const int64_t rows = (int64_t)a.B * a.H;
    int64_t row = first / gw;
    unsigned gi = first - (unsigned)row * gw, h = (unsigned)row % (unsigned)a.H;
    while (row < rows) {
        const int w = (int)gi * 8 + (int)((threadIdx.x & 31) >> 2);
        f(row, (int)h, w, w < a.W);
        row += srow; gi += sg; h += sh;
        if (gi >= gw) { gi -= gw; ++row; ++h; }
        if (h >= (unsigned)a.H) h -= (unsigned)a.H;
    }
}

// The offset of a tap's pixel from (row, w) in pixels, and whether it is in the
// image.
__device__ __forceinline__ bool tap_at(const EdgeArgs &a, int tap, int h, int w, int64_t &off)
{
    const int dy = a.sign * (tap / 3 - 1) * a.dil, dx = a.sign * (tap % 3 - 1) * a.dil;
    off = (int64_t)dy * a.W + dx;
    return (unsigned)(h + dy) < (unsigned)a.H && (unsigned)(w + dx) < (unsigned)a.W;
}

// One channel in, 32 out: y[p, c] = bias[c] + sum_tap s[p + off(tap)] w[c][tap]
// (1 -> 32 forward: W [32][9]; sign = 1) or the input gradient of a 32 -> 1
// layer (W [9][32], sign = -1).  S: bf16 or float; ROUND: s rounded to BF16 and
// kept so in sb.  Results BF16 or FP32; relu clamps, gate masks where gate <= 0.
template <typename S, bool ROUND, bool GRAD, typename OUT>
__global__ void __launch_bounds__(kEdgeThreads) edge_out32_kernel(EdgeArgs a, const S *__restrict__ s,
                                                                  const bf16 *__restrict__ wt,
                                                                  const float *__restrict__ bias,
                                                                  const bf16 *__restrict__ gate, int relu,
                                                                  OUT *__restrict__ y, bf16 *__restrict__ sb, int vec)
{
    const int c0 = (threadIdx.x & 3) * 8;
    float wr[9][8], br[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        br[k] = bias ? bias[c0 + k] : 0.f;
#pragma unroll
        for (int t = 0; t < 9; ++t) wr[t][k] = __bfloat162float(GRAD ? wt[t * kC + c0 + k] : wt[(c0 + k) * 9 + t]);
    }
    for_pixels(a, [&](int64_t row, int h, int w, bool in) {
        if (!in) return;
        const int64_t p = row * a.W + w;
        float acc[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) acc[k] = br[k];
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            int64_t off;
            if (!tap_at(a, t, h, w, off)) continue;
            float v = as_float(s[p + off]);
            if (ROUND) v = round_bf16(v);
            if (ROUND && t == 4 && c0 == 0) sb[p] = __float2bfloat16(v);
#pragma unroll
            for (int k = 0; k < 8; ++k) acc[k] = __fmaf_rn(v, wr[t][k], acc[k]);
        }
        if (relu)
#pragma unroll
            for (int k = 0; k < 8; ++k) acc[k] = fmaxf(acc[k], 0.f);
        if (gate) {
            float gt[8];
            load8(gate + p * kC + c0, vec, gt);
#pragma unroll
            for (int k = 0; k < 8; ++k)
                acc[k] = masked<OUT>(acc[k], gt[k] > 0.f);
        }
        OUT *o = y + p * kC + c0;
        if constexpr (sizeof(OUT) == 2) {
            *reinterpret_cast<uint4 *>(o) = pack8(acc);
        } else if (vec) {
            reinterpret_cast<float4 *>(o)[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
            reinterpret_cast<float4 *>(o)[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) o[k] = acc[k];
        }
    });
}

// 32 channels in, one out: y[p] = bias + sum_tap sum_c v[p + off(tap), c] w
// (32 -> 1 forward: W [9][32], sign = 1) or the input gradient of a 1 -> 32
// layer (W [32][9], sign = -1; rounded to BF16 when `round`).  add (may be
// NULL) is added to the result.
template <typename V, bool GRAD>
__global__ void __launch_bounds__(kEdgeThreads) edge_in32_kernel(EdgeArgs a, const V *__restrict__ v,
                                                                 const bf16 *__restrict__ wt,
                                                                 const float *__restrict__ bias, int relu, int round,
                                                                 const bf16 *__restrict__ gate,
                                                                 const float *__restrict__ add, float *__restrict__ y,
                                                                 int vec)
{
    const int c0 = (threadIdx.x & 3) * 8;
    float wr[9][8];
#pragma unroll
    for (int k = 0; k < 8; ++k)
#pragma unroll
        for (int t = 0; t < 9; ++t) wr[t][k] = __bfloat162float(GRAD ? wt[(c0 + k) * 9 + t] : wt[t * kC + c0 + k]);
    const float b0 = bias ? bias[0] : 0.f;
    for_pixels(a, [&](int64_t row, int h, int w, bool in) {
        const int64_t p = row * a.W + w;
        float acc = 0.f;
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            int64_t off;
            if (!in || !tap_at(a, t, h, w, off)) continue;
            float f[8];
            load8(v + (p + off) * kC + c0, vec, f);
#pragma unroll
            for (int k = 0; k < 8; ++k) acc = __fmaf_rn(f[k], wr[t][k], acc);
        }
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        acc += __shfl_xor_sync(0xffffffffu, acc, 2);
        if (in && (threadIdx.x & 3) == 0) {
            acc += b0;
            if (relu) acc = fmaxf(acc, 0.f);
            if (gate && !(__bfloat162float(gate[p]) > 0.f)) acc = 0.f;
            if (round) acc = round_bf16(acc);
            y[p] = add ? add[p] + acc : acc;
        }
    });
}

// Weight gradient of an edge layer: acc[tap][c] = sum_p v[p, c] s[p + off(tap)].
// 1 -> 32: v = g, s = x, sign = 1, dw [32][9], dbias = sum v.  32 -> 1: v = x,
// s = g, sign = -1 (the pixel of g that sees x[p] through the tap), dw [9][32],
// dbias = sum s.  One partial sum per block is added to dw and dbias.
template <typename V, typename S, bool OUT1>
__global__ void __launch_bounds__(kEdgeThreads) edge_wgrad_kernel(EdgeArgs a, const V *__restrict__ v,
                                                                  const S *__restrict__ s, float *__restrict__ dw,
                                                                  float *__restrict__ db, int vec)
{
    __shared__ float part[9 * kC + kC];
    const int lane = threadIdx.x & 31, c0 = (threadIdx.x & 3) * 8;
    for (int k = threadIdx.x; k < 9 * kC + kC; k += kEdgeThreads) part[k] = 0.f;
    __syncthreads();
    float acc[9][8], bsum[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        bsum[k] = 0.f;
#pragma unroll
        for (int t = 0; t < 9; ++t) acc[t][k] = 0.f;
    }
    for_pixels(a, [&](int64_t row, int h, int w, bool in) {
        if (!in) return;
        const int64_t p = row * a.W + w;
        float f[8];
        load8(v + p * kC + c0, vec, f);
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            int64_t off;
            if (!tap_at(a, t, h, w, off)) continue;
            const float x = as_float(s[p + off]);
#pragma unroll
            for (int k = 0; k < 8; ++k) acc[t][k] = __fmaf_rn(x, f[k], acc[t][k]);
            if (OUT1 && t == 4) bsum[0] += x;
        }
        if (!OUT1)
#pragma unroll
            for (int k = 0; k < 8; ++k) bsum[k] += f[k];
    });
    // over the warp's eight pixels, then the block's warps
#pragma unroll
    for (int k = 0; k < 8; ++k) {
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            float r = acc[t][k];
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
            if (lane < 4) atomicAdd(&part[OUT1 ? t * kC + c0 + k : (c0 + k) * 9 + t], r);
        }
        float r = bsum[k];
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
        if (lane < 4 && (!OUT1 || (k == 0 && lane == 0))) atomicAdd(&part[9 * kC + (OUT1 ? 0 : c0 + k)], r);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < 9 * kC + (OUT1 ? 1 : kC); k += kEdgeThreads)
        atomicAdd(k < 9 * kC ? dw + k : db + (k - 9 * kC), part[k]);
}

unsigned edge_blocks(int B, int H, int W, int per_sm)
{
    const int64_t groups = (int64_t)B * H * ((W + 7) / 8);
    int64_t b = (groups + kEdgeThreads / 32 - 1) / (kEdgeThreads / 32);
    if (b > 152 * per_sm) b = 152 * per_sm;
    return (unsigned)(b < 1 ? 1 : b);
}

// ------------------------------------------------------------------ weights
// W'[i, 2-ky, 2-kx, o] = W[o, ky, kx, i] (the input gradient as a forward convolution)
__global__ void flip_weights_kernel(const bf16 *__restrict__ w, bf16 *__restrict__ wf, int cin, int cout)
{
    const int n = cout * 9 * cin;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        const int o = j / (9 * cin), rem = j - o * 9 * cin, tap = rem / cin, i = rem - tap * cin;
        wf[((size_t)i * 9 + (8 - tap)) * cout + o] = w[j];
    }
}

// The network's weights in BF16 from FP32 masters, one block per layer: the
// edge layers as they are, the inner ones as the tensor cores take them
// ([kc][n][8], see below), for the forward and flipped for the input gradient.
constexpr int kMaxLayers = 16;
constexpr int kPackInner = 2 * 9 * kC * kC;   // elements of an inner layer: forward, flipped
constexpr int kPackEdge = 9 * kC;

struct NetWeights {
    const float *w[kMaxLayers];
    int n;
};

__host__ __device__ constexpr size_t pack_at(int n, int k)   // first element of layer k
{
    return k == 0 ? 0 : (size_t)kPackEdge + (size_t)(k - 1) * kPackInner;
}

__global__ void pack_weights_kernel(NetWeights N, bf16 *__restrict__ pack)
{
    const int k = blockIdx.y;
    const float *w = N.w[k];
    bf16 *out = pack + pack_at(N.n, k);
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (k == 0 || k == N.n - 1) {
        if (j < kPackEdge) out[j] = __float2bfloat16(w[j]);
    } else if (j < 9 * kC * kC) {
        // W[o][tap][i]: K = tap 32 + i, n = o; flipped K = (8 - tap) 32 + o, n = i
        const int o = j / (9 * kC), rem = j - o * 9 * kC, tap = rem / kC, i = rem - tap * kC;
        const bf16 v = __float2bfloat16(w[j]);
        const int kf = tap * kC + i, kg = (8 - tap) * kC + o;
        out[((kf >> 3) * kC + o) * 8 + (kf & 7)] = v;
        out[9 * kC * kC + ((kg >> 3) * kC + i) * 8 + (kg & 7)] = v;
    }
}

// ------------------------------------------------------------------ tcgen05
__device__ __forceinline__ uint32_t s_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor: start address, LBO and SBO in 16-byte
// units, the descriptor version of this architecture (bits 46-47 = 1), no
// swizzle (layout type 0), base offset 0.
__host__ __device__ __forceinline__ uint64_t umma_smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}

// Instruction descriptor of kind::f16: D FP32 (bits 4-5 = 1), A and B BF16
// (bits 7-9 and 10-12 = 1), K-major (bits 15, 16 = 0) or MN-major (1), N >> 3 at
// bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t umma_idesc_bf16(uint32_t M, uint32_t N, bool mn_major = false)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | (mn_major ? (1u << 15) | (1u << 16) : 0u) | ((N >> 3) << 17) |
           ((M >> 4) << 24);
}

__device__ __forceinline__ void umma_bf16(uint32_t taddr, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(taddr),
                 "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
                 : "memory");
}

__device__ __forceinline__ void umma_commit(void *mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(s_u32(mbar))
                 : "memory");
}

// Bounded wait for the barrier's phase; false if it did not complete.
__device__ __forceinline__ bool mbar_wait(void *mbar, uint32_t parity)
{
    for (int it = 0; it < (1 << 24); ++it) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok)
                     : "r"(s_u32(mbar)), "r"(parity)
                     : "memory");
        if (ok) return true;
    }
    return false;
}

__device__ __forceinline__ void tmem_load32(uint32_t taddr, uint32_t (&acc)[kC])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
                 "%13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, "
                 "[%32];"
                 : "=r"(acc[0]), "=r"(acc[1]), "=r"(acc[2]), "=r"(acc[3]), "=r"(acc[4]), "=r"(acc[5]),
                   "=r"(acc[6]), "=r"(acc[7]), "=r"(acc[8]), "=r"(acc[9]), "=r"(acc[10]), "=r"(acc[11]),
                   "=r"(acc[12]), "=r"(acc[13]), "=r"(acc[14]), "=r"(acc[15]), "=r"(acc[16]), "=r"(acc[17]),
                   "=r"(acc[18]), "=r"(acc[19]), "=r"(acc[20]), "=r"(acc[21]), "=r"(acc[22]), "=r"(acc[23]),
                   "=r"(acc[24]), "=r"(acc[25]), "=r"(acc[26]), "=r"(acc[27]), "=r"(acc[28]), "=r"(acc[29]),
                   "=r"(acc[30]), "=r"(acc[31])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Warp 0 allocates `cols` columns of tensor memory (a power of two >= 32) and
// thread 0 the completion barrier; call before a __syncthreads.
__device__ __forceinline__ void tc05_begin(uint32_t *tslot, void *mbar, uint32_t cols)
{
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_u32(tslot)), "r"(cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(s_u32(mbar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
}

__device__ __forceinline__ void tc05_end(uint32_t taddr, uint32_t cols)
{
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
    }
}

__device__ __forceinline__ void cp16(uint32_t dst, const void *src, bool in)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16 : 0) : "memory");
}

// Staged operands visible to the tensor cores, then all threads together.
__device__ __forceinline__ void staged_sync()
{
    asm volatile("cp.async.wait_all;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// The 32 -> 32 convolution: a tile is 128 output pixels of one image row as
// D[128 x 32] = sum over the 18 K-steps (9 taps x 2 halves of 16 input
// channels) of A_s[128 x 16] B_s[16 x 32]^T, one tcgen05.mma (kind::f16) per
// step, issued by one thread.
//
// Shared-memory operands use the canonical no-swizzle K-major layout: core
// matrices of 8 rows x 16 bytes stored contiguously (128 bytes), LBO the
// byte distance between core matrices along K, SBO along M (or N).
//   input  xs[cg][row][pixel][8]: channel group cg (8 channels) of the three
//          rows h - d, h, h + d and pixels w0 - d .. w0 + 127 + d.  A tap's
//          A operand is the same array read from another start address:
//          LBO = one channel group (kXRows5 * kXPix5 * 16 B), SBO = 128 B
//          (8 pixels of 16 B).
//   weights wb[kc][n][8]: K = tap 32 + input channel in groups kc of 8,
//          n the output channel; LBO = 32 * 16 B, SBO = 128 B.
//
// A CTA of 128 threads keeps the weights and walks over tiles with two input
// buffers: the copies of the next tile run while the tensor cores work on the
// present one and its epilogue stores it.  Bound by the memory system (64
// bytes in and out per pixel from HBM, three rows per tile from L2); a CTA per
// tile that staged the weights anew, and had nothing to do while its copies
// were under way, took 62 us forward and 97 us for the gradient at 8 x 256 x
// 256 pixels.
constexpr int kTile5 = 128;                  // output pixels of one tile (M)
constexpr int kXPix5 = kTile5 + 2 * kMaxDil;  // staged pixels per row
constexpr int kXRows5 = 3;
constexpr int kXBytes5 = 4 * kXRows5 * kXPix5 * 16;   // 30,720
constexpr int kWBytes5 = 36 * kC * 16;                // 18,432
constexpr int kSmem5 = 2 * kXBytes5 + kWBytes5 + kC * 4 + 16;   // + bias, mbarrier and TMEM address
constexpr uint32_t kTmemCols5 = 32;                   // FP32 accumulators: N = 32 columns

enum WeightForm { kWPacked = 0, kWPlain = 1, kWFlip = 2 };

struct ConvArgs {
    int B, H, W, dil, relu;
    int form;              // WeightForm of w
    const bf16 *w;
    const float *bias;     // may be NULL
    const bf16 *gate;      // may be NULL: results are zeroed where gate <= 0
};

template <typename IN>
__device__ __forceinline__ void stage_tile(const ConvArgs &a, const IN *__restrict__ x, unsigned char *xs, int64_t tile)
{
    const int tiles_w = (a.W + kTile5 - 1) / kTile5;
    const int64_t row = tile / tiles_w;
    const int w0 = (int)(tile - row * tiles_w) * kTile5, h = (int)(row % a.H);
    const int n4 = (kTile5 + 2 * a.dil) * 4;
#pragma unroll
    for (int r = 0; r < kXRows5; ++r) {
        const int hh = h + (r - 1) * a.dil;
        const bool rin = (unsigned)hh < (unsigned)a.H;
        const IN *src = x + ((row + (rin ? (int64_t)(r - 1) * a.dil : 0)) * a.W) * kC;
        for (int i = threadIdx.x; i < n4; i += 128) {
            const int p = i >> 2, cg = i & 3, ww = w0 + p - a.dil;
            const bool in = rin && (unsigned)ww < (unsigned)a.W;
            const IN *s = src + (in ? (int64_t)ww * kC + cg * 8 : 0);
            unsigned char *dst = xs + ((cg * kXRows5 + r) * kXPix5 + p) * 16;
            if constexpr (sizeof(IN) == 2) {
                cp16(s_u32(dst), s, in);
            } else {
                float f[8] = {};
                if (in) load8(s, true, f);
                *reinterpret_cast<uint4 *>(dst) = pack8(f);
            }
        }
    }
}

// IN, OUT: bf16 or float (float input is rounded to BF16 while staged).  Every
// wait is bounded; a CTA whose MMAs did not complete writes NaN, stops, and
// still frees its tensor memory.
template <typename IN, typename OUT>
__global__ void __launch_bounds__(128) conv32_tc05_kernel(ConvArgs a, const IN *__restrict__ x, OUT *__restrict__ y,
                                                          int64_t tiles)
{
    extern __shared__ __align__(128) unsigned char sm5[];
    unsigned char *wsb = sm5 + 2 * kXBytes5;
    float *bias_s = reinterpret_cast<float *>(wsb + kWBytes5);
    unsigned long long *mbar = reinterpret_cast<unsigned long long *>(bias_s + kC);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(mbar + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    tc05_begin(tslot, mbar, kTmemCols5);
    // weights: wb[kc][n][8] = W[n][kc 8 .. kc 8 + 7] (W is [n][tap][i], K = tap 32 + i);
    // flipped for the input gradient: n = i, K = tap' 32 + o, W[o][8 - tap'][i]
    for (int i = threadIdx.x; i < 36 * kC; i += 128) {
        if (a.form == kWPacked) {
            cp16(s_u32(wsb + i * 16), a.w + (size_t)i * 8, true);
            continue;
        }
        const int kc = i / kC, n = i - kc * kC;
        __align__(16) bf16 e[8];
        const int tp = kc >> 2, c0 = (kc & 3) * 8;
#pragma unroll
        for (int j = 0; j < 8; ++j)
            e[j] = a.form == kWFlip ? a.w[((size_t)(c0 + j) * 9 + (8 - tp)) * kC + n] : a.w[(size_t)n * 9 * kC + kc * 8 + j];
        *reinterpret_cast<uint4 *>(wsb + i * 16) = *reinterpret_cast<const uint4 *>(e);
    }
    if (threadIdx.x < kC) bias_s[threadIdx.x] = a.bias ? a.bias[threadIdx.x] : 0.f;
    int64_t tile = blockIdx.x;
    if (tile < tiles) stage_tile(a, x, sm5, tile);
    const int tiles_w = (a.W + kTile5 - 1) / kTile5;
    uint32_t k = 0;
    uint32_t taddr = 0;
    bool done = true;
    for (; tile < tiles && done; tile += gridDim.x, ++k) {
        unsigned char *xs = sm5 + (k & 1) * kXBytes5;
        staged_sync();
        taddr = *tslot;
        if (threadIdx.x == 0) {
            constexpr uint32_t idesc = umma_idesc_bf16(kTile5, kC);
            const uint32_t xbase = s_u32(xs), wbase = s_u32(wsb);
            constexpr uint32_t kGroup = kXRows5 * kXPix5 * 16;   // A: LBO (next 8 channels)
#pragma unroll 1
            for (int s = 0; s < 18; ++s) {
                const int tap = s >> 1, half = s & 1;
                const int ky = tap / 3, kx = tap - 3 * ky;
                const uint32_t a_addr = xbase + (uint32_t)(2 * half) * kGroup + (uint32_t)(ky * kXPix5 * 16) +
                                        (uint32_t)(kx * a.dil) * 16u;
                umma_bf16(taddr, umma_smem_desc(a_addr, kGroup, 128),
                          umma_smem_desc(wbase + (uint32_t)s * 2u * kC * 16u, kC * 16, 128), idesc, (uint32_t)s);
            }
            umma_commit(mbar);
        }
        // the next tile into the other buffer (its MMAs were waited for)
        if (tile + gridDim.x < tiles) stage_tile(a, x, sm5 + ((k + 1) & 1) * kXBytes5, tile + gridDim.x);
        done = mbar_wait(mbar, k & 1);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // accumulators of this warp's 32 pixels: 32 columns (output channels)
        uint32_t acc[kC];
        tmem_load32(taddr + ((uint32_t)(warp * 32) << 16), acc);
        // epilogue: pixel w0 + 32 warp + lane, 32 channels
        const int64_t row = tile / tiles_w;
        const int ww = (int)(tile - row * tiles_w) * kTile5 + warp * 32 + lane;
        if (ww < a.W) {
            const int64_t off = (row * a.W + ww) * kC;
            const float bad = __int_as_float(0x7fc00000);
#pragma unroll
            for (int o = 0; o < kC; o += 8) {
                float f[8], gt[8];
                if (a.gate) load8(a.gate + off + o, true, gt);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    float v = done ? __uint_as_float(acc[o + j]) + bias_s[o + j] : bad;
                    if (a.relu) v = fmaxf(v, 0.f);
                    if (a.gate) v = masked<OUT>(v, gt[j] > 0.f);
                    f[j] = v;
                }
                if constexpr (sizeof(OUT) == 2) {
                    *reinterpret_cast<uint4 *>(y + off + o) = pack8(f);
                } else {
                    reinterpret_cast<float4 *>(y + off + o)[0] = make_float4(f[0], f[1], f[2], f[3]);
                    reinterpret_cast<float4 *>(y + off + o)[1] = make_float4(f[4], f[5], f[6], f[7]);
                }
            }
        }
        done = __syncthreads_and(done) != 0;   // block-uniform: stop at the first failure
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    tc05_end(*tslot, kTmemCols5);
}

// The 32 -> 32 weight gradient on tcgen05:
//   dW[o, (ky, kx), i] = sum_p g[p, o] x[p + off, i],  dbias[o] = sum_p g[p, o]
// as, per ky, D[(kx, o)][i] = sum over pixels of A[(kx, o)][pixel] B[i][pixel]:
// M = 3 shifts kx x 32 output channels (rows 96..127 zero), N = the 32 input
// channels, K = the 128 pixels of a segment of one image row, 16 per MMA.  The
// shifts are on g: for the x at column w of row h + (ky - 1) d, g at column
// w - (kx - 1) d of row h.  Both operands are MN-major: a pixel's channels are
// contiguous, so the staged data are plain 16-byte copies of what is in memory,
// [channel group][pixel][8], and nothing is transposed (core matrices of 8
// pixels x 8 channels, 128 bytes; LBO the distance of 8 pixels, SBO the one of
// 8 channels).  At the end warp kx reads the accumulators of its shift for each
// ky, the block lays them out as dW in shared memory and adds them to dw, and
// its FP32 sums of g to dbias; a block whose MMAs did not complete adds NaN.
//
// Bound by L2 reads (six rows of 64 bytes per pixel and segment).  The operands
// transposed while staged (K-major, 2-byte stores, nine shifted copies of x)
// took 145 us at 8 x 256 x 256 pixels.
constexpr int kWgGroup5 = kTile5 * 16;                 // one channel group: 128 pixels x 16 bytes
constexpr int kWgABytes5 = 16 * kWgGroup5;             // 3 shifts x 4 groups, 4 zero groups
constexpr int kWgBBytes5 = 3 * 4 * kWgGroup5;          // three rows of x
constexpr int kWgSmem5 = kWgABytes5 + kWgBBytes5 + 16; // + mbarrier and TMEM address
constexpr uint32_t kWgCols5 = 128;                     // 3 x 32 columns, as a power of two
constexpr int kWgCtas5 = 3;                            // CTAs per SM
static_assert(9 * kC * kC * 4 <= kWgABytes5 + kWgBBytes5, "dW fits the staging area");

template <typename G>
__global__ void __launch_bounds__(128) conv32_wgrad_tc05_kernel(const bf16 *__restrict__ x, const G *__restrict__ g,
                                                                float *__restrict__ dw, float *__restrict__ db, int B,
                                                                int H, int W, int rows, int dil)
{
    extern __shared__ __align__(128) unsigned char smw[];
    unsigned char *as = smw;
    unsigned char *bs = smw + kWgABytes5;
    unsigned long long *mbar = reinterpret_cast<unsigned long long *>(smw + kWgABytes5 + kWgBBytes5);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(mbar + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    tc05_begin(tslot, mbar, kWgCols5);
    for (int k = threadIdx.x; k < 4 * kTile5; k += 128)
        *reinterpret_cast<uint4 *>(as + 12 * kWgGroup5 + k * 16) = make_uint4(0u, 0u, 0u, 0u);

    float gsum[kC];   // FP32 sums of g over this thread's pixels (bias gradient)
#pragma unroll
    for (int o = 0; o < kC; ++o) gsum[o] = 0.f;
    const int r0 = blockIdx.x * rows, r1 = min(r0 + rows, B * H);
    const int segs = (W + kTile5 - 1) / kTile5;
    bool done = true;
    uint32_t nseg = 0;
    for (int r = r0; r < r1 && done; ++r) {
        const int h = r % H;
        const G *grow = g + (int64_t)r * W * kC;
        for (int sg = 0; sg < segs && done; ++sg, ++nseg) {
            const int w0 = sg * kTile5;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                // A: g shifted by (q - 1) d; B: row h + (q - 1) d of x
                const int hh = h + (q - 1) * dil;
                const bool rin = (unsigned)hh < (unsigned)H;
                const bf16 *xrow = x + ((int64_t)r + (rin ? (q - 1) * dil : 0)) * W * kC;
                for (int i = threadIdx.x; i < 4 * kTile5; i += 128) {
                    const int p = i >> 2, cg = i & 3, w = w0 + p, wg = w - (q - 1) * dil;
                    const bool xin = rin && w < W, gin = w < W && (unsigned)wg < (unsigned)W;
                    cp16(s_u32(bs + (q * 4 + cg) * kWgGroup5 + p * 16), xin ? xrow + (int64_t)w * kC + cg * 8 : x, xin);
                    unsigned char *ad = as + (q * 4 + cg) * kWgGroup5 + p * 16;
                    if constexpr (sizeof(G) == 2) {
                        cp16(s_u32(ad), gin ? grow + (int64_t)wg * kC + cg * 8 : g, gin);
                    } else {
                        float f[8] = {};
                        if (gin) load8(grow + (int64_t)wg * kC + cg * 8, true, f);
                        *reinterpret_cast<uint4 *>(ad) = pack8(f);
                    }
                }
            }
            staged_sync();
            if (threadIdx.x == 0) {
                constexpr uint32_t idesc = umma_idesc_bf16(kTile5, kC, true);
                const uint32_t abase = s_u32(as), bbase = s_u32(bs), taddr = *tslot;
#pragma unroll 1
                for (int k = 0; k < kTile5 / 16; ++k) {
                    const uint64_t adesc = umma_smem_desc(abase + (uint32_t)(k * 256), 128, kWgGroup5);
#pragma unroll 1
                    for (int q = 0; q < 3; ++q)
                        umma_bf16(taddr + (uint32_t)(q * kC), adesc,
                                  umma_smem_desc(bbase + (uint32_t)(q * 4 * kWgGroup5 + k * 256), 128, kWgGroup5), idesc,
                                  (nseg > 0 || k > 0) ? 1u : 0u);
                }
                umma_commit(mbar);
            }
            // meanwhile the sums of g (the unshifted copy; FP32 g from memory)
            if (w0 + (int)threadIdx.x < W) {
#pragma unroll
                for (int cg = 0; cg < 4; ++cg) {
                    float f[8];
                    if constexpr (sizeof(G) == 2)
                        unpack8(*reinterpret_cast<const uint4 *>(as + (4 + cg) * kWgGroup5 + threadIdx.x * 16), f);
                    else
                        load8(grow + (int64_t)(w0 + (int)threadIdx.x) * kC + cg * 8, true, f);
#pragma unroll
                    for (int j = 0; j < 8; ++j) gsum[cg * 8 + j] += f[j];
                }
            }
            // bounded wait for the segment's MMAs before its operands are overwritten
            done = __syncthreads_and(mbar_wait(mbar, nseg & 1u)) != 0;   // block-uniform: stop at the first failure
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        }
    }
    __syncthreads();
    const uint32_t taddr = *tslot;
    const float bad = __int_as_float(0x7fc00000);
    // bias gradient: the warp's sums, one atomic per channel and warp
#pragma unroll
    for (int o = 0; o < kC; ++o) {
        float v = gsum[o];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (lane == 0) atomicAdd(db + o, done ? v : bad);
    }
    // weight gradient: warp kx holds rows o = lane of shift kx
    float *out = reinterpret_cast<float *>(smw);   // dW of this block
#pragma unroll 1
    for (int q = 0; q < 3; ++q) {
        uint32_t acc[kC];
        tmem_load32(taddr + ((uint32_t)(warp * 32) << 16) + (uint32_t)(q * kC), acc);
        if (warp < 3)
#pragma unroll
            for (int i = 0; i < kC; i += 4)
                *reinterpret_cast<float4 *>(out + ((size_t)lane * 9 + q * 3 + warp) * kC + i) =
                    make_float4(__uint_as_float(acc[i]), __uint_as_float(acc[i + 1]), __uint_as_float(acc[i + 2]),
                                __uint_as_float(acc[i + 3]));
    }
    __syncthreads();
    if (nseg > 0)
        for (int k = threadIdx.x; k < 9 * kC * kC; k += 128) atomicAdd(dw + k, done ? out[k] : bad);
    tc05_end(taddr, kWgCols5);
}

}  // namespace

// ------------------------------------------------------------------ launches
namespace {

int sm_count()
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    return sms;
}

template <typename IN, typename OUT>
cudaError_t launch_conv32(const ConvArgs &a, const IN *x, OUT *y, cudaStream_t s)
{
    cudaError_t e = cudaFuncSetAttribute(conv32_tc05_kernel<IN, OUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem5);
    if (e != cudaSuccess) return e;
    const int sms = sm_count();
    if (sms < 1) return cudaErrorUnknown;
    const int64_t tiles = (int64_t)a.B * a.H * ((a.W + kTile5 - 1) / kTile5);
    const int64_t most = 2 * (int64_t)sms;   // resident at once (80 KB of shared memory each)
    conv32_tc05_kernel<IN, OUT><<<(unsigned)(tiles < most ? tiles : most), 128, kSmem5, s>>>(a, x, y, tiles);
    return cudaGetLastError();
}

template <typename G>
cudaError_t launch_wgrad32(int B, int H, int W, int dil, const bf16 *x, const G *g, float *dw, float *db, cudaStream_t s)
{
    cudaError_t e = cudaFuncSetAttribute(conv32_wgrad_tc05_kernel<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, kWgSmem5);
    if (e != cudaSuccess) return e;
    const int sms = sm_count();
    if (sms < 1) return cudaErrorUnknown;
    const int64_t nrows = (int64_t)B * H, target = kWgCtas5 * (int64_t)sms;
    const int rows = (int)((nrows + target - 1) / target);
    const int blocks = (int)((nrows + rows - 1) / rows);
    conv32_wgrad_tc05_kernel<G><<<blocks, 128, kWgSmem5, s>>>(x, g, dw, db, B, H, W, rows, dil);
    return cudaGetLastError();
}

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// The weight gradient of the 1 -> 32 and 32 -> 1 layers has always been limited
// to rows of this many bytes.
bool edge_too_wide(int W, int cin, int cout, int dil)
{
    return sizeof(float) * (size_t)W * cout + sizeof(bf16) * 3 * (size_t)(W + 2 * dil) * cin > 200 * 1024;
}

sp_status check_layer(int32_t B, int32_t H, int32_t W, int32_t cin, int32_t cout, int32_t dilation)
{
    if (B < 1 || H < 1 || W < 1) return record_error(SP_EINVAL, "B, H, W must be >= 1");
    if (dilation < 1 || dilation > kMaxDil) return record_error(SP_EINVAL, "dilation must be 1..16");
    if (!((cin == 32 && (cout == 32 || cout == 1)) || (cin == 1 && cout == 32)))
        return record_error(SP_EINVAL, "supported channels: 1->32, 32->32, 32->1");
    if ((int64_t)B * H * ((W + kTile5 - 1) / kTile5) > 0x7fffffff && cin == 32 && cout == 32)
        return record_error(SP_EINVAL, "too many tiles");
    return SP_OK;
}

}  // namespace
}  // namespace spx

extern "C" {

sp_status sp_conv3x3_fwd(int32_t B, int32_t H, int32_t W, int32_t cin, int32_t cout, int32_t dilation,
                         const void *x, const void *w, const float *bias, int32_t relu, void *y, void *stream)
{
    using namespace spx;
    clear_error();
    sp_status st = check_layer(B, H, W, cin, cout, dilation);
    if (st != SP_OK) return st;
    if (!x || !w || !y) return record_error(SP_EINVAL, "NULL pointer");
    if (!aligned16(x) || !aligned16(w) || !aligned16(y))
        return record_error(SP_EINVAL, "x, w, y must be 16-byte aligned");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const bf16 *xb = static_cast<const bf16 *>(x), *wb = static_cast<const bf16 *>(w);
    const EdgeArgs ea{B, H, W, dilation, 1};
    cudaError_t e;
    if (cin == 32 && cout == 32) {
        e = launch_conv32(ConvArgs{B, H, W, dilation, relu, kWPlain, wb, bias, nullptr}, xb, static_cast<bf16 *>(y), s);
    } else if (cin == 1) {
        edge_out32_kernel<bf16, false, false, bf16><<<edge_blocks(B, H, W, 8), kEdgeThreads, 0, s>>>(
            ea, xb, wb, bias, nullptr, relu, static_cast<bf16 *>(y), nullptr, 1);
        e = cudaGetLastError();
    } else {
        edge_in32_kernel<bf16, false><<<edge_blocks(B, H, W, 8), kEdgeThreads, 0, s>>>(
            ea, xb, wb, bias, relu, 0, nullptr, nullptr, static_cast<float *>(y), 1);
        e = cudaGetLastError();
    }
    return e == cudaSuccess ? SP_OK : record_error(SP_ECUDA, cudaGetErrorString(e));
}

sp_status sp_conv3x3_bwd_data(int32_t B, int32_t H, int32_t W, int32_t cin, int32_t cout, int32_t dilation,
                              const float *g, const void *w, const void *gate, float *dx, void *stream)
{
    using namespace spx;
    clear_error();
    sp_status st = check_layer(B, H, W, cin, cout, dilation);
    if (st != SP_OK) return st;
    if (!g || !w || !dx) return record_error(SP_EINVAL, "NULL pointer");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const bf16 *wb = static_cast<const bf16 *>(w), *gb = static_cast<const bf16 *>(gate);
    const EdgeArgs ea{B, H, W, dilation, -1};
    cudaError_t e;
    if (cin == 32 && cout == 32) {
        if (!aligned16(g) || !aligned16(w) || !aligned16(dx))
            return record_error(SP_EINVAL, "g, w, dx must be 16-byte aligned");
        if (gate && !aligned16(gate)) return record_error(SP_EINVAL, "gate must be 16-byte aligned");
        e = launch_conv32(ConvArgs{B, H, W, dilation, 0, kWFlip, wb, nullptr, gb}, g, dx, s);
    } else if (cin == 32) {
        edge_out32_kernel<float, false, true, float><<<edge_blocks(B, H, W, 8), kEdgeThreads, 0, s>>>(
            ea, g, wb, nullptr, gb, 0, dx, nullptr, aligned16(dx) && aligned16(gate) ? 1 : 0);
        e = cudaGetLastError();
    } else {
        edge_in32_kernel<float, true><<<edge_blocks(B, H, W, 8), kEdgeThreads, 0, s>>>(
            ea, g, wb, nullptr, 0, 0, gb, nullptr, dx, aligned16(g) ? 1 : 0);
        e = cudaGetLastError();
    }
    return e == cudaSuccess ? SP_OK : record_error(SP_ECUDA, cudaGetErrorString(e));
}

sp_status sp_conv3x3_bwd_weight(int32_t B, int32_t H, int32_t W, int32_t cin, int32_t cout, int32_t dilation,
                                const void *x, const float *g, float *dw, float *dbias, void *stream)
{
    using namespace spx;
    clear_error();
    sp_status st = check_layer(B, H, W, cin, cout, dilation);
    if (st != SP_OK) return st;
    if (!x || !g || !dw || !dbias) return record_error(SP_EINVAL, "NULL pointer");
    const bool inner = cin == 32 && cout == 32;
    if (inner && (!aligned16(x) || !aligned16(g))) return record_error(SP_EINVAL, "x, g must be 16-byte aligned");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const bf16 *xb = static_cast<const bf16 *>(x);
    cudaError_t e = cudaMemsetAsync(dw, 0, sizeof(float) * (size_t)cout * 9 * cin, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(dbias, 0, sizeof(float) * (size_t)cout, s);
    if (e != cudaSuccess) return record_error(SP_ECUDA, cudaGetErrorString(e));
    if (inner) {
        e = launch_wgrad32(B, H, W, dilation, xb, g, dw, dbias, s);
    } else {
        if (edge_too_wide(W, cin, cout, dilation))
            return record_error(SP_EINVAL, "image too wide for the weight-gradient kernel");
        const unsigned blocks = edge_blocks(B, H, W, 2);
        if (cin == 1)
            edge_wgrad_kernel<float, bf16, false><<<blocks, kEdgeThreads, 0, s>>>(
                EdgeArgs{B, H, W, dilation, 1}, g, xb, dw, dbias, aligned16(g) ? 1 : 0);
        else
            edge_wgrad_kernel<bf16, float, true><<<blocks, kEdgeThreads, 0, s>>>(
                EdgeArgs{B, H, W, dilation, -1}, xb, g, dw, dbias, aligned16(xb) ? 1 : 0);
        e = cudaGetLastError();
    }
    return e == cudaSuccess ? SP_OK : record_error(SP_ECUDA, cudaGetErrorString(e));
}

sp_status sp_conv3x3_flip_weights(int32_t cin, int32_t cout, const void *w, void *wf, void *stream)
{
    spx::clear_error();
    if (cin < 1 || cout < 1 || !w || !wf) return spx::record_error(SP_EINVAL, "bad arguments");
    const int n = cout * 9 * cin;
    spx::flip_weights_kernel<<<(n + 255) / 256, 256, 0, static_cast<cudaStream_t>(stream)>>>(
        static_cast<const spx::bf16 *>(w), static_cast<spx::bf16 *>(wf), cin, cout);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? SP_OK : spx::record_error(SP_ECUDA, cudaGetErrorString(e));
}

}  // extern "C"

namespace spx {
namespace {

sp_status check_net(int32_t B, int32_t H, int32_t W, int32_t n, const int32_t *dil)
{
    if (n < 2 || n > kMaxLayers || !dil) return record_error(SP_EINVAL, "2 to 16 layers");
    for (int k = 0; k < n; ++k) {
        const sp_status st = check_layer(B, H, W, k == 0 ? 1 : 32, k == n - 1 ? 1 : 32, dil[k]);
        if (st != SP_OK) return st;
    }
    return SP_OK;
}

}  // namespace
}  // namespace spx

extern "C" {

int64_t sp_convnet_pack_elems(int32_t layers)
{
    return layers < 2 || layers > spx::kMaxLayers ? -1 : (int64_t)(spx::pack_at(layers, layers - 1) + spx::kPackEdge);
}

sp_status sp_convnet_fwd(int32_t B, int32_t H, int32_t W, int32_t layers, const int32_t *dilation,
                         const float *const *w, const float *const *bias, const float *z, int32_t keep, void *acts,
                         void *pack, float *out, void *stream)
{
    using namespace spx;
    clear_error();
    sp_status st = check_net(B, H, W, layers, dilation);
    if (st != SP_OK) return st;
    if (!w || !bias || !z || !acts || !pack || !out) return record_error(SP_EINVAL, "NULL pointer");
    NetWeights N;
    N.n = layers;
    for (int k = 0; k < layers; ++k) {
        if (!w[k]) return record_error(SP_EINVAL, "NULL pointer");
        N.w[k] = w[k];
    }
    if (!aligned16(acts) || !aligned16(pack)) return record_error(SP_EINVAL, "acts, pack must be 16-byte aligned");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    bf16 *pk = static_cast<bf16 *>(pack), *act = static_cast<bf16 *>(acts);
    const size_t slab = (size_t)B * H * W * kC;
    bf16 *zb = act + slab * (size_t)(keep ? layers - 1 : 2);   // z as the first layer sees it
    pack_weights_kernel<<<dim3((9 * kC * kC + 255) / 256, layers), 256, 0, s>>>(N, pk);
    edge_out32_kernel<float, true, false, bf16><<<edge_blocks(B, H, W, 8), kEdgeThreads, 0, s>>>(
        EdgeArgs{B, H, W, dilation[0], 1}, z, pk, bias[0], nullptr, 1, act, zb, 1);
    cudaError_t e = cudaGetLastError();
    auto at = [&](int k) { return act + slab * (size_t)(keep ? k : (k & 1)); };   // layer k's activations
    for (int k = 1; k < layers - 1 && e == cudaSuccess; ++k)
        e = launch_conv32(ConvArgs{B, H, W, dilation[k], 1, kWPacked, pk + pack_at(layers, k), bias[k], nullptr}, at(k - 1),
                          at(k), s);
    if (e == cudaSuccess) {
        edge_in32_kernel<bf16, false><<<edge_blocks(B, H, W, 8), kEdgeThreads, 0, s>>>(
            EdgeArgs{B, H, W, dilation[layers - 1], 1}, at(layers - 2), pk + pack_at(layers, layers - 1), bias[layers - 1],
            0, 0, nullptr, z, out, 1);
        e = cudaGetLastError();
    }
    return e == cudaSuccess ? SP_OK : record_error(SP_ECUDA, cudaGetErrorString(e));
}

sp_status sp_convnet_bwd(int32_t B, int32_t H, int32_t W, int32_t layers, const int32_t *dilation, const void *acts,
                         const void *pack, const float *g, void *work, float *dparam, float *dx, void *stream)
{
    using namespace spx;
    clear_error();
    sp_status st = check_net(B, H, W, layers, dilation);
    if (st != SP_OK) return st;
    if (!acts || !pack || !g || !work || !dparam) return record_error(SP_EINVAL, "NULL pointer");
    if (!aligned16(acts) || !aligned16(pack) || !aligned16(work))
        return record_error(SP_EINVAL, "acts, pack, work must be 16-byte aligned");
    if (edge_too_wide(W, 1, 32, dilation[0]) || edge_too_wide(W, 32, 1, dilation[layers - 1]))
        return record_error(SP_EINVAL, "image too wide for the weight-gradient kernel");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const bf16 *pk = static_cast<const bf16 *>(pack), *act = static_cast<const bf16 *>(acts);
    const size_t slab = (size_t)B * H * W * kC;
    bf16 *gk[2] = {static_cast<bf16 *>(work), static_cast<bf16 *>(work) + slab};   // gradients of the activations
    // dparam: per layer dW, then dbias
    auto dw = [&](int k) { return dparam + (k == 0 ? 0 : (size_t)(kPackEdge + kC) + (size_t)(k - 1) * (9 * kC * kC + kC)); };
    auto db = [&](int k) { return dw(k) + (k == 0 || k == layers - 1 ? kPackEdge : 9 * kC * kC); };
    const int L = layers - 1;
    cudaError_t e = cudaMemsetAsync(dparam, 0, sizeof(float) * (size_t)(db(L) + 1 - dparam), s);
    if (e != cudaSuccess) return record_error(SP_ECUDA, cudaGetErrorString(e));
    // last layer: g FP32; the gradient of the activations below gated and in BF16
    edge_wgrad_kernel<bf16, float, true><<<edge_blocks(B, H, W, 2), kEdgeThreads, 0, s>>>(
        EdgeArgs{B, H, W, dilation[L], -1}, act + slab * (size_t)(L - 1), g, dw(L), db(L), 1);
    edge_out32_kernel<float, false, true, bf16><<<edge_blocks(B, H, W, 8), kEdgeThreads, 0, s>>>(
        EdgeArgs{B, H, W, dilation[L], -1}, g, pk + pack_at(layers, L), nullptr, act + slab * (size_t)(L - 1), 0, gk[0], nullptr, 1);
    e = cudaGetLastError();
    int cur = 0;
    for (int k = L - 1; k >= 1 && e == cudaSuccess; --k) {
        const bf16 *below = act + slab * (size_t)(k - 1);
        e = launch_wgrad32(B, H, W, dilation[k], below, gk[cur], dw(k), db(k), s);
        if (e == cudaSuccess)
            e = launch_conv32(ConvArgs{B, H, W, dilation[k], 0, kWPacked, pk + pack_at(layers, k) + 9 * kC * kC, nullptr, below},
                              gk[cur], gk[cur ^ 1], s);
        cur ^= 1;
    }
    if (e == cudaSuccess) {
        edge_wgrad_kernel<bf16, bf16, false><<<edge_blocks(B, H, W, 2), kEdgeThreads, 0, s>>>(
            EdgeArgs{B, H, W, dilation[0], 1}, gk[cur], act + slab * (size_t)L, dw(0), db(0), 1);
        if (dx)
            edge_in32_kernel<bf16, true><<<edge_blocks(B, H, W, 8), kEdgeThreads, 0, s>>>(
                EdgeArgs{B, H, W, dilation[0], -1}, gk[cur], pk, nullptr, 0, 1, nullptr, nullptr, dx, 1);
        e = cudaGetLastError();
    }
    return e == cudaSuccess ? SP_OK : record_error(SP_ECUDA, cudaGetErrorString(e));
}

}  // extern "C"
