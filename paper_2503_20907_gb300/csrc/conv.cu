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
#include <type_traits>

#include "common.cuh"
#include "../../include/warmstart_conv.h"

namespace spx {
namespace {

typedef __nv_bfloat16 bf16;

constexpr int kC = 32;              // channels of the inner layers
constexpr int kMaxDil = 16;         // largest dilation of the taps

// ------------------------------------------------------------------ edge layers
// Four lanes hold a pixel's 32 channels, eight each (an octet: 16 bytes of
// BF16); a warp takes eight consecutive pixels of an image row at a time.  The
// weights come from shared memory (four addresses per warp, no conflicts), which
// leaves the registers to the loads in flight and room for 32 warps per SM; the
// weight gradients keep an octet's 72 partial sums in registers (16 warps).  The
// floor is 5 us of HBM (64 bytes per pixel) and 4 us of FMAs (288 per pixel) at
// 8 x 256 x 256 pixels; measured, one kernel at a time from a cold cache, are 25
// and 27 us out (32 and 37 us with the weights in registers and 16 warps), 41 us
// in (61 us) and 35 and 38 us for the weight gradients: load latency and issue
// slots.  One thread per pixel or per output instead (2-byte loads, 64 bytes
// apart, or a block per 16 rows) took 54 to 267 us forward and 0.72 and 1.81 ms
// for the two weight gradients.
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

// The ReLU: a NaN stays one (fmaxf would take it to 0).
__device__ __forceinline__ float relu_of(float v)
{
    float r;
    asm("max.NaN.f32 %0, %1, 0f00000000;" : "=f"(r) : "f"(v));
    return r;
}

// The ReLU's mask: a factor of 0 or 1 on the BF16 gradients of the network
// (non-finite values stay non-finite), a selection on the FP32 results.
template <typename OUT>
__device__ __forceinline__ float masked(float v, bool on)
{
    if constexpr (sizeof(OUT) == 2) return __fmul_rn(v, on ? 1.f : 0.f);
    return on ? v : 0.f;
}

// This warp's pixel groups: group k is row k / gw (over B H), columns
// 8 (k % gw) .. + 7.  Calls f(inner, row, h, w, in) with the lane's pixel; inner
// (a type) says that all of the group's pixels and their taps are in the image
// and that vectors are aligned (vec): without a test at each tap their loads are
// in flight together.
template <typename F>
__device__ __forceinline__ void for_pixels(const EdgeArgs &a, bool vec, F f)
{
    // the position is carried along: no division per group
    const unsigned gw = (unsigned)(a.W + 7) / 8, step = gridDim.x * (kEdgeThreads / 32);
    const unsigned first = blockIdx.x * (kEdgeThreads / 32) + (threadIdx.x >> 5);
    const unsigned srow = step / gw, sg = step - srow * gw, sh = srow % (unsigned)a.H;
    const int64_t rows = (int64_t)a.B * a.H;
    int64_t row = first / gw;
    unsigned gi = first - (unsigned)row * gw, h = (unsigned)row % (unsigned)a.H;
    while (row < rows) {
        const int w0 = (int)gi * 8, w = w0 + (int)((threadIdx.x & 31) >> 2);
        if (vec && (int)h >= a.dil && (int)h + a.dil < a.H && w0 >= a.dil && w0 + 7 + a.dil < a.W)
            f(std::true_type{}, row, (int)h, w, true);
        else
            f(std::false_type{}, row, (int)h, w, w < a.W);
        row += srow; gi += sg; h += sh;
        if (gi >= gw) { gi -= gw; ++row; ++h; }
        if (h >= (unsigned)a.H) h -= (unsigned)a.H;
    }
}

// The offset of a tap's pixel from (row, w) in pixels, and whether it is in the
// image.
template <typename INNER>
__device__ __forceinline__ bool tap_at(const EdgeArgs &a, INNER, int tap, int h, int w, int64_t &off)
{
    const int dy = a.sign * (tap / 3 - 1) * a.dil, dx = a.sign * (tap % 3 - 1) * a.dil;
    off = (int64_t)dy * a.W + dx;
    return INNER::value || ((unsigned)(h + dy) < (unsigned)a.H && (unsigned)(w + dx) < (unsigned)a.W);
}

// One channel in, 32 out: y[p, c] = bias[c] + sum_tap s[p + off(tap)] w[c][tap]
// (1 -> 32 forward: W [32][9]; sign = 1) or the input gradient of a 32 -> 1
// layer (W [9][32], sign = -1).  S: bf16 or float; ROUND: s rounded to BF16 and
// kept so in sb.  Results BF16 or FP32; relu clamps, gate masks where gate <= 0.
template <typename S, bool ROUND, bool GRAD, typename OUT>
__global__ void __launch_bounds__(kEdgeThreads, 4) edge_out32_kernel(EdgeArgs a, const S *s,
                                                                  const bf16 *wt,
                                                                  const float *bias,
                                                                  const bf16 *gate, int relu,
                                                                  OUT *y, bf16 *sb, int vec)
{
    chain_begin();
    const int c0 = (threadIdx.x & 3) * 8;
    __shared__ __align__(16) float ws[9 * kC];   // [tap][channel]
    for (int i = threadIdx.x; i < 9 * kC; i += kEdgeThreads)
        ws[i] = __bfloat162float(GRAD ? wt[i] : wt[(i % kC) * 9 + i / kC]);
    float br[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) br[k] = bias ? bias[c0 + k] : 0.f;
    __syncthreads();
    for_pixels(a, vec, [&](auto inner, int64_t row, int h, int w, bool in) {
        if (!in) return;
        const int64_t p = row * a.W + w;
        float acc[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) acc[k] = br[k];
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            int64_t off;
            if (!tap_at(a, inner, t, h, w, off)) continue;
            float v = as_float(s[p + off]);
            if (ROUND) v = round_bf16(v);
            if (ROUND && t == 4 && c0 == 0) sb[p] = __float2bfloat16(v);
            float wr[8];
            load8(ws + t * kC + c0, true, wr);
#pragma unroll
            for (int k = 0; k < 8; ++k) acc[k] = __fmaf_rn(v, wr[k], acc[k]);
        }
        if (relu)
#pragma unroll
            for (int k = 0; k < 8; ++k) acc[k] = relu_of(acc[k]);
        if (gate) {
            float gt[8];
            load8(gate + p * kC + c0, inner.value || vec, gt);
#pragma unroll
            for (int k = 0; k < 8; ++k)
                acc[k] = masked<OUT>(acc[k], gt[k] > 0.f);
        }
        OUT *o = y + p * kC + c0;
        if constexpr (sizeof(OUT) == 2) {
            *reinterpret_cast<uint4 *>(o) = pack8(acc);
        } else if (inner.value || vec) {
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
__global__ void __launch_bounds__(kEdgeThreads, 4) edge_in32_kernel(EdgeArgs a, const V *v,
                                                                 const bf16 *wt,
                                                                 const float *bias, int relu, int round,
                                                                 const bf16 *gate,
                                                                 const float *add, float *y,
                                                                 int vec)
{
    chain_begin();
    const int c0 = (threadIdx.x & 3) * 8;
    __shared__ __align__(16) float ws[9 * kC];   // [tap][channel]
    for (int i = threadIdx.x; i < 9 * kC; i += kEdgeThreads)
        ws[i] = __bfloat162float(GRAD ? wt[(i % kC) * 9 + i / kC] : wt[i]);
    __syncthreads();
    const float b0 = bias ? bias[0] : 0.f;
    for_pixels(a, vec, [&](auto inner, int64_t row, int h, int w, bool in) {
        const int64_t p = row * a.W + w;
        float acc = 0.f, acc1 = 0.f;
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            int64_t off;
            if (!in || !tap_at(a, inner, t, h, w, off)) continue;
            float f[8], wr[8];
            load8(v + (p + off) * kC + c0, inner.value || vec, f);
            load8(ws + t * kC + c0, true, wr);
#pragma unroll
            for (int k = 0; k < 8; k += 2) {
                acc = __fmaf_rn(f[k], wr[k], acc);
                acc1 = __fmaf_rn(f[k + 1], wr[k + 1], acc1);
            }
        }
        acc += acc1;
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        acc += __shfl_xor_sync(0xffffffffu, acc, 2);
        if (in && (threadIdx.x & 3) == 0) {
            acc += b0;
            if (relu) acc = relu_of(acc);
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
__global__ void __launch_bounds__(kEdgeThreads, 2) edge_wgrad_kernel(EdgeArgs a, const V *v,
                                                                  const S *s, float *dw,
                                                                  float *db, int vec)
{
    chain_begin();
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
    for_pixels(a, vec, [&](auto inner, int64_t row, int h, int w, bool in) {
        if (!in) return;
        const int64_t p = row * a.W + w;
        float f[8];
        load8(v + p * kC + c0, inner.value || vec, f);
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            int64_t off;
            if (!tap_at(a, inner, t, h, w, off)) continue;
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

// Blocks of an edge kernel: all that are resident at once on this GPU's 152 SMs
// (twice as many forward, whose blocks are short), or one per eight pixel groups.
unsigned edge_blocks(int B, int H, int W, int per_sm)
{
    const int64_t groups = (int64_t)B * H * ((W + 7) / 8);
    int64_t b = (groups + kEdgeThreads / 32 - 1) / (kEdgeThreads / 32);
    if (b > 152 * per_sm) b = 152 * per_sm;
    return (unsigned)(b < 1 ? 1 : b);
}

// ------------------------------------------------------------------ weights
// W'[i, 2-ky, 2-kx, o] = W[o, ky, kx, i] (the input gradient as a forward convolution)
__global__ void flip_weights_kernel(const bf16 *w, bf16 *wf, int cin, int cout)
{
    chain_begin();
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

__global__ void pack_weights_kernel(NetWeights N, bf16 *pack)
{
    chain_begin();
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

// The same operand `bytes` further on (a multiple of 16; shared-memory addresses
// stay below 2^18, so the sum does not leave the address field).
__device__ __forceinline__ uint64_t umma_step(uint64_t desc, uint32_t bytes) { return desc + (bytes >> 4); }

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
// thread 0 the two completion barriers; call before a __syncthreads.
__device__ __forceinline__ void tc05_begin(uint32_t *tslot, unsigned long long *mbar, uint32_t cols)
{
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_u32(tslot)), "r"(cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(s_u32(mbar)) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(s_u32(mbar + 1)) : "memory");
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

__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

// Waits until at most PENDING of this thread's copy groups are under way, makes
// what was staged visible to the tensor cores, and joins the block; true if
// `good` holds for all threads.
template <int PENDING>
__device__ __forceinline__ bool staged_sync(bool good)
{
    asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    good = __syncthreads_and(good) != 0;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    return good;
}

// How the image rows of a 32 -> 32 layer are shared out.  Rows of one residue
// modulo the dilation form a chain: each row of the chain meets its neighbours
// in it, so a CTA that walks along a chain stages every input row once, in a
// ring, instead of three times.  A unit is 128 columns of `rows` successive
// rows of a chain; one CTA per unit.
struct ChainArgs {
    int B, H, W, dil;
    int strips, chains, segs, rows;   // per image: 128-column strips, chains; per chain: segments of `rows`
};

struct Unit {
    int64_t b;
    int h0, n, w0;   // image, first row, rows, first column
};

__device__ __forceinline__ Unit unit_of(const ChainArgs &a, unsigned u)
{
    Unit t;
    const unsigned seg = u % (unsigned)a.segs;
    u /= (unsigned)a.segs;
    const unsigned c = u % (unsigned)a.chains;
    u /= (unsigned)a.chains;
    t.w0 = (int)(u % (unsigned)a.strips) * 128;
    t.b = u / (unsigned)a.strips;
    const int64_t h0 = c + (int64_t)seg * a.rows * a.dil;
    t.n = h0 < a.H ? min(a.rows, (int)((a.H - h0 + a.dil - 1) / a.dil)) : 0;
    t.h0 = (int)h0;
    return t;
}

// Four warps stage, and store the results; a fifth issues the MMAs meanwhile
// (issued by one of the four, they held up the block's next copies: 32 to 35 us
// and 57 us instead of 26 to 28 us and 49 us forward and weight gradient, 8 x 256 x
// 256 pixels).
constexpr int kThreads5 = 160;
constexpr int kTile5 = 128;                   // pixels of a row per tile: M forward, K of the weight gradient
constexpr int kHalo5 = kTile5 + 2 * kMaxDil;  // with the taps on both sides
// Staged rows are [channel group of 8][pixel][8]; a group is 32 bytes longer
// than its pixels, so that the four groups of two pixels, which eight lanes
// write together, lie in different banks.
constexpr int kHaloGroup5 = kHalo5 * 16 + 32;   // 2,592
constexpr int kHaloRow5 = 4 * kHaloGroup5;
constexpr int kTileGroup5 = kTile5 * 16 + 32;   // 2,080
constexpr int kTileRow5 = 4 * kTileGroup5;

// Stages `pixels` pixels of image row (b, h) from column w on (zeros outside the
// image) at dst and, unless NULL, again at copy: 16 bytes per copy, FP32 input
// rounded to BF16 on the way.
template <typename IN>
__device__ __forceinline__ void stage_row(const ChainArgs &a, const IN *x, int64_t b, int h, int w,
                                          int pixels, int group, unsigned char *dst, unsigned char *copy)
{
    const bool rin = (unsigned)h < (unsigned)a.H;
    const IN *src = x + ((b * a.H + (rin ? h : 0)) * a.W) * kC;
    const int cg = threadIdx.x & 3;
    for (int p = threadIdx.x >> 2; p < pixels; p += 32) {
        const bool in = rin && (unsigned)(w + p) < (unsigned)a.W;
        const IN *s = src + (in ? (int64_t)(w + p) * kC + cg * 8 : 0);
        const int at = cg * group + p * 16;
        if constexpr (sizeof(IN) == 2) {
            cp16(s_u32(dst + at), s, in);
            if (copy) cp16(s_u32(copy + at), s, in);
        } else {
            float f[8] = {};
            if (in) load8(s, true, f);
            const uint4 v = pack8(f);
            *reinterpret_cast<uint4 *>(dst + at) = v;
            if (copy) *reinterpret_cast<uint4 *>(copy + at) = v;
        }
    }
}

// The 32 -> 32 convolution: a tile is 128 output pixels of one image row as
// D[128 x 32] = sum over the 18 K-steps (9 taps x 2 halves of 16 input
// channels) of A_s[128 x 16] B_s[16 x 32]^T, one tcgen05.mma (kind::f16) per
// step, issued by one thread.
//
// Shared-memory operands use the canonical no-swizzle K-major layout: core
// matrices of 8 rows x 16 bytes stored contiguously (128 bytes), LBO the
// byte distance between core matrices along K, SBO along M (or N).
//   input  a ring of staged rows, pixels w0 - d .. w0 + 127 + d.  A tap's A
//          operand is its row read from another pixel on: LBO = one channel
//          group, SBO = 128 B (8 pixels of 16 B).
//   weights wb[kc][n][8]: K = tap 32 + input channel in groups kc of 8,
//          n the output channel; LBO = 32 * 16 B, SBO = 128 B.
//
// Three CTAs of 160 threads per SM, each with its weights, a ring of five rows
// and two accumulators: while the tensor cores work on a tile, the block stores
// the one before and copies the row two tiles ahead.  Bound by the latency of a
// tile's chain (copies, MMAs, read-back, stores; 64 bytes in and out per pixel
// at 2.6 TB/s): 26 us forward and 28 us for the gradient at 8 x 256 x 256
// pixels.  A CTA per tile, staging the weights and all three rows anew, took 62
// and 97 us; several tiles per CTA but three rows per tile 50 and 60 us.
constexpr int kRing5 = 5;
constexpr int kWBytes5 = 36 * kC * 16;   // 18,432
constexpr int kSmem5 = kRing5 * kHaloRow5 + kWBytes5 + kC * 4 + 24;   // + bias, barriers and TMEM address
constexpr int kCtas5 = 3;                // per SM
constexpr uint32_t kTmemCols5 = 64;      // two accumulators of 32 columns

enum WeightForm { kWPacked = 0, kWPlain = 1, kWFlip = 2 };

struct ConvArgs {
    int relu, form;        // form: WeightForm of w
    const bf16 *w;
    const float *bias;     // may be NULL
    const bf16 *gate;      // may be NULL: results are masked where gate <= 0
};

// IN, OUT: bf16 or float (float input is rounded to BF16 while staged).  Every
// wait is bounded; when MMAs do not complete, the rest of the unit is NaN and
// the block still frees its tensor memory.
template <typename IN, typename OUT>
__global__ void __launch_bounds__(kThreads5) conv32_tc05_kernel(ChainArgs ch, ConvArgs a, const IN *x,
                                                          OUT *y)
{
    chain_begin();
    extern __shared__ __align__(128) unsigned char sm5[];
    unsigned char *wsb = sm5 + kRing5 * kHaloRow5;
    float *bias_s = reinterpret_cast<float *>(wsb + kWBytes5);
    unsigned long long *mbar = reinterpret_cast<unsigned long long *>(bias_s + kC);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(mbar + 2);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const Unit u = unit_of(ch, blockIdx.x);
    if (u.n < 1) return;

    tc05_begin(tslot, mbar, kTmemCols5);
    // weights: wb[kc][n][8] = W[n][kc 8 .. kc 8 + 7] (W is [n][tap][i], K = tap 32 + i);
    // flipped for the input gradient: n = i, K = tap' 32 + o, W[o][8 - tap'][i]
    for (int i = threadIdx.x; i < 36 * kC; i += kThreads5) {
        const int kc = i / kC, n = i - kc * kC;
        if (a.form != kWFlip) {
            cp16(s_u32(wsb + i * 16), a.w + (a.form == kWPacked ? (size_t)i * 8 : (size_t)n * 9 * kC + kc * 8), true);
            continue;
        }
        __align__(16) bf16 e[8];
        const int tp = kc >> 2, c0 = (kc & 3) * 8;
#pragma unroll
        for (int j = 0; j < 8; ++j) e[j] = a.w[((size_t)(c0 + j) * 9 + (8 - tp)) * kC + n];
        *reinterpret_cast<uint4 *>(wsb + i * 16) = *reinterpret_cast<const uint4 *>(e);
    }
    if (threadIdx.x < kC) bias_s[threadIdx.x] = a.bias ? a.bias[threadIdx.x] : 0.f;
    // staged row j is image row h0 + (j - 1) d; tile k takes rows k, k + 1, k + 2.  One copy
    // group per row, empty past the last.
    auto stage = [&](int j) {
        if (warp < 4 && j < u.n + 2)
            stage_row(ch, x, u.b, u.h0 + (j - 1) * ch.dil, u.w0 - ch.dil, kTile5 + 2 * ch.dil, kHaloGroup5,
                      sm5 + (j % kRing5) * kHaloRow5, nullptr);
        cp_commit();
    };
    for (int j = 0; j < kRing5; ++j) stage(j);
    bool good = true;
    uint32_t taddr = 0;
    for (int k = 0; k <= u.n; ++k) {
        if (k < u.n) {
            good = staged_sync<kRing5 - 4>(good);   // rows up to k + 2 are there
            taddr = *tslot;
            if (good && threadIdx.x == 128) {
                constexpr uint32_t idesc = umma_idesc_bf16(kTile5, kC);
                const uint32_t d = taddr + (uint32_t)(k & 1) * kC;
                const uint64_t wdesc = umma_smem_desc(s_u32(wsb), kC * 16, 128);
#pragma unroll
                for (int ky = 0; ky < 3; ++ky) {
                    const uint64_t row = umma_smem_desc(s_u32(sm5) + (uint32_t)((k + ky) % kRing5) * kHaloRow5, kHaloGroup5, 128);
#pragma unroll
                    for (int kx = 0; kx < 3; ++kx)
#pragma unroll
                        for (int half = 0; half < 2; ++half) {
                            const uint32_t s = (uint32_t)((ky * 3 + kx) * 2 + half);
                            umma_bf16(d, umma_step(row, 2u * half * kHaloGroup5 + (uint32_t)(kx * ch.dil) * 16u),
                                      umma_step(wdesc, s * 2u * kC * 16u), idesc, s);
                        }
                }
                umma_commit(mbar + (k & 1));
            }
        }
        if (k == 0) continue;
        const int t = k - 1;   // the tile whose MMAs end next; its first row then makes room
        const int w = u.w0 + warp * 32 + lane;   // this thread's pixel (the fifth warp has none)
        const bool mine = warp < 4 && w < ch.W;
        const int64_t off = ((u.b * ch.H + u.h0 + t * ch.dil) * ch.W + w) * kC;
        uint4 gate[4] = {};
        if (a.gate && mine)
#pragma unroll
            for (int j = 0; j < 4; ++j) gate[j] = reinterpret_cast<const uint4 *>(a.gate + off)[j];
        if (good) good = mbar_wait(mbar + (t & 1), (uint32_t)(t >> 1) & 1u);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        stage(t + kRing5);
        if (warp == 4) continue;
        // accumulators of this warp's 32 pixels: 32 columns (output channels)
        uint32_t acc[kC];
        __syncwarp();
        tmem_load32(taddr + ((uint32_t)(warp * 32) << 16) + (uint32_t)(t & 1) * kC, acc);
        if (mine) {
            const float bad = __int_as_float(0x7fc00000);
#pragma unroll
            for (int o = 0; o < kC; o += 8) {
                float f[8], gt[8], bv[8];
                if (a.gate) unpack8(gate[o / 8], gt);
                load8(bias_s + o, true, bv);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    float v = __uint_as_float(acc[o + j]) + bv[j];
                    if (a.relu) v = relu_of(v);
                    if (a.gate) v = masked<OUT>(v, gt[j] > 0.f);
                    f[j] = good ? v : bad;
                }
                if constexpr (sizeof(OUT) == 2) {
                    *reinterpret_cast<uint4 *>(y + off + o) = pack8(f);
                } else {
                    reinterpret_cast<float4 *>(y + off + o)[0] = make_float4(f[0], f[1], f[2], f[3]);
                    reinterpret_cast<float4 *>(y + off + o)[1] = make_float4(f[4], f[5], f[6], f[7]);
                }
            }
        }
    }
    tc05_end(taddr, kTmemCols5);
}

// The 32 -> 32 weight gradient on tcgen05:
//   dW[o, (ky, kx), i] = sum_p g[p, o] x[p + off, i],  dbias[o] = sum_p g[p, o]
// as, per kx, D[(ky, i)][o] = sum over pixels of A[(ky, i)][pixel] B[o][pixel]:
// M = 3 rows of x x 32 input channels (a fourth row of the ring rides along
// unused), N = the 32 output channels, K = the 128 pixels of a tile of one image
// row, 16 per MMA.  For the x at column w of row h + (ky - 1) d, g at column
// w - (kx - 1) d of row h: the staged row of g read from another pixel on.  Both
// operands are MN-major: a pixel's channels are contiguous, so what is staged is
// a plain copy of memory and nothing is transposed (core matrices of 8 pixels x
// 8 channels, 128 bytes; LBO the distance of 8 pixels, SBO the one of 8
// channels).  A's rows must lie in a row: the ring of six rows of x has its first
// three again behind the sixth.  At the end warp ky adds the accumulators of its
// row to dw, 32 input channels at a time, and the block its FP32 sums of g to
// dbias; a block whose MMAs did not complete adds NaN.
//
// Bound by the chain of a tile (copies, MMAs, sums of g, about 1 us each for 16
// tiles per CTA): 38 us at 8 x 256 x 256 pixels.  The operands transposed while
// staged (K-major, 2-byte stores, nine shifted copies of x) took 145 us, three
// rows of x and three shifted copies of g per tile 99 us.
constexpr int kWgRing5 = 6, kWgG5 = 3;                 // staged rows of x (and 3 again) and of g
constexpr int kWgABytes5 = (kWgRing5 + 3) * kTileRow5;
constexpr int kWgSmem5 = kWgABytes5 + kWgG5 * kHaloRow5 + 24;   // + barriers and TMEM address
constexpr uint32_t kWgCols5 = 128;                     // 3 x 32 columns, as a power of two
constexpr int kWgCtas5 = 2;                            // CTAs per SM

template <typename G>
__global__ void __launch_bounds__(kThreads5) conv32_wgrad_tc05_kernel(ChainArgs ch, const bf16 *x,
                                                                const G *g, float *dw,
                                                                float *db)
{
    chain_begin();
    extern __shared__ __align__(128) unsigned char smw[];
    __shared__ float bias_s[4][kC];
    unsigned char *gs = smw + kWgABytes5;
    unsigned long long *mbar = reinterpret_cast<unsigned long long *>(gs + kWgG5 * kHaloRow5);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(mbar + 2);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, cg = threadIdx.x & 3;
    const Unit u = unit_of(ch, blockIdx.x);
    if (u.n < 1) return;

    tc05_begin(tslot, mbar, kWgCols5);
    // copy group j: row j of x (image row h0 + (j - 1) d) and row j - 3 of g (h0 + (j - 3) d).
    // Tile k takes rows k .. k + 2 of x and row k of g, and its MMAs read row k + 3 of x.
    auto stage = [&](int j) {
        if (warp < 4 && j < u.n + 2) {
            const int slot = j % kWgRing5;
            stage_row(ch, x, u.b, u.h0 + (j - 1) * ch.dil, u.w0, kTile5, kTileGroup5, smw + slot * kTileRow5,
                      slot < 3 ? smw + (kWgRing5 + slot) * kTileRow5 : nullptr);
        }
        if (warp < 4 && j >= 3 && j < u.n + 3)
            stage_row(ch, g, u.b, u.h0 + (j - 3) * ch.dil, u.w0 - ch.dil, kTile5 + 2 * ch.dil, kHaloGroup5,
                      gs + (j % kWgG5) * kHaloRow5, nullptr);
        cp_commit();
    };
    for (int j = 0; j < kWgRing5; ++j) stage(j);

    float gsum[8];   // FP32 sums of g over this thread's pixels, channels 8 cg .. (bias gradient)
#pragma unroll
    for (int o = 0; o < 8; ++o) gsum[o] = 0.f;
    bool good = true;
    uint32_t taddr = 0;
    for (int k = 0; k <= u.n; ++k) {
        if (k < u.n) {
            good = staged_sync<1>(good);   // groups up to k + 3 are there
            taddr = *tslot;
            const unsigned char *grow = gs + (k % kWgG5) * kHaloRow5;
            if (good && threadIdx.x == 128) {
                constexpr uint32_t idesc = umma_idesc_bf16(kTile5, kC, true);
                const uint64_t adesc = umma_smem_desc(s_u32(smw) + (uint32_t)(k % kWgRing5) * kTileRow5, 128, kTileGroup5);
                const uint64_t gdesc = umma_smem_desc(s_u32(grow), 128, kHaloGroup5);
#pragma unroll
                for (int s = 0; s < kTile5 / 16; ++s)
#pragma unroll
                    for (int kx = 0; kx < 3; ++kx)
                        umma_bf16(taddr + (uint32_t)(kx * kC), umma_step(adesc, (uint32_t)s * 256u),
                                  umma_step(gdesc, (uint32_t)s * 256u + (uint32_t)((2 - kx) * ch.dil) * 16u), idesc,
                                  (k > 0 || s > 0) ? 1u : 0u);
                umma_commit(mbar + (k & 1));
            }
            // meanwhile the sums of g (FP32 g from memory)
            for (int p = threadIdx.x >> 2; warp < 4 && p < kTile5 && u.w0 + p < ch.W; p += 32) {
                float f[8];
                if constexpr (sizeof(G) == 2)
                    unpack8(*reinterpret_cast<const uint4 *>(grow + cg * kHaloGroup5 + (p + ch.dil) * 16), f);
                else
                    load8(g + ((u.b * ch.H + u.h0 + k * ch.dil) * ch.W + u.w0 + p) * kC + cg * 8, true, f);
#pragma unroll
                for (int j = 0; j < 8; ++j) gsum[j] += f[j];
            }
        }
        if (k == 0) continue;
        if (good) good = mbar_wait(mbar + ((k - 1) & 1), (uint32_t)((k - 1) >> 1) & 1u);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        stage(k - 1 + kWgRing5);
    }
    good = __syncthreads_and(good) != 0;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const float bad = __int_as_float(0x7fc00000);
    // bias gradient: the warps' sums, then one 128-byte addition per block (every block adds to
    // the same line: one atomic per channel and warp took 15 us at 8 x 256 x 256 pixels)
#pragma unroll
    for (int o = 0; o < 8; ++o) {
        float v = gsum[o];
#pragma unroll
        for (int off = 4; off < 32; off <<= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (warp < 4 && lane < 4) bias_s[warp][cg * 8 + o] = v;
    }
    __syncthreads();
    if (warp == 4) {
        const float v = (bias_s[0][lane] + bias_s[1][lane]) + (bias_s[2][lane] + bias_s[3][lane]);
        atomicAdd(db + lane, good ? v : bad);
    }
    // weight gradient: warp ky holds rows i = lane of the row ky of x
#pragma unroll 1
    for (int kx = 0; kx < 3 && warp < 3; ++kx) {
        uint32_t acc[kC];
        tmem_load32(taddr + ((uint32_t)(warp * 32) << 16) + (uint32_t)(kx * kC), acc);
#pragma unroll
            for (int o = 0; o < kC; ++o)
                atomicAdd(dw + ((size_t)o * 9 + warp * 3 + kx) * kC + lane, good ? __uint_as_float(acc[o]) : bad);
    }
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

// Segments per chain: as many units as keep all slots (resident CTAs) busy, with
// as few starts as possible; a start costs about `start` rows (copies until the
// first tile can begin, and the end of the block).
ChainArgs share_out(int B, int H, int W, int dil, int64_t slots, int start, unsigned &units)
{
    ChainArgs c{B, H, W, dil, (W + kTile5 - 1) / kTile5, dil < H ? dil : H, 1, 1};
    const int64_t len = (H + c.chains - 1) / c.chains, base = (int64_t)B * c.strips * c.chains;
    int64_t best = -1;
    for (int waves = 1; waves <= 3; ++waves) {   // the most segments that so many waves hold
        int64_t segs = waves * slots / base;
        segs = segs < 1 ? 1 : segs > len ? len : segs;
        const int64_t rows = (len + segs - 1) / segs, cost = (base * segs + slots - 1) / slots * (rows + start);
        if (best < 0 || cost < best) { best = cost; c.segs = (int)((len + rows - 1) / rows); c.rows = (int)rows; }
    }
    units = (unsigned)(base * c.segs);
    return c;
}

template <typename IN, typename OUT>
cudaError_t launch_conv32(int B, int H, int W, int dil, const ConvArgs &a, const IN *x, OUT *y, cudaStream_t s)
{
    cudaError_t e = cudaFuncSetAttribute(conv32_tc05_kernel<IN, OUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem5);
    if (e != cudaSuccess) return e;
    const int sms = sm_count();
    if (sms < 1) return cudaErrorUnknown;
    unsigned units;
    const ChainArgs c = share_out(B, H, W, dil, kCtas5 * (int64_t)sms, 4, units);
    launch_chained(conv32_tc05_kernel<IN, OUT>, units, kThreads5, kSmem5, s, c, a, x, y);
    return cudaGetLastError();
}

template <typename G>
cudaError_t launch_wgrad32(int B, int H, int W, int dil, const bf16 *x, const G *g, float *dw, float *db, cudaStream_t s)
{
    cudaError_t e = cudaFuncSetAttribute(conv32_wgrad_tc05_kernel<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, kWgSmem5);
    if (e != cudaSuccess) return e;
    const int sms = sm_count();
    if (sms < 1) return cudaErrorUnknown;
    unsigned units;
    const ChainArgs c = share_out(B, H, W, dil, kWgCtas5 * (int64_t)sms, 6, units);
    launch_chained(conv32_wgrad_tc05_kernel<G>, units, kThreads5, kWgSmem5, s, c, x, g, dw, db);
    return cudaGetLastError();
}

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// Rows that the entry points of the weight gradient of the 1 -> 32 and 32 -> 1
// layers refuse (warmstart_conv.h): a limit of the interface, whose first kernels
// staged whole rows in shared memory; the present ones hold none.
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
        e = launch_conv32(B, H, W, dilation, ConvArgs{relu, kWPlain, wb, bias, nullptr}, xb, static_cast<bf16 *>(y), s);
    } else if (cin == 1) {
        launch_chained(edge_out32_kernel<bf16, false, false, bf16>, edge_blocks(B, H, W, 8), kEdgeThreads, 0, s, ea, xb, wb, bias, nullptr, relu, static_cast<bf16 *>(y), nullptr, 1);
        e = cudaGetLastError();
    } else {
        launch_chained(edge_in32_kernel<bf16, false>, edge_blocks(B, H, W, 8), kEdgeThreads, 0, s, ea, xb, wb, bias, relu, 0, nullptr, nullptr, static_cast<float *>(y), 1);
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
        e = launch_conv32(B, H, W, dilation, ConvArgs{0, kWFlip, wb, nullptr, gb}, g, dx, s);
    } else if (cin == 32) {
        launch_chained(edge_out32_kernel<float, false, true, float>, edge_blocks(B, H, W, 8), kEdgeThreads, 0, s, ea, g, wb, nullptr, gb, 0, dx, nullptr, aligned16(dx) && aligned16(gate) ? 1 : 0);
        e = cudaGetLastError();
    } else {
        launch_chained(edge_in32_kernel<float, true>, edge_blocks(B, H, W, 8), kEdgeThreads, 0, s, ea, g, wb, nullptr, 0, 0, gb, nullptr, dx, aligned16(g) ? 1 : 0);
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
            launch_chained(edge_wgrad_kernel<float, bf16, false>, blocks, kEdgeThreads, 0, s, EdgeArgs{B, H, W, dilation, 1}, g, xb, dw, dbias, aligned16(g) ? 1 : 0);
        else
            launch_chained(edge_wgrad_kernel<bf16, float, true>, blocks, kEdgeThreads, 0, s, EdgeArgs{B, H, W, dilation, -1}, xb, g, dw, dbias, aligned16(xb) ? 1 : 0);
        e = cudaGetLastError();
    }
    return e == cudaSuccess ? SP_OK : record_error(SP_ECUDA, cudaGetErrorString(e));
}

sp_status sp_conv3x3_flip_weights(int32_t cin, int32_t cout, const void *w, void *wf, void *stream)
{
    spx::clear_error();
    if (cin < 1 || cout < 1 || !w || !wf) return spx::record_error(SP_EINVAL, "bad arguments");
    const int n = cout * 9 * cin;
    spx::launch_chained(spx::flip_weights_kernel, (n + 255) / 256, 256, 0, static_cast<cudaStream_t>(stream), static_cast<const spx::bf16 *>(w), static_cast<spx::bf16 *>(wf), cin, cout);
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
    launch_chained(pack_weights_kernel, dim3((9 * kC * kC + 255) / 256, layers), 256, 0, s, N, pk);
    launch_chained(edge_out32_kernel<float, true, false, bf16>, edge_blocks(B, H, W, 8), kEdgeThreads, 0, s, EdgeArgs{B, H, W, dilation[0], 1}, z, pk, bias[0], nullptr, 1, act, zb, 1);
    cudaError_t e = cudaGetLastError();
    auto at = [&](int k) { return act + slab * (size_t)(keep ? k : (k & 1)); };   // layer k's activations
    for (int k = 1; k < layers - 1 && e == cudaSuccess; ++k)
        e = launch_conv32(B, H, W, dilation[k], ConvArgs{1, kWPacked, pk + pack_at(layers, k), bias[k], nullptr}, at(k - 1),
                          at(k), s);
    if (e == cudaSuccess) {
        launch_chained(edge_in32_kernel<bf16, false>, edge_blocks(B, H, W, 8), kEdgeThreads, 0, s, EdgeArgs{B, H, W, dilation[layers - 1], 1}, at(layers - 2), pk + pack_at(layers, layers - 1), bias[layers - 1],
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
    launch_chained(edge_wgrad_kernel<bf16, float, true>, edge_blocks(B, H, W, 2), kEdgeThreads, 0, s, EdgeArgs{B, H, W, dilation[L], -1}, act + slab * (size_t)(L - 1), g, dw(L), db(L), 1);
    launch_chained(edge_out32_kernel<float, false, true, bf16>, edge_blocks(B, H, W, 8), kEdgeThreads, 0, s, EdgeArgs{B, H, W, dilation[L], -1}, g, pk + pack_at(layers, L), nullptr, act + slab * (size_t)(L - 1), 0, gk[0], nullptr, 1);
    e = cudaGetLastError();
    int cur = 0;
    for (int k = L - 1; k >= 1 && e == cudaSuccess; --k) {
        const bf16 *below = act + slab * (size_t)(k - 1);
        e = launch_wgrad32(B, H, W, dilation[k], below, gk[cur], dw(k), db(k), s);
        if (e == cudaSuccess)
            e = launch_conv32(B, H, W, dilation[k], ConvArgs{0, kWPacked, pk + pack_at(layers, k) + 9 * kC * kC, nullptr, below},
                              gk[cur], gk[cur ^ 1], s);
        cur ^= 1;
    }
    if (e == cudaSuccess) {
        launch_chained(edge_wgrad_kernel<bf16, bf16, false>, edge_blocks(B, H, W, 2), kEdgeThreads, 0, s, EdgeArgs{B, H, W, dilation[0], 1}, gk[cur], act + slab * (size_t)L, dw(0), db(0), 1);
        if (dx)
            launch_chained(edge_in32_kernel<bf16, true>, edge_blocks(B, H, W, 8), kEdgeThreads, 0, s, EdgeArgs{B, H, W, dilation[0], -1}, gk[cur], pk, nullptr, 0, 1, nullptr, nullptr, dx, 1);
        e = cudaGetLastError();
    }
    return e == cudaSuccess ? SP_OK : record_error(SP_ECUDA, cudaGetErrorString(e));
}

}  // extern "C"
