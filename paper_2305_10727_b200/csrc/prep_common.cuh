// Device and host helpers shared by the operand-preparation kernels (elementwise.cu, int4.cu).
#pragma once

#include <cuda_fp16.h>

#include <atomic>

#include "common.cuh"
#include "quant_math.cuh"

namespace gpusq {

constexpr int kThreads = 256;

// ---- keep-two rule (Sec. 1 / Sec. 3.1; criterion: two largest magnitudes, lower index wins ties) ----
// Element i beats j when mag_i > mag_j, or when they are equal and i < j.  The
// two elements that win at least two of their three comparisons are kept.
// Returns the 4-bit keep mask (bit i = element i kept); exactly two bits set.
template <typename T>
__device__ __forceinline__ uint32_t keep_two_mask(T m0, T m1, T m2, T m3)
{
    const int b01 = m0 >= m1, b02 = m0 >= m2, b03 = m0 >= m3;
    const int b12 = m1 >= m2, b13 = m1 >= m3, b23 = m2 >= m3;
    const int w0 = b01 + b02 + b03;
    const int w1 = (1 - b01) + b12 + b13;
    const int w2 = (1 - b02) + (1 - b12) + b23;
    const int w3 = (1 - b03) + (1 - b13) + (1 - b23);
    return (uint32_t)(w0 >= 2) | ((uint32_t)(w1 >= 2) << 1) | ((uint32_t)(w2 >= 2) << 2) |
           ((uint32_t)(w3 >= 2) << 3);
}

// ------------------------------------------------------------ quantisation
// code = clamp(round-half-even(x / scale), -127, 127), IEEE division.
__device__ __forceinline__ int quant_code(float x, float scale, int qmax = 127)
{
    int q = __float2int_rn(__fdiv_rn(x, scale));
    return max(-qmax, min(qmax, q));
}

__device__ __forceinline__ float scale_from_amax(float amax, float qmax = 127.0f)
{
    return amax == 0.0f ? 1.0f : __fdiv_rn(amax, qmax);
}

__device__ __forceinline__ float block_max(float v, float *red)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();  // red may still be read from a previous use
    if (lane == 0) red[warp] = v;
    __syncthreads();
    float r = red[0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) r = fmaxf(r, red[w]);
    return r;
}

// First statement of a kernel launched with launch_behind(): what was launched before is complete from
// here on, and what is launched next may be set up.
__device__ __forceinline__ void begin_behind()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

int quant_weight_common(const float *Wp, int8_t *Wq, float *w_scale, int N, int K, void *stream, float qmax);

constexpr int kMaxDevices = 64;
constexpr int kMaxPartials = 2048;   // workspace: one 32-bit partial maximum per block ...
constexpr int kWorkspaceExtra = 64;  // ... and, behind them, the control words of the one-launch kernel

__device__ __forceinline__ uint32_t absmax_bits8(uint4 v)
{
    // |binary16| as unsigned 15-bit patterns order like the magnitudes (no NaN expected)
    uint32_t a = __vmaxu2(v.x & 0x7FFF7FFFu, v.y & 0x7FFF7FFFu);
    uint32_t b = __vmaxu2(v.z & 0x7FFF7FFFu, v.w & 0x7FFF7FFFu);
    a = __vmaxu2(a, b);
    return max(a & 0xFFFFu, a >> 16);
}

// Partial maxima, one per block of at most two per SM: eight 16-byte loads in flight per thread.
constexpr int kAbsmaxThreads = 512;
static __global__ void __launch_bounds__(kAbsmaxThreads)
act_absmax_kernel(const uint4 *__restrict__ X, uint32_t *__restrict__ partial, int64_t vec8)
{
    __shared__ uint32_t red[kAbsmaxThreads / 32];
    begin_behind();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    uint32_t m = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < vec8; i += 8 * stride) {
        uint4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = i + u * stride < vec8 ? __ldg(X + i + u * stride) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int u = 0; u < 8; ++u) m = max(m, absmax_bits8(v[u]));
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) {
        m = __reduce_max_sync(0xffffffffu, threadIdx.x < kAbsmaxThreads / 32 ? red[threadIdx.x] : 0u);
        if (threadIdx.x == 0) partial[blockIdx.x] = m;
    }
}

inline int absmax_blocks(int64_t vec8)
{
    const int64_t want = ceil_div(vec8, kAbsmaxThreads), most = 2 * (int64_t)num_sms();
    return (int)(want < most ? want : most < kMaxPartials ? most : kMaxPartials);
}

// eight binary16 values (16 bytes) -> eight INT8 codes (8 bytes); one exactness test for all eight
__device__ __forceinline__ float2 h2f(uint32_t h2) { return __half22float2(*reinterpret_cast<const __half2 *>(&h2)); }

template <bool kClamp>
__device__ __forceinline__ uint2 quant8_f16(uint4 v, const QuantScale &a)
{
    uint32_t differ = 0;
    const float2 f0 = h2f(v.x), f1 = h2f(v.y), f2 = h2f(v.z), f3 = h2f(v.w);
    float2 m0 = quant2_sums<kClamp>(f0, a, differ), m1 = quant2_sums<kClamp>(f1, a, differ);
    float2 m2 = quant2_sums<kClamp>(f2, a, differ), m3 = quant2_sums<kClamp>(f3, a, differ);
    if (differ != 0u || a.always_divide) {
        m0 = quant2_exact<kClamp>(f0, a);
        m1 = quant2_exact<kClamp>(f1, a);
        m2 = quant2_exact<kClamp>(f2, a);
        m3 = quant2_exact<kClamp>(f3, a);
    }
    return make_uint2(pack4_low_bytes(m0, m1), pack4_low_bytes(m2, m3));
}

// One product per value: the codes of eight binary16 values when find_single_product() found a factor.
template <bool kClamp>
__device__ __forceinline__ uint2 quant8_single(uint4 v, const QuantScale &a)
{
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    const __half2 bound = __float2half2_rn(a.x_max);
    float2 m[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        __half2 h = *reinterpret_cast<const __half2 *>(&w[i]);
        if (kClamp) h = __hmin2(__hmax2(h, __hneg2(bound)), bound);
        m[i] = __ffma2_rn(__half22float2(h), a.c, make_float2(kRoundMagic, kRoundMagic));
    }
    return make_uint2(pack4_low_bytes(m[0], m[1]), pack4_low_bytes(m[2], m[3]));
}

// Looks for a factor c, next to 1/s, with which rounding x * c gives the code of EVERY binary16 x, and
// leaves it in a.c.  The product's code and the true quotient's are both steps that never fall as x
// grows, so they are the same function if they agree at the binary16 numbers around every threshold
// (k + 1/2) s: the nearest one and its two neighbours (the threshold itself is known to 2^-23 of its
// value, far less than a binary16 step; between the upper neighbour of one threshold and the lower one
// of the next both are constant).  Negative x mirror.  kClamp: values beyond +-qmax s are first clamped
// to the binary16 number next to it, which must have the largest code itself.
// Tried are 1/s rounded and the next number above it: a scale computed as max / 127 has a value (half the
// maximum) exactly on a threshold that rounds up.  One of them holds for 98 of 100 computed and all but
// 2 in 600 supplied scales; the others take the bracketing products.
// To be called by all threads of the block (it is a barrier).
template <bool kClamp>
__device__ __forceinline__ bool find_single_product(QuantScale &a)
{
    const float c0 = a.c.x, c1 = __uint_as_float(__float_as_uint(a.c.x) + 1u);
    bool ok0 = !a.always_divide, ok1 = ok0;
    auto look = [&](int bits) {
        const float x = __half2float(__ushort_as_half((unsigned short)bits));
        const float exact = quant_exact_sum<false>(x, a.s, a.qmax);
        ok0 = ok0 && __fmaf_rn(x, c0, kRoundMagic) == exact;
        ok1 = ok1 && __fmaf_rn(x, c1, kRoundMagic) == exact;
        return exact;
    };
    // one neighbour of one threshold, one division, per thread and step
    for (int t = threadIdx.x; t < 3 * (int)a.qmax; t += blockDim.x) {
        const int k = t / 3, h = __half_as_ushort(__float2half_rn(__fmul_rn((float)k + 0.5f, a.s))) + t - 3 * k - 1;
        if (h >= 0 && h < 0x7C00) look(h);
    }
    if (kClamp) {
        const int b = __half_as_ushort(__float2half_rn(a.x_max));
        if (b >= 0x7C00 || look(b) != kRoundMagic + a.qmax) ok0 = ok1 = false;
    }
    if (__syncthreads_and(ok0)) return true;
    if (!__syncthreads_and(ok1)) return false;
    a.c = make_float2(c1, c1);
    return true;
}

inline int grid_for(int64_t items, int per_sm)
{
    int64_t blocks = ceil_div(items, kThreads);
    int64_t cap = (int64_t)num_sms() * per_sm;
    return (int)(blocks < cap ? (blocks < 1 ? 1 : blocks) : cap);
}

// Asks for a split of an SM's 228 KB between shared memory (percent) and L1, once per device.  Without it a kernel that is
// set up while a GEMM drains gets the GEMM's split, 28 KB of L1, through which all its loads have to pass.
template <auto kKernel>
inline void prefer_carveout(int percent)
{
    static std::atomic<uint64_t> asked{0};
    static_assert(kMaxDevices == 64, "a bit per device");
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices || asked.load(std::memory_order_relaxed) >> dev & 1) return;
    if (cudaFuncSetAttribute(kKernel, cudaFuncAttributePreferredSharedMemoryCarveout, percent) != cudaSuccess) (void)cudaGetLastError();
    asked.fetch_or((uint64_t)1 << dev, std::memory_order_relaxed);
}

// Launch that may be set up while the previous kernel of the stream drains; the kernel itself waits
// (griddepcontrol.wait) before it touches memory.
template <typename... P, typename... A>
inline int launch_behind(void (*kernel)(P...), dim3 grid, dim3 threads, cudaStream_t stream, A... args)
{
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = threads;
    cfg.stream = stream;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kernel, args...) != cudaSuccess) {
        (void)cudaGetLastError();
        return GPUSQ_ERR_CUDA;
    }
    return GPUSQ_OK;
}

}  // namespace gpusq
