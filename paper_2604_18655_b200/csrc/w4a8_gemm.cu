// The paper's own precision regime for a single projection (Sec. 3.3 "LLM Quantization": activations quantised
// per tensor to Int8, weights per channel to Int4): y[m][n] = (sum_k qx[m][k] * qw[n][k]) * (x_scale * w_scale[n]) with
// the contraction in exact integer arithmetic on the tensor cores (mma.sync m16n8k32, s8 x s8 -> s32).
//
// Few rows (M <= 64), so the weights are the 16-row operand: a CTA owns 16 output channels, its eight warps split K in
// spans of 256 inputs, and within a span thread (g, t) of a warp reads the 64 inputs [64 t, 64 t + 64) of channels g
// and g + 8 (two 16-byte loads each: the INT4 bytes as they are stored, channel-major) and of activation row g of
// every 8-row tile.  Which input lands in which k slot of an MMA does not matter for a dot product as long as both
// operands agree, and here the slot depends on t alone: one 32-bit word of nibbles (inputs 8i .. 8i+7) splits into the
// even inputs (low nibbles) and the odd ones (high nibbles), the activation bytes are zipped the same way (prmt).
// Integer partial sums are added across warps in shared memory (any order: exact), then scaled in float32.
#include "common.cuh"

namespace mlora {

constexpr int WA_WARPS = 8;
constexpr int WA_THREADS = WA_WARPS * 32;
constexpr int WA_CH = 16;            // output channels per CTA
constexpr int WA_SPAN = 256;         // inputs per warp step

__device__ __forceinline__ void mma_s8(int (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                       uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint4 ldg_nc16(const void* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
// four stored nibbles (q + 8) in the low halves of four bytes -> four int8 values q
__device__ __forceinline__ uint32_t nib_to_s8(uint32_t v) { return __vsub4(v & 0x0f0f0f0fu, 0x08080808u); }

template <int NT>
__global__ void __launch_bounds__(WA_THREADS) w4a8_kernel(const unsigned char* __restrict__ qw, const __half* __restrict__ w_scale,
                                                         const signed char* qx, float x_scale, int M, int K, int N,
                                                         float* __restrict__ y) {
  __shared__ int red[WA_WARPS][NT][32][4];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int n0 = blockIdx.x * WA_CH;
  int acc[NT][4];
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0;
  const unsigned char* w_lo = qw + (size_t)(n0 + g) * (K / 2);
  const unsigned char* w_hi = qw + (size_t)(n0 + g + 8) * (K / 2);
  const int spans = K / WA_SPAN;
  // the next span's weights are always in flight; the first ones are asked for in L2 ahead of the wait for the kernel before
  // this one (programmatic launch; usually the quantisation of the activations)
  uint32_t nl[8], nh[8];
  auto load = [&](int sp) {
    const int k0 = sp * WA_SPAN + t * 64;
    *reinterpret_cast<uint4*>(nl) = ldg_nc16(w_lo + k0 / 2);
    *reinterpret_cast<uint4*>(nl + 4) = ldg_nc16(w_lo + k0 / 2 + 16);
    *reinterpret_cast<uint4*>(nh) = ldg_nc16(w_hi + k0 / 2);
    *reinterpret_cast<uint4*>(nh + 4) = ldg_nc16(w_hi + k0 / 2 + 16);
  };
  if (warp < spans) {
    const size_t o = (size_t)(warp * WA_SPAN + t * 64) / 2;
    asm volatile("prefetch.global.L2 [%0];\n\tprefetch.global.L2 [%1];" ::"l"(w_lo + o), "l"(w_hi + o) : "memory");
  }
  asm volatile("griddepcontrol.wait;\n\tgriddepcontrol.launch_dependents;" ::: "memory");
  if (warp < spans) load(warp);
  for (int sp = warp; sp < spans; sp += WA_WARPS) {
    const int k0 = sp * WA_SPAN + t * 64;
    uint32_t wl[8], wh[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) { wl[i] = nl[i]; wh[i] = nh[i]; }
    if (sp + WA_WARPS < spans) load(sp + WA_WARPS);
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      const int row = nt * 8 + g;
      uint32_t xs[16];
      if (row < M) {
        const signed char* xr = qx + (size_t)row * K + k0;
#pragma unroll
        for (int q = 0; q < 4; ++q) *reinterpret_cast<uint4*>(xs + 4 * q) = *(reinterpret_cast<const uint4*>(xr) + q);
      } else {
#pragma unroll
        for (int q = 0; q < 16; ++q) xs[q] = 0u;
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        // inputs 8i .. 8i+7 of the thread's 64: even ones in k slots 4t .. 4t+3, odd ones in slots 16+4t .. 16+4t+3
        const uint32_t b0 = __byte_perm(xs[2 * i], xs[2 * i + 1], 0x6420);
        const uint32_t b1 = __byte_perm(xs[2 * i], xs[2 * i + 1], 0x7531);
        mma_s8(acc[nt], nib_to_s8(wl[i]), nib_to_s8(wh[i]), nib_to_s8(wl[i] >> 4), nib_to_s8(wh[i] >> 4), b0, b1);
      }
    }
  }
#pragma unroll
  for (int nt = 0; nt < NT; ++nt)
    *reinterpret_cast<int4*>(red[warp][nt][lane]) = make_int4(acc[nt][0], acc[nt][1], acc[nt][2], acc[nt][3]);
  __syncthreads();
  for (int i = threadIdx.x; i < NT * 32 * 4; i += WA_THREADS) {
    const int e = i & 3, ln = (i >> 2) & 31, nt = i >> 7;
    int sum = 0;
#pragma unroll
    for (int w = 0; w < WA_WARPS; ++w) sum += red[w][nt][ln][e];
    // accumulator element e of lane (g', t'): channel g' (+8 for e >= 2), activation row 8 nt + 2 t' + (e & 1)
    const int n = n0 + (ln >> 2) + ((e & 2) ? 8 : 0);
    const int row = nt * 8 + 2 * (ln & 3) + (e & 1);
    if (row < M) y[(size_t)row * N + n] = (float)sum * (x_scale * __half2float(w_scale[n]));
  }
}

// per-tensor INT8 activations: q = clip(round_half_even(x / scale), -127, 127), the division in float32; eight values a thread
__device__ __forceinline__ unsigned quant_act(__half x, float scale) {
  int q = __float2int_rn(__fdiv_rn(__half2float(x), scale));
  q = q > 127 ? 127 : (q < -127 ? -127 : q);
  return (unsigned)q & 0xffu;
}
__global__ void quant_act_kernel(const __half* x, long long count, float scale, signed char* out) {
  asm volatile("griddepcontrol.wait;\n\tgriddepcontrol.launch_dependents;" ::: "memory");
  const long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * 8;
  if (i + 8 <= count && ((reinterpret_cast<uintptr_t>(x) & 15) | (reinterpret_cast<uintptr_t>(out) & 7)) == 0) {
    const uint4 v = *reinterpret_cast<const uint4*>(x + i);
    const __half* h = reinterpret_cast<const __half*>(&v);
    uint2 o = make_uint2(0u, 0u);
#pragma unroll
    for (int e = 0; e < 4; ++e) { o.x |= quant_act(h[e], scale) << (8 * e); o.y |= quant_act(h[4 + e], scale) << (8 * e); }
    *reinterpret_cast<uint2*>(out + i) = o;
  } else {
    for (long long k = i; k < i + 8 && k < count; ++k) out[k] = (signed char)quant_act(x[k], scale);
  }
}

cudaError_t launch_quant_act(const __half* x, long long count, float scale, signed char* out, cudaStream_t st) {
  // (programmatic although it waits at once: in a chain of programmatic launches no full dependency, which the device
  // resolved in steps of 2 us, stands between one call and the next)
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)((count + 1023) / 1024)); cfg.blockDim = dim3(128); cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, quant_act_kernel, x, count, scale, out);
}

bool w4a8_shape_ok(int M, int K, int N) {
  // 127 * 8 * K must stay below 2^31 for the 32-bit accumulators
  return M >= 1 && M <= 64 && K >= WA_SPAN && K % WA_SPAN == 0 && N >= WA_CH && N % WA_CH == 0 &&
         (long long)K * 127 * 8 < (1ll << 31);
}

cudaError_t launch_w4a8(const unsigned char* w, const __half* ws, const signed char* x, float x_scale, int M, int K, int N,
                        float* y, cudaStream_t st) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(N / WA_CH)); cfg.blockDim = dim3(WA_THREADS); cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (M <= 8) return cudaLaunchKernelEx(&cfg, w4a8_kernel<1>, w, ws, x, x_scale, M, K, N, y);
  if (M <= 16) return cudaLaunchKernelEx(&cfg, w4a8_kernel<2>, w, ws, x, x_scale, M, K, N, y);
  if (M <= 32) return cudaLaunchKernelEx(&cfg, w4a8_kernel<4>, w, ws, x, x_scale, M, K, N, y);
  return cudaLaunchKernelEx(&cfg, w4a8_kernel<8>, w, ws, x, x_scale, M, K, N, y);
}

}  // namespace mlora
