// RMSNorm (Sec. 3.1) fused with the LoRA shrink T[m] = (alpha/r) * h[m] A_a(m)^T  (first half of the
// low-rank term of Eq. 1-4), the adapter gathered per row from the run-time pointer table (Sec. 3.2 (c)).
// One CTA per (row, slice of the rank indices): the row is normalised (or loaded), kept in shared memory,
// and each warp forms rank-r inner products with 128-bit loads of A and a warp-level reduction.
#include "common.cuh"

namespace mlora {

// one entry of T for the tcgen05 projection: value and rounding remainder (LoraArgs::text)
__device__ __forceinline__ void text_store(const LoraArgs& l, int m, int seg, int k, float v) {
  __half* row = l.text + ((size_t)m * l.nseg + seg) * 2 * l.ke + k;
  const __half h = __float2half_rn(v);
  row[0] = h;
  row[l.ke] = __float2half_rn(v - __half2float(h));
}
// zeros everywhere outside the r columns of the row from k0 on (WRAP: round and round)
template <bool WRAP>
__device__ __forceinline__ void text_clear(const LoraArgs& l, int m, int seg, int k0, int r, int tid, int nthreads) {
  __half* row = l.text + ((size_t)m * l.nseg + seg) * 2 * l.ke;
  const int k1 = k0 + r, kw = k1 - l.ke;
  for (int k = tid; k < 2 * l.ke; k += nthreads) {
    const int kk = k < l.ke ? k : k - l.ke;
    if ((kk < k0 || kk >= k1) && (!WRAP || kk >= kw)) row[k] = __float2half_rn(0.f);
  }
}

constexpr int SHRINK_THREADS = 256;
constexpr int SHRINK_JCHUNK = 8;   // rank indices per CTA

__global__ void __launch_bounds__(SHRINK_THREADS) norm_shrink_kernel(const ShrinkArgs p, const int jchunks) {
  // (as a programmatic launch it waits at once and only then lets the projection behind it start, which streams its weights
  // meanwhile and reads the call's inputs ahead of its own wait: everything earlier is complete then)
  asm volatile("griddepcontrol.wait;\n\tgriddepcontrol.launch_dependents;" ::: "memory");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __half* hrow = reinterpret_cast<__half*>(smem_raw);          // [K]
  __shared__ float red[SHRINK_THREADS / 32];
  const int m = blockIdx.x;
  const int K = p.K;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (p.x_f32 != nullptr) {
    const float* x = p.x_f32 + (size_t)m * K;
    float ss = 0.f;
    for (int k = threadIdx.x * 4; k < K; k += SHRINK_THREADS * 4) {
      const float4 v = *reinterpret_cast<const float4*>(x + k);
      ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
    }
    ss = warp_sum(ss);
    if (lane == 0) red[warp] = ss;
    __syncthreads();
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < SHRINK_THREADS / 32; ++w) tot += red[w];
    const float inv = rsqrtf(tot / (float)K + p.eps);
    for (int k = threadIdx.x * 4; k < K; k += SHRINK_THREADS * 4) {
      const float4 v = *reinterpret_cast<const float4*>(x + k);
      const uint2 gv = *reinterpret_cast<const uint2*>(p.gain + k);
      const float2 g01 = __half22float2(u32_as_h2(gv.x)), g23 = __half22float2(u32_as_h2(gv.y));
      const __half2 o01 = __floats2half2_rn(v.x * inv * g01.x, v.y * inv * g01.y);
      const __half2 o23 = __floats2half2_rn(v.z * inv * g23.x, v.w * inv * g23.y);
      const uint2 o = make_uint2(h2_as_u32(o01), h2_as_u32(o23));
      *reinterpret_cast<uint2*>(hrow + k) = o;
      if (blockIdx.y == 0) *reinterpret_cast<uint2*>(p.h_out + (size_t)m * K + k) = o;
    }
  } else {
    const __half* h = p.h_in + (size_t)m * K;
    for (int k = threadIdx.x * 8; k < K; k += SHRINK_THREADS * 8)
      *reinterpret_cast<uint4*>(hrow + k) = *reinterpret_cast<const uint4*>(h + k);
  }
  __syncthreads();

  if (p.lora.adapter_idx == nullptr) return;
  const int r = p.lora.rank;
  const int a = p.lora.adapter_idx[m / p.lora.rows_per_stream];
  const int seg = blockIdx.y / jchunks;
  const int jc = blockIdx.y % jchunks;
  const int j0 = jc * SHRINK_JCHUNK, j1 = min(r, j0 + SHRINK_JCHUNK);
  float* T = p.lora.T + ((size_t)m * p.lora.nseg + seg) * r;
  const __half* A = nullptr;
  if (a >= 0 && a < p.lora.n_slots) A = p.lora.tabA[(size_t)a * p.lora.tab_stride + p.lora.seg[seg].proj_index];
  if (A == nullptr) {
    for (int j = j0 + threadIdx.x; j < j1; j += SHRINK_THREADS) T[j] = 0.f;
    return;
  }
  const float s = p.lora.scale[a];
  for (int j = j0 + warp; j < j1; j += SHRINK_THREADS / 32) {
    const __half* arow = A + (size_t)j * K;
    float acc = 0.f;
    for (int k = lane * 8; k < K; k += 32 * 8) {
      const uint4 av = *reinterpret_cast<const uint4*>(arow + k);
      const uint4 hv = *reinterpret_cast<const uint4*>(hrow + k);
      const uint32_t aw[4] = {av.x, av.y, av.z, av.w};
      const uint32_t hw[4] = {hv.x, hv.y, hv.z, hv.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 af = __half22float2(u32_as_h2(aw[e])), hf = __half22float2(u32_as_h2(hw[e]));
        acc = fmaf(af.x, hf.x, acc);
        acc = fmaf(af.y, hf.y, acc);
      }
    }
    acc = warp_sum(acc);
    if (lane == 0) T[j] = s * acc;
  }
}

// LoRA shrink on mma.sync for passes whose rows are grouped by stream (one adapter per rows_per_stream rows: DS2D trees,
// decode steps of many streams).  One CTA per (up to 16 rows of a stream, segment, 8 rank indices); its sixteen warps split
// K in contiguous ranges and the partial fragments are added in warp order.  Per 16 features a thread loads 8 consecutive
// features of an activation row (rows g and g+8 of the tile) and of an A row (rank index j0 + g): the two k16 steps
// use features {0,1 | 2,3} and {4,5 | 6,7} of that piece for the fragment's (k 2t.. | k 2t+8..) slots -- any pairing of
// slots with features is valid as long as both operands use the same one.  The activations are the fp16 rows the
// GEMM reads, so the A matrix of a stream is fetched once per 16 rows.  Programmatic launch: the A rows (immutable) are
// asked for ahead of the wait; the projection behind this kernel is let go behind it, so that it finds the activations
// complete and only has to wait for T.
constexpr int SHRINK_MMA_WARPS = 16;
__global__ void __launch_bounds__(SHRINK_MMA_WARPS * 32) shrink_mma_kernel(const ShrinkArgs p, const int tiles_per_stream) {
  __shared__ float red[SHRINK_MMA_WARPS][32][4];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int T = p.lora.rows_per_stream, stream = blockIdx.x / tiles_per_stream;
  const int m0 = stream * T + (blockIdx.x - stream * tiles_per_stream) * 16, m_end = min(p.M, (stream + 1) * T);
  const int r = p.lora.rank, K = p.K;
  const int jtiles = (r + 7) / 8;
  const int seg = blockIdx.y / jtiles, j0 = (blockIdx.y % jtiles) * 8;
  const int mA = m0 + g, mB = mA + 8;
  const int a = p.lora.adapter_idx[stream];
  const __half* A = nullptr;
  if (a >= 0 && a < p.lora.n_slots) A = p.lora.tabA[(size_t)a * p.lora.tab_stride + p.lora.seg[seg].proj_index];
  const float s = A != nullptr ? p.lora.scale[a] : 0.f;
  // a warp takes a contiguous range of 64-feature blocks; per block a thread reads 32 contiguous bytes of each of
  // its three rows, so a warp fetches whole 128-byte lines
  const int nblk = K / 64, per = (nblk + SHRINK_MMA_WARPS - 1) / SHRINK_MMA_WARPS;
  const int b0 = warp * per, b1 = min(nblk, b0 + per);
  const uint4* Ar = A != nullptr ? reinterpret_cast<const uint4*>(A + (size_t)min(j0 + g, r - 1) * K) + 2 * t : nullptr;
  if (A != nullptr && t == 0)
    for (int b = b0; b < b1; ++b) asm volatile("prefetch.global.L1 [%0];" ::"l"(Ar + b * 8) : "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  if (A != nullptr) {
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
    const uint4* hA = reinterpret_cast<const uint4*>(p.h_in + (size_t)min(mA, p.M - 1) * K) + 2 * t;
    const uint4* hB = reinterpret_cast<const uint4*>(p.h_in + (size_t)min(mB, p.M - 1) * K) + 2 * t;
    const bool okA = mA < m_end, okB = mB < m_end, okJ = j0 + g < r;
    auto block = [&](const uint4 (&va)[2], const uint4 (&vb)[2], const uint4 (&vw)[2]) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const uint32_t f0[4] = {va[q].x, vb[q].x, va[q].y, vb[q].y}, f1[4] = {va[q].z, vb[q].z, va[q].w, vb[q].w};
        mma_16816(acc, f0, vw[q].x, vw[q].y);
        mma_16816(acc, f1, vw[q].z, vw[q].w);
      }
    };
    int b = b0;
    for (; b + 2 <= b1; b += 2) {                              // two blocks' loads in flight
      uint4 va[2][2], vb[2][2], vw[2][2];
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int o = (b + u) * 8 + q;
          va[u][q] = okA ? __ldcg(hA + o) : zero; vb[u][q] = okB ? __ldcg(hB + o) : zero; vw[u][q] = okJ ? __ldg(Ar + o) : zero;
        }
      block(va[0], vb[0], vw[0]);
      block(va[1], vb[1], vw[1]);
    }
    for (; b < b1; ++b) {
      uint4 va[2], vb[2], vw[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int o = b * 8 + q;
        va[q] = okA ? __ldcg(hA + o) : zero; vb[q] = okB ? __ldcg(hB + o) : zero; vw[q] = okJ ? __ldg(Ar + o) : zero;
      }
      block(va, vb, vw);
    }
  }
  *reinterpret_cast<float4*>(red[warp][lane]) = make_float4(acc[0], acc[1], acc[2], acc[3]);
  __syncthreads();
  if (warp < 4) {
    // accumulator element e = warp of every lane's fragment: [0],[1] = row mA, rank j0 + 2t, +1;  [2],[3] = row mB
    const int e = warp;
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < SHRINK_MMA_WARPS; ++w) tot += red[w][lane][e];
    const int m = (e < 2) ? mA : mB, j = j0 + 2 * t + (e & 1);
    if (m < m_end && j < r) {
      if (p.lora.text != nullptr) text_store(p.lora, m, seg, (stream * r + j) & p.lora.ke_mask, s * tot);
      else p.lora.T[((size_t)m * p.lora.nseg + seg) * r + j] = s * tot;
    }
  } else if (p.lora.text != nullptr && j0 == 0) {
    for (int m = m0 + warp - 4; m < min(m0 + 16, m_end); m += 12) text_clear<true>(p.lora, m, seg, stream * r & p.lora.ke_mask, r, lane, 32);
  }
}

cudaError_t launch_shrink_rows(const ShrinkArgs& a, cudaStream_t st) {
  const int T = a.lora.rows_per_stream, tps = (T + 15) / 16;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)((a.M + T - 1) / T * tps), (unsigned)(a.lora.nseg * ((a.lora.rank + 7) / 8)));
  cfg.blockDim = dim3(SHRINK_MMA_WARPS * 32);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  // Small grids: start beside the projection that is still running, whose SMs have the largest shared-memory share
  // (with another share they would have to drain first).  Larger grids only take room from the projection behind, the sooner the
  // more rows it has.  Milliseconds of two tree passes with no grid, those up to 48 CTAs and those up to 96 let in: llama1b
  // 128 rows 2.65 / 2.54 / 2.54, 240 rows 3.35 / 3.17 / 3.17, 512 rows 4.67 / 4.67 / 4.82; llama3b 128 rows of rank 32 6.47 / 6.36 /
  // 6.02, 192 rows 7.18 / 7.36 / 7.28 (on the wrong side), 256 rows of rank 16 6.69 / 6.81 / 6.82 (as well), of rank 32 7.25 / 7.25 / 7.42.
  attr[1].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
  attr[1].val.sharedMemCarveout = 100;
  cfg.attrs = attr;
  cfg.numAttrs = a.pdl ? ((long long)cfg.gridDim.x * cfg.gridDim.y <= (a.M <= 128 ? 96 : 48) ? 2 : 1) : 0;
  return cudaLaunchKernelEx(&cfg, shrink_mma_kernel, a, tps);
}

// The same for rows that pick their adapters one by one (the single-projection call): a CTA takes an adapter, eight of its
// rank indices and a share of K, finds the rows that use the adapter, and keeps its fragments of A in registers over them,
// 16 rows at a time.  The S CTAs of a cluster split K; the first one adds their sums up in rank order.  (One row per CTA read
// every adapter once per row: 115 MB through L2 and 18 us for 250 rows of 14336 inputs and 8 adapters.)
constexpr int SG_BLOCKS = 2;                 // 64-feature blocks of a warp per CTA: K share = 16 warps x 2 x 64 at most
constexpr int SG_MAX_ROWS = 4096;
// TEXT: T goes into the matrix that the projection reads; else to fp32 T, and rows without an adapter are not looked at.
// (fp32 T: two CTAs an SM asked for, else the compiler takes 70 registers and one fits; 256 rows of 14336 x 4096 with 64 adapters of
// rank 64 96 -> 91 us, of 4096 x 4096 45.6 -> 41.4.  TEXT has 62 by itself; asking for two moved it to 64 and some calls by 1.5 %.)
template <int S, bool TEXT>
__global__ void __launch_bounds__(SHRINK_MMA_WARPS * 32, TEXT ? 0 : 2) shrink_gather_kernel(const ShrinkArgs p) {
  __shared__ float red[SHRINK_MMA_WARPS][32][4];
  __shared__ float part[S][128];             // first CTA of a cluster: the CTAs' sums of a group of 16 rows
  __shared__ short rows[SG_MAX_ROWS];
  __shared__ int s_n, s_w[SHRINK_MMA_WARPS];
  // (a programmatic launch that waits at once and only then lets the projection start, which reads the activations and B
  // ahead of its own wait: everything earlier is complete then)
  asm volatile("griddepcontrol.wait;\n\tgriddepcontrol.launch_dependents;" ::: "memory");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int rank = S > 1 ? (int)blockIdx.x : 0, j0 = blockIdx.y * 8, a = blockIdx.z, r = p.lora.rank, K = p.K;
  const __half* const A = p.lora.tabA[(size_t)a * p.lora.tab_stride + p.lora.seg[0].proj_index];
  const float s = TEXT || A != nullptr ? p.lora.scale[a] : 0.f;
  // this warp's blocks of A, while the rows are looked up
  const int nblk = K / 64, b_lo = (nblk * (rank * SHRINK_MMA_WARPS + warp)) / (S * SHRINK_MMA_WARPS), b_hi = (nblk * (rank * SHRINK_MMA_WARPS + warp + 1)) / (S * SHRINK_MMA_WARPS);
  const uint4* const Ar = reinterpret_cast<const uint4*>(A + (size_t)min(j0 + g, r - 1) * K) + 2 * t;
  uint4 w[SG_BLOCKS][2];
#pragma unroll
  for (int b = 0; b < SG_BLOCKS; ++b)
#pragma unroll
    for (int q = 0; q < 2; ++q) w[b][q] = (A != nullptr && b_lo + b < b_hi && j0 + g < r) ? *(Ar + (b_lo + b) * 8 + q) : make_uint4(0u, 0u, 0u, 0u);
  // rows of the adapter, in rising order (every CTA of a cluster finds the same list); adapter 0's CTAs also see to the rows
  // without one
  if (threadIdx.x == 0) s_n = 0;
  __syncthreads();
  for (int base = 0; base < p.M; base += SHRINK_MMA_WARPS * 32) {
    const int m = base + threadIdx.x;
    const int am = m < p.M ? p.lora.adapter_idx[m] : -1;
    const bool mine = m < p.M && am == a && (!TEXT || A != nullptr);
    const unsigned bal = __ballot_sync(0xffffffffu, mine);
    if (lane == 0) s_w[warp] = __popc(bal);
    __syncthreads();
    int off = s_n;
    for (int q = 0; q < warp; ++q) off += s_w[q];
    if (mine) rows[off + __popc(bal & ((1u << lane) - 1u))] = (short)m;
    __syncthreads();
    if (threadIdx.x == 0) { int n = s_n; for (int q = 0; q < SHRINK_MMA_WARPS; ++q) n += s_w[q]; s_n = n; }
    if (TEXT && rank == 0 && j0 == 0) {
      unsigned none = __ballot_sync(0xffffffffu, m < p.M && ((a == 0 && (am < 0 || am >= p.lora.n_slots)) || (am == a && A == nullptr)));
      for (; none != 0u; none &= none - 1u) text_clear<false>(p.lora, base + warp * 32 + __ffs(none) - 1, 0, 0, 0, lane, 32);
    }
    __syncthreads();
  }
  const int n = s_n;
  for (int r0 = 0; r0 < n; r0 += 16) {
    const int mA = rows[min(r0 + g, n - 1)], mB = rows[min(r0 + g + 8, n - 1)];
    const uint4* const hA = reinterpret_cast<const uint4*>(p.h_in + (size_t)mA * K) + 2 * t;
    const uint4* const hB = reinterpret_cast<const uint4*>(p.h_in + (size_t)mB * K) + 2 * t;
    uint4 va[SG_BLOCKS][2], vb[SG_BLOCKS][2];
#pragma unroll
    for (int b = 0; b < SG_BLOCKS; ++b)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const bool ok = b_lo + b < b_hi;
        va[b][q] = ok ? *(hA + (b_lo + b) * 8 + q) : make_uint4(0u, 0u, 0u, 0u);
        vb[b][q] = ok ? *(hB + (b_lo + b) * 8 + q) : make_uint4(0u, 0u, 0u, 0u);
      }
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int b = 0; b < SG_BLOCKS; ++b)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const uint32_t f0[4] = {va[b][q].x, vb[b][q].x, va[b][q].y, vb[b][q].y}, f1[4] = {va[b][q].z, vb[b][q].z, va[b][q].w, vb[b][q].w};
        mma_16816(acc, f0, w[b][q].x, w[b][q].y);
        mma_16816(acc, f1, w[b][q].z, w[b][q].w);
      }
    for (int b = b_lo + SG_BLOCKS; b < b_hi; ++b)          // (a K share beyond what the registers hold)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const uint4 xa = *(hA + b * 8 + q), xb = *(hB + b * 8 + q), xw = (TEXT || A != nullptr) && j0 + g < r ? *(Ar + b * 8 + q) : make_uint4(0u, 0u, 0u, 0u);
        const uint32_t f0[4] = {xa.x, xb.x, xa.y, xb.y}, f1[4] = {xa.z, xb.z, xa.w, xb.w};
        mma_16816(acc, f0, xw.x, xw.y);
        mma_16816(acc, f1, xw.z, xw.w);
      }
    *reinterpret_cast<float4*>(red[warp][lane]) = make_float4(acc[0], acc[1], acc[2], acc[3]);
    __syncthreads();
    const int e = warp & 3;                                // threads 0-127: accumulator element e of every lane's fragment
    float tot = 0.f;
    if (warp < 4) {
#pragma unroll
      for (int q = 0; q < SHRINK_MMA_WARPS; ++q) tot += red[q][lane][e];
      if constexpr (S > 1) {
        uint32_t dst;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"((uint32_t)__cvta_generic_to_shared(&part[rank][threadIdx.x])), "r"(0));
        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dst), "f"(tot) : "memory");
      }
    }
    if constexpr (S > 1) asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (rank == 0 && warp < 4) {
      if constexpr (S > 1) {
        tot = 0.f;
#pragma unroll
        for (int q = 0; q < S; ++q) tot += part[q][threadIdx.x];
      }
      const int k = r0 + g + (e >= 2 ? 8 : 0), j = j0 + 2 * t + (e & 1);
      if (k < n && j < r) {
        if (TEXT) text_store(p.lora, rows[k], 0, a * r + j, s * tot);
        else p.lora.T[(size_t)rows[k] * r + j] = s * tot;
      }
    }
    if (TEXT && rank == 0 && j0 == 0 && warp >= 4)
      for (int k = r0 + warp - 4; k < min(r0 + 16, n); k += SHRINK_MMA_WARPS - 4) text_clear<false>(p.lora, rows[k], 0, a * r, r, lane, 32);
    if constexpr (S > 1) asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    else __syncthreads();
  }
}

template <int S, bool TEXT>
static cudaError_t launch_gather(const ShrinkArgs& a, cudaStream_t st) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(S, (unsigned)((a.lora.rank + 7) / 8), (unsigned)a.lora.n_slots);
  cfg.blockDim = dim3(SHRINK_MMA_WARPS * 32);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = S; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = S > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, shrink_gather_kernel<S, TEXT>, a);
}
// T of rows with adapters of their own (LoraArgs::text with slots = adapters; or fp32)
template <bool TEXT>
static cudaError_t launch_gather_split(const ShrinkArgs& a, cudaStream_t st) {
  // K split so that a warp's share fits its registers, as long as the grid stays within a few CTAs an SM
  const int per = SHRINK_MMA_WARPS * SG_BLOCKS * 64, ctas = (a.lora.rank + 7) / 8 * a.lora.n_slots;
  if (a.K > 4 * per && ctas <= 64) return launch_gather<8, TEXT>(a, st);
  if (a.K > 2 * per && ctas <= 128) return launch_gather<4, TEXT>(a, st);
  if (a.K > per && ctas <= 256) return launch_gather<2, TEXT>(a, st);
  return launch_gather<1, TEXT>(a, st);
}
cudaError_t launch_shrink_gather(const ShrinkArgs& a, cudaStream_t st) {
  return a.lora.text != nullptr ? launch_gather_split<true>(a, st) : launch_gather_split<false>(a, st);
}

// The expand of rows that pick their adapters one by one from many: y[m] += T[m] B (Eq. 1-4, second factor), after the
// projection.  A CTA takes an adapter (or, more adapters than rows, a row's adapter, if no row before has it) and 256 columns of
// its B, which it reads once, in shared memory, for all rows that use the adapter: fp32 sums, rank indices in rising order.
// Bound by B of the adapters in use; inside the tensor-core projection every row tile paid for every adapter instead, 64 of
// them or 7 that occur (32 rows of 4096 x 4096, 64 adapters of rank 64: 37.6 us, 17.8 with this kernel).
constexpr int EXP_COLS = 256, EXP_ROWS = 16, EXP_RANK = 64, EXP_THREADS = 256;
__global__ void __launch_bounds__(EXP_THREADS) expand_rows_kernel(const LoraArgs l, const int M, const int by_row, float* __restrict__ y, const int N) {
  __shared__ __align__(16) __half s_B[EXP_RANK][EXP_COLS];
  __shared__ __align__(16) float s_T[EXP_ROWS][EXP_RANK];
  __shared__ short rows[4096];
  __shared__ int s_w[EXP_THREADS / 32], s_n;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, r = l.rank, n0 = blockIdx.x * EXP_COLS;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // (the call's inputs, complete before the kernels ahead started)
  const int a = by_row ? l.adapter_idx[blockIdx.y] : (int)blockIdx.y;
  const __half* const B = a >= 0 && a < l.n_slots ? l.tabB[(size_t)a * l.tab_stride + l.seg[0].proj_index] : nullptr;
  // (every CTA takes the wait: a kernel that waits for this one must find the projection done, too)
  if (B == nullptr) { asm volatile("griddepcontrol.wait;" ::: "memory"); return; }
  auto fetch_B = [&](int j0) {                             // rank indices j0 .. of the CTA's columns
    const int nj = min(EXP_RANK, r - j0);
    for (int i = tid; i < nj * (EXP_COLS / 8); i += EXP_THREADS) {
      const int j = i / (EXP_COLS / 8), c = (i % (EXP_COLS / 8)) * 8;
      if (n0 + c < N)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(&s_B[j][c])), "l"(B + (size_t)(j0 + j) * N + n0 + c) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (tid == 0) s_n = 0;
  __syncthreads();
  for (int base = 0; base < M; base += EXP_THREADS) {      // the adapter's rows, in rising order
    const int m = base + tid;
    const bool mine = m < M && l.adapter_idx[m] == a;
    const unsigned bal = __ballot_sync(0xffffffffu, mine);
    if (lane == 0) s_w[warp] = __popc(bal);
    __syncthreads();
    int off = s_n, all = 0;
    for (int q = 0; q < EXP_THREADS / 32; ++q) { if (q < warp) off += s_w[q]; all += s_w[q]; }
    if (mine) rows[off + __popc(bal & ((1u << lane) - 1u))] = (short)m;
    __syncthreads();
    if (tid == 0) s_n += all;
    __syncthreads();
  }
  const int n = s_n;
  const bool on = n > 0 && (!by_row || rows[0] == (int)blockIdx.y);
  if (on) fetch_B(0);
  asm volatile("griddepcontrol.wait;" ::: "memory");      // T and the projection's y
  if (!on) return;
  const int c = (tid & (EXP_COLS / 2 - 1)) * 2, grp = tid / (EXP_COLS / 2);   // two columns, every second row
  for (int j0 = 0; j0 < r; j0 += EXP_RANK) {
    const int nj = min(EXP_RANK, r - j0);
    if (j0 > 0) { __syncthreads(); fetch_B(j0); }
    for (int r0 = 0; r0 < n; r0 += EXP_ROWS) {
      const int nr = min(EXP_ROWS, n - r0);
      if (r0 > 0) __syncthreads();
      for (int i = tid; i < nr * EXP_RANK; i += EXP_THREADS) {
        const int q = i / EXP_RANK, j = i % EXP_RANK;
        s_T[q][j] = j < nj ? __ldcg(l.T + (size_t)rows[r0 + q] * r + j0 + j) : 0.f;
      }
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();
      if (n0 + c < N) {
        for (int q = grp; q < nr; q += 4) {                // two rows at a time
          const bool two = q + 2 < nr;
          float2* const y0 = reinterpret_cast<float2*>(y + (size_t)rows[r0 + q] * N + n0 + c);
          float2* const y1 = two ? reinterpret_cast<float2*>(y + (size_t)rows[r0 + q + 2] * N + n0 + c) : y0;
          const float2 o0 = __ldcg(y0), o1 = __ldcg(y1);
          const float *t0 = s_T[q], *t1 = s_T[two ? q + 2 : q];
          float a0 = 0.f, b0 = 0.f, a1 = 0.f, b1 = 0.f;
#pragma unroll 4
          for (int j = 0; j < nj; ++j) {
            const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&s_B[j][c]));
            const float u = t0[j], v = t1[j];
            a0 = fmaf(u, b.x, a0); b0 = fmaf(u, b.y, b0);
            a1 = fmaf(v, b.x, a1); b1 = fmaf(v, b.y, b1);
          }
          *y0 = make_float2(o0.x + a0, o0.y + b0);
          if (two) *y1 = make_float2(o1.x + a1, o1.y + b1);
        }
      }
    }
  }
}
cudaError_t launch_expand_rows(const LoraArgs& l, int M, float* y, int N, cudaStream_t st) {
  const int by_row = l.n_slots > M;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)((N + EXP_COLS - 1) / EXP_COLS), (unsigned)(by_row ? M : l.n_slots));
  cfg.blockDim = dim3(EXP_THREADS);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, expand_rows_kernel, l, M, by_row, y, N);
}

cudaError_t init_shrink() {
  cudaError_t e;
#define SG_SET(S) \
  if ((e = full_carveout(shrink_gather_kernel<S, true>)) != cudaSuccess) return e; \
  if ((e = full_carveout(shrink_gather_kernel<S, false>)) != cudaSuccess) return e;
  SG_SET(1) SG_SET(2) SG_SET(4) SG_SET(8)
#undef SG_SET
  if ((e = full_carveout(expand_rows_kernel)) != cudaSuccess) return e;
  return cudaFuncSetAttribute(norm_shrink_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SHRINK_MAX_K * (int)sizeof(__half));
}

cudaError_t launch_shrink(const ShrinkArgs& a, cudaStream_t st) {
  // Runs of 16 rows share an adapter: the norm (if any) as its own pass, the shrink on mma.sync from the fp16 rows.
  // With a norm this costs a second launch, which pays only when the shrink is large.
  const bool big = (long long)a.lora.rank * a.lora.nseg * a.K >= 150000;
  if (a.lora.adapter_idx != nullptr && a.lora.rows_per_stream % 16 == 0 && a.M >= 32 && (a.x_f32 == nullptr || big)) {
    ShrinkArgs r = a;
    if (a.x_f32 != nullptr) {
      ShrinkArgs n = a;
      n.lora.adapter_idx = nullptr;
      dim3 grid(a.M, 1);
      norm_shrink_kernel<<<grid, SHRINK_THREADS, (size_t)a.K * sizeof(__half), st>>>(n, 1);
      const cudaError_t e = cudaGetLastError();
      if (e != cudaSuccess) return e;
      r.h_in = a.h_out;
    }
    return launch_shrink_rows(r, st);
  }
  int jchunks = 1, gy = 1;
  if (a.lora.adapter_idx != nullptr) {
    jchunks = (a.lora.rank + SHRINK_JCHUNK - 1) / SHRINK_JCHUNK;
    gy = jchunks * a.lora.nseg;
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)a.M, (unsigned)gy);
  cfg.blockDim = dim3(SHRINK_THREADS); cfg.dynamicSmemBytes = (size_t)a.K * sizeof(__half); cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = a.pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, norm_shrink_kernel, a, jchunks);
}

}  // namespace mlora
