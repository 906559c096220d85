// Attention of passes with several rows per stream (DS2D trees, prefill) and of decode steps of many streams on the
// 5th-generation tensor cores: shared prompt segment, own segments, tree-ancestor or causal mask (Sec. 3.4, 3.5, App. A).
//
// A CTA takes a kv head, NQ blocks of up to 128 query rows (row = pass row x query head of the group) and a range of keys,
// 128 at a time.  Warp roles: four softmax warps per block (a thread owns a row: tensor-memory lane = row, so the running
// maximum and sum need no shuffles), one warp for the TMA copies, one for the MMAs.
//   S = Q K^T   both operands in shared memory (128-byte swizzle), 128 x 128 fp32 accumulator in tensor memory
//   P           written back over S as fp16: the A operand of the second product, read from tensor memory
//   O += P V    V as it lies in the cache (key-major: an MN-major B operand), accumulator in tensor memory
// The running maximum is only raised (and O rescaled) when a tile exceeds it by more than 2^8: P stays below 256, well
// inside fp16, and the sum is kept in fp32.  With NQ = 2 the tensor core works on one block while the other's softmax runs.
// What bounds it: 16384 exponentials per tile against 16 per clock and SM (1024 cycles; the two products of head size 128
// take as long).
// Trees: the prefix is cut into chunks that serve the rows of ALL streams, an own segment into chunks that serve its stream;
// partial results go to the scratch that attn_merge_kernel combines.  Causal passes need no partials: one CTA sees all keys of its
// rows, longest rows first.  q, and the K/V rows of the pass, are rotated and in the cache already (the q,k,v projection's
// epilogue puts them there).
#include <cuda.h>
#include <cudaTypedefs.h>

#include "tc.cuh"

namespace mlora {

constexpr int AT_KEYS = 128;                 // keys per tile
constexpr int AT_ROWS = 128;                 // query rows per block (tensor-memory lanes)
template <int HD, int NQ> struct AtCfg {
  static constexpr int NS = (HD == 128 && NQ == 1) ? 1 : 2;              // K and V tiles in flight
  static constexpr uint32_t TILE = AT_KEYS * HD * 2;                     // bytes of a K, V or Q tile
  static constexpr size_t SMEM = (size_t)TILE * (NQ + 2 * NS) + 1024;
  static constexpr int THREADS = NQ * 128 + 64;
  static constexpr int COLS = NQ == 1 ? 256 : 512;
  static constexpr int OCC = NQ == 1 ? 2 : 1;
};

struct AtItem { int own, s, v_lo, v_hi, k0, k1, slot; };

__device__ __forceinline__ void at_copy3(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar) : "memory");
}
__device__ __forceinline__ void at_copy4(uint32_t dst, const CUtensorMap* map, int x, int y, int z, int w, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar) : "memory");
}
// 32 lanes x 32 columns, not waited for
__device__ __forceinline__ void at_ld32(uint32_t addr, float* f) {
  uint32_t* v = reinterpret_cast<uint32_t*>(f);
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
        "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
        "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(addr) : "memory");
}
__device__ __forceinline__ void at_st32(uint32_t addr, const uint32_t* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%32], "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31};"
      ::"r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
        "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]),
        "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]),
        "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31]), "r"(addr) : "memory");
}
__device__ __forceinline__ float at_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// the low bits of a 32-bit word that stand for keys below `lim`
__device__ __forceinline__ uint32_t at_low_bits(int lim) { return lim >= 32 ? 0xffffffffu : (lim <= 0 ? 0u : (1u << lim) - 1u); }

template <int HD, int NQ>
__global__ void __launch_bounds__(AtCfg<HD, NQ>::THREADS, AtCfg<HD, NQ>::OCC)
attn_tc_kernel(const __grid_constant__ AttnArgs p, const int rb_rows, const int rb_all, const int rb_own, const float scale_log2,
               const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_pk,
               const __grid_constant__ CUtensorMap map_pv, const __grid_constant__ CUtensorMap map_ok,
               const __grid_constant__ CUtensorMap map_ov) {
  using C = AtCfg<HD, NQ>;
  constexpr int NS = C::NS, HALVES = HD / 64;
  constexpr uint32_t TILE = C::TILE, HALF = AT_KEYS * 128;               // a tile = HD / 64 column halves of 128 rows x 128 bytes
  extern __shared__ __align__(1024) unsigned char at_smem[];
  __shared__ __align__(8) uint64_t q_full, k_full[NS], k_empty[NS], v_full[NS], v_empty[NS], s_full[NQ], p_full[NQ], o_done[NQ];
  __shared__ uint32_t tmem_s;
  const uint32_t base = (tc_smem_u32(at_smem) + 1023u) & ~1023u;
  const uint32_t q_sm = base, k_sm = base + NQ * TILE, v_sm = k_sm + NS * TILE;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int kh = blockIdx.y, g = p.Hq / p.Hkv;
  const int R_all = p.n * p.T * g;

  // ---- which rows, which keys
  AtItem it{};
  int S_own = 0;
  if (p.causal) {
    const int b = gridDim.x - 1 - blockIdx.x;              // the longest first
    it.v_lo = b * NQ * rb_rows; it.v_hi = R_all;
    it.k1 = p.P + min(p.T, (it.v_lo + NQ * rb_rows - 1) / g + 1);
  } else {
    int item = blockIdx.x;
    if (item < p.n_prefix_chunks * rb_all) {
      it.slot = item / rb_all;
      it.v_lo = (item % rb_all) * NQ * rb_rows; it.v_hi = R_all;
      it.k0 = it.slot * p.prefix_chunk; it.k1 = min(p.P, it.k0 + p.prefix_chunk);
    } else {
      item -= p.n_prefix_chunks * rb_all;
      const int rb = item % rb_own, chunk = item / rb_own % p.n_own_chunks;
      it.own = 1; it.slot = p.n_prefix_chunks + chunk; it.s = item / (rb_own * p.n_own_chunks);
      it.v_lo = it.s * p.T * g + rb * NQ * rb_rows; it.v_hi = (it.s + 1) * p.T * g;
      S_own = p.suffix_len[it.s];
      it.k0 = chunk * p.own_chunk; it.k1 = S_own + p.T;
      // (the last chunk takes what is left, whatever bound the chunks were planned with)
      if (chunk + 1 < p.n_own_chunks) it.k1 = min(it.k1, it.k0 + p.own_chunk);
      if (it.k1 <= it.k0) return;                          // nothing here yet (the merge skips this slot too)
    }
  }
  int n_w[NQ];                                             // key tiles of each block
#pragma unroll
  for (int w = 0; w < NQ; ++w) {
    const int lo = it.v_lo + w * rb_rows;
    int ke = it.k1;
    if (p.causal) ke = min(ke, p.P + min(p.T, (lo + rb_rows - 1) / g + 1));
    n_w[w] = lo < it.v_hi ? (ke - it.k0 + AT_KEYS - 1) / AT_KEYS : 0;
  }
  int n_max = n_w[0];
  if (NQ == 2) n_max = max(n_max, n_w[NQ - 1]);

  if (tid == 0) {
    TC_MBAR_INIT(&q_full, 1);
    for (int i = 0; i < NS; ++i) { TC_MBAR_INIT(k_full + i, 1); TC_MBAR_INIT(k_empty + i, 1); TC_MBAR_INIT(v_full + i, 1); TC_MBAR_INIT(v_empty + i, 1); }
    for (int w = 0; w < NQ; ++w) { TC_MBAR_INIT(s_full + w, 1); TC_MBAR_INIT(p_full + w, 4); TC_MBAR_INIT(o_done + w, 1); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == NQ * 4 + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem_u32(&tmem_s)), "r"((uint32_t)C::COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_s, 0);
  bool alive = true;

  if (warp == NQ * 4) {
    // ---- copies
    const uint32_t elected = tc_elect();
    const bool early = !p.causal && !it.own;               // prefix keys are not written by the pass
    auto load = [&](uint32_t dst, const CUtensorMap* mp, const CUtensorMap* mo, int key, uint32_t bar) {
      if (elected) {
        tc_expect_tx(bar, TILE);
#pragma unroll
        for (int h = 0; h < HALVES; ++h) {
          if (it.own) at_copy4(dst + h * HALF, mo, h * 64, key, kh, it.s, bar);
          else at_copy3(dst + h * HALF, mp, h * 64, key, kh, bar);
        }
      }
      __syncwarp();
    };
    auto load_q = [&]() {
      asm volatile("griddepcontrol.wait;" ::: "memory");
      if (elected) {
        int blocks = 0;
#pragma unroll
        for (int w = 0; w < NQ; ++w) blocks += n_w[w] > 0;
        tc_expect_tx(tc_smem_u32(&q_full), blocks * HALVES * (uint32_t)rb_rows * 128u);
#pragma unroll
        for (int w = 0; w < NQ; ++w)
          if (n_w[w] > 0)
#pragma unroll
            for (int h = 0; h < HALVES; ++h)
              at_copy3(q_sm + w * TILE + h * HALF, &map_q, h * 64, kh * g, (it.v_lo + w * rb_rows) / g, tc_smem_u32(&q_full));
      }
      __syncwarp();
    };
    if (!early) load_q();
    int issued = 0;
    for (int j = 0; j < n_max && alive; ++j) {
      const int st = j % NS; const uint32_t ph = (uint32_t)((j / NS) & 1) ^ 1u;
      const int key = it.k0 + j * AT_KEYS;
      alive = tc_wait(tc_smem_u32(k_empty + st), ph, p.status);
      if (!alive) break;
      load(k_sm + st * TILE, &map_pk, &map_ok, key, tc_smem_u32(k_full + st));
      if (early && j == 0) load_q();
      alive = tc_wait(tc_smem_u32(v_empty + st), ph, p.status);
      if (alive) load(v_sm + st * TILE, &map_pv, &map_ov, key, tc_smem_u32(v_full + st));
      issued = j + 1;
    }
    // no copy may be in flight when the CTA ends (passes at once unless a wait gave up somewhere)
    tc_wait(tc_smem_u32(&q_full), 0u, p.status);
    for (int j = issued > NS ? issued - NS : 0; j < issued; ++j) {
      tc_wait(tc_smem_u32(k_full + j % NS), (uint32_t)((j / NS) & 1), p.status);
      if (alive) tc_wait(tc_smem_u32(v_full + j % NS), (uint32_t)((j / NS) & 1), p.status);
    }
  } else if (warp == NQ * 4 + 1) {
    // ---- MMAs: S(w, j + 1) goes out right behind O(w, j), so that the tensor core has the other block's work meanwhile
    const uint32_t elected = tc_elect();
    // K-major operands: 1024 bytes between 8-row groups.  V: MN-major, 128-byte rows of 64 features, 8-key groups 1024
    // bytes apart, column halves HALF apart.
    constexpr uint64_t DESC = ((uint64_t)1 << 46) | ((uint64_t)2 << 61) | ((uint64_t)(1024 >> 4) << 32);
    constexpr uint64_t DESC_K = DESC | ((uint64_t)1 << 16), DESC_V = DESC | ((uint64_t)(HALF >> 4) << 16);
    auto desc = [](uint64_t proto, uint32_t a) { return proto | (uint64_t)((a & 0x3FFFF) >> 4); };
    auto keys16 = [&](int j) { return (min(AT_KEYS, it.k1 - it.k0 - j * AT_KEYS) + 15) >> 4; };
    auto qk = [&](int w, int j) {
      if (elected) {
        const uint32_t idesc = (1u << 4) | ((uint32_t)(keys16(j) * 2) << 17) | ((AT_ROWS >> 4) << 24);
        const uint32_t qa = q_sm + w * TILE, ka = k_sm + (j % NS) * TILE;
#pragma unroll
        for (int kk = 0; kk < HD / 16; ++kk) {
          const uint32_t off = (kk >> 2) * HALF + (kk & 3) * 32;
          asm volatile(
              "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
              "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
              ::"r"(tmem + w * 128), "l"(desc(DESC_K, qa + off)), "l"(desc(DESC_K, ka + off)), "r"(idesc), "r"(kk > 0 ? 1u : 0u) : "memory");
        }
        tc_commit(tc_smem_u32(s_full + w));
      }
      __syncwarp();
    };
    auto pv = [&](int w, int j) {
      if (elected) {
        constexpr uint32_t idesc = (1u << 4) | (1u << 16) | ((uint32_t)(HD >> 3) << 17) | ((AT_ROWS >> 4) << 24);
        const uint32_t va = v_sm + (j % NS) * TILE;
        const int n16 = keys16(j);
        for (int kk = 0; kk < n16; ++kk)
          asm volatile(
              "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
              "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
              ::"r"(tmem + NQ * 128 + w * HD), "r"(tmem + w * 128 + kk * 8), "l"(desc(DESC_V, va + kk * 2048)), "r"(idesc), "r"((j > 0 || kk > 0) ? 1u : 0u) : "memory");
        tc_commit(tc_smem_u32(o_done + w));
      }
      __syncwarp();
    };
    auto wait = [&](uint64_t* bar, int phase) {
      if (alive) alive = tc_wait(tc_smem_u32(bar), (uint32_t)(phase & 1), p.status);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      return alive;
    };
    if (wait(&q_full, 0) && wait(k_full, 0)) {
#pragma unroll
      for (int w = 0; w < NQ; ++w) if (n_w[w] > 0) qk(w, 0);
      if (elected) tc_commit(tc_smem_u32(k_empty));
      __syncwarp();
    }
    for (int j = 0; j < n_max && alive; ++j) {
#pragma unroll
      for (int w = 0; w < NQ; ++w) {
        if (j >= n_w[w]) continue;
        if (!wait(p_full + w, j) || !wait(v_full + j % NS, j / NS)) break;
        pv(w, j);
        if (j + 1 < n_w[w]) {
          if (!wait(k_full + (j + 1) % NS, (j + 1) / NS)) break;
          qk(w, j + 1);
        }
      }
      if (elected) {
        tc_commit(tc_smem_u32(v_empty + j % NS));
        if (j + 1 < n_max) tc_commit(tc_smem_u32(k_empty + (j + 1) % NS));
      }
      __syncwarp();
    }
  } else {
    // ---- softmax: thread = row
    const int w = warp >> 2;
    const int row = (warp & 3) * 32 + lane, v = it.v_lo + w * rb_rows + row;
    const bool row_ok = row < rb_rows && v < it.v_hi;
    const int m = row_ok ? v / g : 0;
    const int n_tiles = n_w[w];
    const uint32_t s_t = tmem + w * 128 + ((uint32_t)((warp & 3) * 32) << 16), o_t = s_t - w * 128 + NQ * 128 + w * HD;
    const int lim = !row_ok ? 0 : (p.causal ? p.P + m + 1 : it.k1);      // keys below it are visible (own segments: see the mask)
    unsigned long long anc = 0ull;
    if (it.own && row_ok) anc = p.anc[m];
    float m_used = -INFINITY, l = 0.f;
    for (int j = 0; j < n_tiles; ++j) {
      const int k0 = it.k0 + j * AT_KEYS;
      if (alive) alive = tc_wait(tc_smem_u32(s_full + w), (uint32_t)(j & 1), p.status);
      alive = __all_sync(0xffffffffu, alive);
      if (!alive) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      float s[AT_KEYS];
#pragma unroll
      for (int c = 0; c < 4; ++c) at_ld32(s_t + c * 32, s + c * 32);
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      if (!__all_sync(0xffffffffu, !it.own && lim - k0 >= AT_KEYS)) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int kb = k0 + c * 32;
          uint32_t vis;
          if (it.own) {
            const int d = kb - S_own;                      // the tree's bit 0 sits at key S_own
            vis = at_low_bits(-d) | (d >= 0 ? (d < 64 ? (uint32_t)(anc >> d) : 0u) : (d > -32 ? (uint32_t)(anc << -d) : 0u));
            if (!row_ok) vis = 0u;
          } else {
            vis = at_low_bits(lim - kb);
          }
#pragma unroll
          for (int i = 0; i < 32; ++i)
            if (!((vis >> i) & 1u)) s[c * 32 + i] = -INFINITY;
        }
      }
      float mx[4] = {s[0], s[1], s[2], s[3]};
#pragma unroll
      for (int i = 4; i < AT_KEYS; ++i) mx[i & 3] = fmaxf(mx[i & 3], s[i]);
      const float mt = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * scale_log2;
      if (__any_sync(0xffffffffu, mt > m_used + 8.f)) {    // (also the first tile: m_used = -inf)
        const float mn = fmaxf(m_used, mt);
        const float f = m_used == -INFINITY ? 0.f : at_ex2(m_used - mn);
        m_used = mn;
        l *= f;
        if (j > 0) {
          if (alive) alive = tc_wait(tc_smem_u32(o_done + w), (uint32_t)((j - 1) & 1), p.status);
          alive = __all_sync(0xffffffffu, alive);
          if (!alive) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
          for (int c = 0; c < HD; c += 16) {
            float o[16];
            tc_ld_32x32b_x16(o_t + c, o);
            uint32_t u[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) u[i] = __float_as_uint(o[i] * f);
            tc_st_32x32b_x16(o_t + c, u);
          }
        }
      }
      const float mb = m_used == -INFINITY ? 0.f : m_used;
      float ls[4] = {0.f, 0.f, 0.f, 0.f};
      uint32_t pf[32];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          const float a = at_ex2(fmaf(s[h * 64 + 2 * i], scale_log2, -mb)), b = at_ex2(fmaf(s[h * 64 + 2 * i + 1], scale_log2, -mb));
          ls[(2 * i) & 3] += a; ls[(2 * i + 1) & 3] += b;
          pf[i] = h2_as_u32(__floats2half2_rn(a, b));
        }
        at_st32(s_t + h * 32, pf);
      }
      l += (ls[0] + ls[1]) + (ls[2] + ls[3]);
      const int valid = it.k1 - k0;
      if (it.own && valid < AT_KEYS) {
        // the tail of an own segment's V tile is memory nobody wrote yet: its weights are zero, its values must be finite
        if (alive) alive = tc_wait(tc_smem_u32(v_full + j % NS), (uint32_t)((j / NS) & 1), p.status);
        const int last = (valid + 15) & ~15;
        for (int i = tid & 127; i < (last - valid) * (HD / 8); i += 128) {
          const int r = valid + i / (HD / 8), pc = i % (HD / 8);
          asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(v_sm + (j % NS) * TILE + (pc >> 3) * HALF + r * 128 + (pc & 7) * 16), "r"(0u) : "memory");
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) tc_arrive(tc_smem_u32(p_full + w));
    }
    if (n_tiles > 0 && alive) alive = tc_wait(tc_smem_u32(o_done + w), (uint32_t)((n_tiles - 1) & 1), p.status);
    alive = __all_sync(0xffffffffu, alive);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // the tiles' memory is about to be reused: with two blocks both have to be done with it (not by waiting for the other's
    // o_done: a parity only tells apart phases next to each other, and these warps have not followed that barrier)
    if constexpr (NQ == 2) asm volatile("bar.sync 1, %0;" ::"n"(NQ * 128) : "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (n_tiles > 0 && alive) {
      // a thread holds a row: through shared memory (the tiles have all been read), so that a warp stores whole rows (rows
      // straight from the threads took 2.5 us of a CTA's 9 for 64 features, 5 for 128)
      constexpr int LD = HD + 4;
      float* const buf = reinterpret_cast<float*>(at_smem + (base - tc_smem_u32(at_smem))) + (size_t)(tid >> 5) * 32 * LD;
      const float inv = p.causal ? (l > 0.f ? 1.f / l : 0.f) : 1.f;
#pragma unroll 1
      for (int c = 0; c < HD; c += 16) {
        float o[16];
        tc_ld_32x32b_x16(o_t + c, o);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          *reinterpret_cast<float4*>(buf + lane * LD + c + 4 * i) = make_float4(o[4 * i] * inv, o[4 * i + 1] * inv, o[4 * i + 2] * inv, o[4 * i + 3] * inv);
      }
      __syncwarp();
      const int slots = p.n_prefix_chunks + p.n_own_chunks;
      const size_t idx = ((size_t)kh * R_all + (row_ok ? v : 0)) * slots + it.slot;
      const int v0 = v - lane, rows = min(32, min(rb_rows - (row - lane), it.v_hi - v0));
      constexpr int RPI = 128 / HD;                        // rows a warp stores at a time
      const int r_l = lane / (HD / 4), d = (lane % (HD / 4)) * 4;
#pragma unroll 4
      for (int r = r_l; r < rows; r += RPI) {
        const float4 o = *reinterpret_cast<const float4*>(buf + r * LD + d);
        if (p.causal) {
          const int mm = (v0 + r) / g;
          *reinterpret_cast<uint2*>(p.out + ((size_t)mm * p.Hq + kh * g + (v0 + r - mm * g)) * HD + d) =
              make_uint2(h2_as_u32(__floats2half2_rn(o.x, o.y)), h2_as_u32(__floats2half2_rn(o.z, o.w)));
        } else {
          *reinterpret_cast<float4*>(p.part_o + (((size_t)kh * R_all + v0 + r) * slots + it.slot) * HD + d) = o;
        }
      }
      if (row_ok && !p.causal) *reinterpret_cast<float2*>(p.part_ml + idx * 2) = make_float2(m_used, l);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == NQ * 4 + 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)C::COLS) : "memory");
}

// A row of queries with all heads of its group has to fit a block.
bool attn_tc_shape(const AttnArgs& a) { return a.Hq / a.Hkv <= AT_ROWS; }

// Blocks and chunks of a pass.  Causal passes: two blocks a CTA where that still gives half the SMs a CTA.  Trees: the
// prefix in as many chunks (whole tiles) as two CTAs an SM take; then the longest own segment that the host's bound allows,
// in at most as many, by a CTA's time (about 2 us a tile of an own segment, one behind the other, and two and a half tiles'
// worth of fixed cost) and the waves that all CTAs make.  Unsplit, 4096 own keys of one stream (prefix 512, 32 heads of 64)
// took 71.7 us, 19.4 in 33 chunks; of eight streams 75.4 us, 49.1 us in two; 256 own keys of eight streams 16.4 us
// unsplit, 15.9 us in two chunks, 17.4 in three (a second wave).  The bound counts in whole tiles, so that the launch shape of
// a captured pass changes every 128 keys at most.
void attn_plan_tc(AttnArgs& a, int sm_count) {
  const int g = a.Hq / a.Hkv, rb = g * (AT_ROWS / g), R_all = a.n * a.T * g;
  a.stream_mode = 0;
  if (a.causal) {
    a.tc_nq = a.Hkv * ((R_all + 2 * rb - 1) / (2 * rb)) >= sm_count / 2 ? 2 : 1;
    a.n_prefix_chunks = 0; a.n_own_chunks = 0; a.prefix_chunk = a.own_chunk = AT_KEYS;
    return;
  }
  a.tc_nq = 1;
  const int blocks = (R_all + rb - 1) / rb, tiles = (a.P + AT_KEYS - 1) / AT_KEYS;
  int want = 2 * sm_count / (a.Hkv * blocks);
  if (want < 1) want = 1;
  if (want > tiles) want = tiles;
  const int per = tiles > 0 ? (tiles + want - 1) / want : 1;
  a.prefix_chunk = per * AT_KEYS;
  a.n_prefix_chunks = (tiles + per - 1) / per;
  const int rb_own = (a.T * g + rb - 1) / rb, own_tiles = (a.suffix_bound + a.T + AT_KEYS - 1) / AT_KEYS;
  const int per_chunk = a.Hkv * a.n * rb_own, others = a.n_prefix_chunks * blocks * a.Hkv;
  double best = 0.0;
  for (int c = 1; c <= own_tiles && (c == 1 || c * per_chunk <= 2 * sm_count); ++c) {
    const int own_per = (own_tiles + c - 1) / c, chunks = (own_tiles + own_per - 1) / own_per;
    const int waves = (others + chunks * per_chunk + 2 * sm_count - 1) / (2 * sm_count);
    const double cost = waves * (2.5 + (own_per > per ? own_per : per));
    if (c == 1 || cost < best) { best = cost; a.n_own_chunks = chunks; a.own_chunk = own_per * AT_KEYS; }
  }
}

static cudaError_t at_map(const void* base, int rank, const cuuint64_t* dims, const cuuint64_t* strides, const cuuint32_t* box, CUtensorMap* out) {
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
  if (enc == nullptr) return cudaErrorNotSupported;
  const CUresult r = enc(out, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, rank, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                         CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <int HD, int NQ>
static cudaError_t at_launch(const AttnArgs& a, cudaStream_t st) {
  using C = AtCfg<HD, NQ>;
  const int g = a.Hq / a.Hkv, rb = g * (AT_ROWS / g), M = a.n * a.T, R_all = M * g;
  const cuuint64_t H = sizeof(__half);
  CUtensorMap mq, mpk, mpv, mok, mov;
  cudaError_t e;
  {
    const cuuint64_t d[3] = {HD, (cuuint64_t)a.Hq, (cuuint64_t)M}, s[2] = {HD * H, a.Hq * HD * H};
    const cuuint32_t b[3] = {64, (cuuint32_t)g, (cuuint32_t)(rb / g)};
    if ((e = at_map(a.q, 3, d, s, b, &mq)) != cudaSuccess) return e;
  }
  mpk = mpv = mok = mov = mq;
  const int prefix_keys = a.causal ? a.P + a.T : a.P;      // (a causal pass's own rows lie behind the prefix)
  if (prefix_keys > 0) {
    const cuuint64_t d[3] = {HD, (cuuint64_t)prefix_keys, (cuuint64_t)a.Hkv}, s[2] = {HD * H, a.prefix_head_stride * H};
    const cuuint32_t b[3] = {64, AT_KEYS, 1};
    if ((e = at_map(a.prefix_k, 3, d, s, b, &mpk)) != cudaSuccess || (e = at_map(a.prefix_v, 3, d, s, b, &mpv)) != cudaSuccess) return e;
  }
  if (!a.causal) {
    const cuuint64_t d[4] = {HD, a.own_head_stride / HD, (cuuint64_t)a.Hkv, (cuuint64_t)a.n}, s[3] = {HD * H, a.own_head_stride * H, a.own_stream_stride * H};
    const cuuint32_t b[4] = {64, AT_KEYS, 1, 1};
    if ((e = at_map(a.own_k, 4, d, s, b, &mok)) != cudaSuccess || (e = at_map(a.own_v, 4, d, s, b, &mov)) != cudaSuccess) return e;
  }
  const int rb_all = (R_all + NQ * rb - 1) / (NQ * rb), rb_own = (a.T * g + NQ * rb - 1) / (NQ * rb);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(a.causal ? rb_all : a.n_prefix_chunks * rb_all + a.n * a.n_own_chunks * rb_own), (unsigned)a.Hkv);
  cfg.blockDim = dim3(C::THREADS); cfg.dynamicSmemBytes = C::SMEM; cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = a.pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, attn_tc_kernel<HD, NQ>, a, rb, rb_all, rb_own, 1.4426950408889634f / sqrtf((float)HD), mq, mpk, mpv, mok, mov);
}

cudaError_t launch_attention_tc(const AttnArgs& a, cudaStream_t st) {
  // (causal passes store their rows themselves; the others leave that to the merge, which takes any `out`)
  for (const void* ptr : {(const void*)a.q, (const void*)a.prefix_k, (const void*)a.prefix_v, (const void*)a.own_k, (const void*)a.own_v,
                          a.causal ? (const void*)a.out : (const void*)nullptr})
    if (reinterpret_cast<uintptr_t>(ptr) & 15) return cudaErrorMisalignedAddress;
  if (a.hd == 64) return a.tc_nq == 2 ? at_launch<64, 2>(a, st) : at_launch<64, 1>(a, st);
  return a.tc_nq == 2 ? at_launch<128, 2>(a, st) : at_launch<128, 1>(a, st);
}

cudaError_t init_attention_tc() {
  cudaError_t e;
#define AT_ATTR(HD, NQ) \
  if ((e = full_carveout(attn_tc_kernel<HD, NQ>)) != cudaSuccess) return e; \
  if ((e = cudaFuncSetAttribute(attn_tc_kernel<HD, NQ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)AtCfg<HD, NQ>::SMEM)) != cudaSuccess) return e;
  AT_ATTR(64, 1) AT_ATTR(64, 2) AT_ATTR(128, 1) AT_ATTR(128, 2)
#undef AT_ATTR
  return cudaSuccess;
}

}  // namespace mlora
