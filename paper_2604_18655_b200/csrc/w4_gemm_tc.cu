// INT4 group-quantised GEMM on the 5th-generation tensor cores for passes with many rows (DS2D verify passes, prefill
// chunks, batches of rows): Y^T[n][m] = sum_k Wdeq[k][n] h[m][k]  (Sec. 3.1 projections with the INT4 weights of
// Sec. 3.3), the LoRA expand T B (Eq. 1-4, second factor) as further k-steps, and the projection's epilogue, in one kernel.
//
// "Swap-AB": the 128 output features of a CTA are the UMMA M dimension, NR rows the N dimension.  Warp roles:
//   - groups of four warps dequantise, two groups up to 128 rows and four beyond: group q takes every second (fourth) k-step
//     (64 input features) from step q on, two n-tiles (32 features) a warp.  The packed bytes come through a private cp.async ring; ldmatrix hands every lane the words of
//     its k16 slices, dequant8() unpacks them (exactly fp16(q * scale), as on every other path), and one tcgen05.st per
//     n-tile puts them into TENSOR MEMORY, where the MMA reads its A operand.  The dequantised weights therefore never
//     touch shared memory, which only carries the activations, and no proxy fence is needed per step.
//   - one thread issues the TMA copies of the activation tiles (128-byte swizzle, rows past M read as zero),
//   - one thread issues the MMAs (4 x K 16 per step, fp32 accumulator in tensor memory).
// Adapters: T = s x A^T arrives as an fp16 matrix [M][segment][value | rounding remainder][slot * rank + j, round and round]
// that is zero outside the row's own slot (a slot = a stream of the pass, or an adapter of the single-projection call), so
// that y += T B is two more MMAs per 64 (slot, rank) indices with B as the A operand, read from the caller's matrices by the
// dequantising warps.  Value + remainder keep T at fp32 accuracy.
// Few output features and many SMs: a cluster of S CTAs splits K, each CTA ends with NR / S rows: the others push their
// accumulators into its shared memory (distributed shared memory, reused activation tiles) and it adds them in rank order
// -- no partial sums in global memory, bit-reproducible.
// RMSNorm: the producer of the residual writes x * gain (fp16, large rows scaled down: row_down) and the rows' sums of squares
// (fixed point, order independent); this kernel scales its finished sums by 1/rms.
// Every mbarrier wait is bounded; a wait that runs out sets the status word and the CTA winds down (it still waits,
// bounded, for its MMAs and copies, takes its cluster barriers, and frees its tensor memory).
#include <cuda.h>
#include <cudaTypedefs.h>

#include "tc.cuh"

namespace mlora {

constexpr int TC_BM = 128;                 // output features per CTA (UMMA M)
constexpr int TC_BK = 64;                  // input features per step: one 128-byte swizzle row of fp16
constexpr int TC_WSLOT = 1024 + 64;        // ring slot of a warp: two tiles of nibbles, two scale entries

// GR = groups of four dequantising warps: two where two CTAs share an SM, four where one has it alone (beyond 128 rows, and
// smaller tiles whose grid leaves every CTA an SM: launch_gemm_tc).
// Weight stages in tensor memory (32 columns each, behind the NR accumulator columns), activation tiles, ring depth in
// visits; the accumulator and the stages fill 256 or 512 columns.
template <int NR, int GRP> struct TcCfg {
  static constexpr int GR = GRP, OCC = GR == 2 ? 2 : 1, COLS = NR > 128 ? 512 : 256;
  static constexpr int NA = (COLS - NR) / 32 < 8 ? (COLS - NR) / 32 : 8;
  static constexpr int NB = NR == 32 ? 8 : (NR <= 96 ? 6 : 4);
  static constexpr int WD = 4;
  static constexpr int THREADS = GR * 128 + 64;       // + one warp for the activation copies, one for the MMAs
  static constexpr size_t SMEM = (size_t)NB * NR * TC_BK * 2 + (size_t)WD * GR * 4 * TC_WSLOT + 1024;
};

template <int NR, int S, int EPI, int GRP>
__global__ void __launch_bounds__(TcCfg<NR, GRP>::THREADS, TcCfg<NR, GRP>::OCC)
w4_gemm_tc_kernel(const __grid_constant__ GemmArgs p, int* status, const __grid_constant__ CUtensorMap act_map,
                  const __grid_constant__ CUtensorMap text_map) {
  using C = TcCfg<NR, GRP>;
  constexpr int NA = C::NA, NB = C::NB, WD = C::WD, GR = C::GR, TC_WARPS = GR * 4;
  constexpr uint32_t B_BYTES = NR * TC_BK * 2;
  constexpr int CW = NR / S;                          // rows (accumulator columns) this CTA finishes
  extern __shared__ __align__(1024) unsigned char tc_smem_raw[];
  // 1024-byte aligned activation tiles (the swizzle pattern is tied to address bits 7..9), then the warps' weight rings
  unsigned char* const base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(tc_smem_raw) + 1023) & ~(uintptr_t)1023);
  unsigned char* const wring = base + (size_t)NB * B_BYTES;
  __shared__ __align__(8) uint64_t b_full[NB], b_empty[NB], a_full[NA], a_empty[NA], done_bar, acc_free;
  __shared__ uint32_t tmem_base_s;
  __shared__ __align__(16) float s_inv[CW];                         // the factor of the finished sums; EPI_RESID: of the new fp16 rows
  __shared__ unsigned long long s_ssq[2][CW];
  __shared__ int s_pos[CW];                           // EPI_QKV: the rows' positions ...
  __shared__ size_t s_dst[CW];                        // ... and their places in the cache

  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int rank = S > 1 ? (int)blockIdx.x : 0;       // position in the K-splitting cluster
  const WLayout L = make_wlayout(p.K, p.N, p.G);
  const int slabs = (p.N + TC_BM - 1) / TC_BM, tiles = slabs * ((p.M + NR - 1) / NR);

  const int first = blockIdx.y + blockIdx.z * gridDim.y, stride = gridDim.y * gridDim.z;
  const bool single = stride >= tiles;                // (then the grid is slabs x row blocks)

  // ---- a tile = 128 output features x NR rows.  Its steps: KT k-tiles of the weights, then the expand's blocks of 64
  // (slot, rank index) pairs, per segment that the features touch; a CTA of a cluster takes a contiguous share of them.
  struct Tile { int slab, m0, seg0, nE, kb0, u0, u1; };
  auto stream_of = [&](int m) { return p.stream_magic ? (int)__umulhi((unsigned)m, p.stream_magic) : m; };   // m / rows per stream
  auto tile_of = [&](int t) {
    Tile x;
    // (one tile a CTA: no division)
    const int mb = single ? (int)blockIdx.z : t / slabs;
    x.slab = single ? (int)blockIdx.y : t - mb * slabs; x.m0 = mb * NR;
    x.seg0 = 0; x.nE = 0; x.kb0 = 0;
    int nseg_in = 0;
    if (p.lora.text != nullptr) {
      int s_lo = 0, s_hi = p.lora.k_slots - 1;
      if (!p.lora.slot_is_adapter) { s_lo = stream_of(x.m0); s_hi = min(s_hi, stream_of(min(p.M, x.m0 + NR) - 1)); }
      x.kb0 = (s_lo * p.lora.rank) & ~63;
      x.nE = ((s_hi + 1) * p.lora.rank - x.kb0 + 63) >> 6;
      int c, seg1;
      map_col(p.mode, x.slab * TC_BM, p.seg_n0, p.seg_n1, x.seg0, c);
      map_col(p.mode, min(p.N, x.slab * TC_BM + TC_BM) - 1, p.seg_n0, p.seg_n1, seg1, c);
      if (p.mode == MODE_GATEUP) { x.seg0 = 0; seg1 = 1; }
      nseg_in = seg1 - x.seg0 + 1;
    }
    // (an expand step counts as three: two activation tiles, and its weights are not on their way long before)
    const int ext = x.nE * nseg_in, total = L.KT + 3 * ext;
    auto cut = [&](int q) { const int w = (total * q) / S; return w <= L.KT ? w : (q == S ? L.KT + ext : L.KT + (w - L.KT) / 3); };
    x.u0 = cut(rank); x.u1 = cut(rank + 1);
    return x;
  };
  // n-tile (16 features) of the slab that lanes 16 h .. 16 h + 15 of accumulator quarter q hold: consecutive ones; with
  // RoPE in the epilogue a pair of tiles half a head apart, so that a feature's partner sits 16 lanes on
  const int rope_gap = EPI == EPI_QKV ? p.hd >> 5 : 0;   // 2 (hd 64) or 4 (hd 128) tiles
  auto ntile_of = [&](int q, int h) { return rope_gap == 0 ? 2 * q + h : (rope_gap == 4 ? q + 4 * h : (q >> 1) * 4 + (q & 1) + 2 * h); };

  if (tid == 0) {
    for (int s = 0; s < NB; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem_u32(b_full + s)) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem_u32(b_empty + s)) : "memory");
    }
    for (int s = 0; s < NA; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 4;" ::"r"(tc_smem_u32(a_full + s)) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem_u32(a_empty + s)) : "memory");
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem_u32(&done_bar)) : "memory");
    TC_MBAR_INIT(&acc_free, TC_WARPS);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == TC_WARPS + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem_u32(&tmem_base_s)), "r"((uint32_t)C::COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_base_s, 0);
  bool alive = true;
  // this CTA's share of the next projection's weights, asked for in L2: that kernel starts when this one is done and then
  // finds its first tiles a short trip away (from HBM they took 1.8 us of a 9 us CTA)
  if (tid == TC_WARPS * 32 + 32 && p.pf_bytes != 0) {
    const unsigned n_cta = gridDim.x * gridDim.y * gridDim.z, cta = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    const unsigned per = ((p.pf_bytes / n_cta) + 15u) & ~15u, b0 = per * cta, b1 = min(b0 + per, p.pf_bytes & ~15u);
    for (unsigned o = b0; o < b1; o += 16384u)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p.pf_w + o), "r"(min(b1 - o, 16384u)) : "memory");
  }

  if (warp == TC_WARPS) {
    // ---- activation copies (the warp waits, an elected lane issues): x = multiples of 64 features, rows m0 ..
    {
      // programmatic launch: set-up and the first weights run while the kernel ahead finishes.  With late_wait the
      // kernel ahead only produces T: the activations were complete before it let this one start.
      const uint32_t elected = tc_elect();
      bool waited = false;
      if (!p.late_wait) { asm volatile("griddepcontrol.wait;" ::: "memory"); waited = true; }
      int sb = 0, issued = 0, m0 = 0; uint32_t pb = 1;
      auto copy = [&](const CUtensorMap* map, int x) {
        if (alive) alive = tc_wait(tc_smem_u32(b_empty) + 8 * sb, pb, status);
        if (!alive) return;
        if (elected) {
          const uint32_t bar = tc_smem_u32(b_full) + 8 * sb, dst = tc_smem_u32(base) + sb * B_BYTES;
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(B_BYTES) : "memory");
          asm volatile(
              "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
              ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(m0), "r"(bar) : "memory");
        }
        __syncwarp();
        ++issued;
        if (++sb == NB) { sb = 0; pb ^= 1u; }
      };
      for (int t = first; t < tiles && alive; t += stride) {
        const Tile x = tile_of(t);
        m0 = x.m0;
        for (int u = x.u0; u < x.u1 && alive; ++u) {
          if (u < L.KT) copy(&act_map, u * TC_BK);
          else {
            if (!waited) { asm volatile("griddepcontrol.wait;" ::: "memory"); waited = true; }
            const int e = u - L.KT, sg = (e >= x.nE) + (e >= 2 * x.nE), seg = x.seg0 + sg;
            const int c = (x.kb0 + (e - sg * x.nE) * 64) & p.lora.ke_mask;
            copy(&text_map, (seg * 2) * p.lora.ke + c);
            copy(&text_map, (seg * 2 + 1) * p.lora.ke + c);
          }
        }
      }
      // no copy may still be in flight when the CTA ends: the newest phase of every tile (passes at once unless a wait
      // gave up somewhere)
      for (int j = issued > NB ? issued - NB : 0; j < issued; ++j)
        tc_wait(tc_smem_u32(b_full + j % NB), (uint32_t)((j / NB) & 1), status);
    }
    __syncwarp();
  } else if (warp == TC_WARPS + 1) {
    // ---- MMA issuer.  The whole warp runs the loop and one elected lane issues: operands that the compiler can prove
    // uniform go straight into uniform registers (a lane == 0 branch around everything cost 1000 cycles a step)
    {
      // instruction descriptor: D fp32, A and B fp16, both K-major, N = NR, M = 128
      constexpr uint32_t IDESC = (1u << 4) | ((uint32_t)(NR >> 3) << 17) | ((uint32_t)(TC_BM >> 4) << 24);
      const uint32_t elected = tc_elect();
      const uint32_t base_u = tc_smem_u32(base);
      const uint32_t bf = tc_smem_u32(b_full), be = tc_smem_u32(b_empty), af = tc_smem_u32(a_full), ae = tc_smem_u32(a_empty);
      const uint32_t idesc = IDESC;
      uint32_t acc = 0;
      // the four MMAs of one step: 16 features further along K = 8 columns of the weights, 32 bytes inside the swizzled
      // 128-byte row
      auto issue = [&](int sa, int sb) {
        const uint32_t at = tmem + NR + sa * 32;
        const uint64_t bdesc = tc_desc(base_u + sb * B_BYTES);
#pragma unroll
        for (int kk = 0; kk < TC_BK / 16; ++kk)
          asm volatile(
              "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
              "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
              ::"r"(tmem), "r"(at + kk * 8), "l"(bdesc + (uint64_t)(kk * 2)), "r"(idesc), "r"(kk > 0 ? 1u : acc) : "memory");
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(be + 8 * sb) : "memory");
        acc = 1;
      };
      auto release = [&](int sa) {
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(ae + 8 * sa) : "memory");
      };
      int sa = 0, sb = 0; uint32_t pa = 0, pb = 0, p_acc = 1;
      for (int t = first; t < tiles && alive; t += stride) {
      const Tile x = tile_of(t);
      const int nsteps = x.u1 - x.u0, n_main = max(0, min(L.KT, x.u1) - x.u0);
      // the accumulator is the epilogue's until it has read it
      alive = tc_wait(tc_smem_u32(&acc_free), p_acc, status);
      p_acc ^= 1u;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      acc = 0;
      int i = 0;
      // two steps a round: a test of a barrier costs about 90 cycles even when its phase is over, as much as the MMAs of
      // a step of 32 rows, so the four tests of a round go out together
#pragma unroll 1
      for (; i + 2 <= n_main && alive; i += 2) {
        const int sa1 = sa + 1 == NA ? 0 : sa + 1, sb1 = sb + 1 == NB ? 0 : sb + 1;
        const uint32_t pa1 = sa1 ? pa : pa ^ 1u, pb1 = sb1 ? pb : pb ^ 1u;
        const bool t0 = tc_test(af + 8 * sa, pa), t1 = tc_test(bf + 8 * sb, pb), t2 = tc_test(af + 8 * sa1, pa1), t3 = tc_test(bf + 8 * sb1, pb1);
        if (!(t0 && t1)) alive = tc_wait(af + 8 * sa, pa, status) && tc_wait(bf + 8 * sb, pb, status);
        if (!alive) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (elected) { issue(sa, sb); release(sa); }
        __syncwarp();
        if (!(t2 && t3)) alive = tc_wait(af + 8 * sa1, pa1, status) && tc_wait(bf + 8 * sb1, pb1, status);
        if (!alive) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        acc = 1;
        if (elected) { issue(sa1, sb1); release(sa1); }
        __syncwarp();
        sa = sa1 + 1 == NA ? 0 : sa1 + 1; pa = sa ? pa1 : pa1 ^ 1u;
        sb = sb1 + 1 == NB ? 0 : sb1 + 1; pb = sb ? pb1 : pb1 ^ 1u;
      }
      // a last odd step; the expand's steps, whose weights meet two activation tiles (value, remainder)
#pragma unroll 1
      for (; i < nsteps && alive; ++i) {
        alive = tc_wait(af + 8 * sa, pa, status);
        for (int part = i < n_main ? 1 : 0; part < 2 && alive; ++part) {
          alive = tc_wait(bf + 8 * sb, pb, status);
          if (!alive) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          if (elected) { issue(sa, sb); if (part == 1) release(sa); }
          acc = 1;
          __syncwarp();
          if (++sb == NB) { sb = 0; pb ^= 1u; }
        }
        if (++sa == NA) { sa = 0; pa ^= 1u; }
      }
      if (elected) tc_commit(tc_smem_u32(&done_bar));
      __syncwarp();
      }
    }
  } else {
    // ---- dequantising warps: group grp takes every other step, quarter wq the features 32 wq .. 32 wq + 31
    const int grp = warp >> 2, wq = warp & 3, g = lane >> 2;
    const int gshift = L.G == 64 ? 0 : (L.G == 128 ? 1 : (L.G == 256 ? 2 : 3));   // k-tiles per scale entry, log2
    const uint32_t ring0 = tc_smem_u32(wring) + (uint32_t)(warp * WD) * TC_WSLOT;
    // lane 4g + j of a tile owns features 16j .. 16j + 15 of its rows; its 16 bytes go to piece (j, g), so that ldmatrix
    // (matrix j = the eight rows' pieces) hands lane (g, t) word t of them: features 16j + 4t .. + 3, the order in which
    // the fragment store below lays k16 slice j down
    const uint32_t dpos = (uint32_t)((lane & 3) * 128 + (lane >> 2) * 16);
    // The loop is bound by the instructions it issues (about 130 a visit, 72 of them the unpacking of 64 weights a lane),
    // so the fetch keeps running pointers: k-tile f_r of its chunk, the tile's bytes, the chunk's scale entries
    int f_left = 0, f_r = 0, f_c = 0;                       // fetches still to issue in this tile
    const unsigned char *f_w = nullptr, *f_s = nullptr;
    ptrdiff_t f_d = 0;
    uint32_t f_dst = ring0;
    const uint32_t ring_end = ring0 + WD * TC_WSLOT;
    auto fetch_tile = [&](const Tile& x) {                  // the running pointers at the warp's first step of a tile
      // past the last n-tile the warp reads tile 0 again: those accumulator lanes are never stored
      const int nt0 = x.slab * (TC_BM / TILE_N) + ntile_of(wq, 0), nt1 = x.slab * (TC_BM / TILE_N) + ntile_of(wq, 1);
      const unsigned char* const unit0 = p.w + (size_t)(nt0 < L.NT ? nt0 : 0) * L.unit_bytes;
      const unsigned char* const unit1 = p.w + (size_t)(nt1 < L.NT ? nt1 : 0) * L.unit_bytes;
      f_left = (min(x.u1, L.KT) - x.u0 - grp + GR - 1) / GR;
      f_r = (x.u0 + grp) & 7; f_c = (x.u0 + grp) >> 3;
      f_w = unit0 + (size_t)f_c * L.chunk_full + f_r * 512 + lane * 16;
      f_d = unit1 - unit0;
      f_s = (lane & 2 ? unit1 : unit0) + (size_t)f_c * L.chunk_full + (f_c == L.nchunks - 1 ? L.kc_last : CHUNK_KT) * 512 + (lane & 1) * 16;
    };
    auto fetch_w = [&]() {
      if (f_left > 0) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(f_dst + dpos), "l"(f_w) : "memory");
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(f_dst + 512 + dpos), "l"(f_w + f_d) : "memory");
        if (lane < 4)                                     // two scale entries of 32 bytes
          asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(f_dst + 1024 + lane * 16), "l"(f_s + ((f_r >> gshift) << 5)) : "memory");
        --f_left;
        f_r += GR; f_w += GR * 512;
        if (f_r >= CHUNK_KT) {
          f_r -= CHUNK_KT; f_w += L.chunk_full - CHUNK_KT * 512; f_s += L.chunk_full;
          if (++f_c == L.nchunks - 1) f_s -= (CHUNK_KT - L.kc_last) * 512;
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      f_dst = f_dst + TC_WSLOT == ring_end ? ring0 : f_dst + TC_WSLOT;
    };
    // lane l looks up the addresses (column 0) of B's rows for the (slot, rank index) pairs k0 + l and k0 + 32 + l
    auto expand_rows = [&](int seg, int k0, unsigned long long (&adr)[2]) {
      const int r = p.lora.rank, ldb = p.lora.seg[seg].n;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int k = k0 + h * 32 + lane, s = k / r, j = k - s * r;
        adr[h] = 0ull;
        if (s < p.lora.k_slots) {
          const int a = p.lora.slot_is_adapter ? s : __ldg(p.lora.adapter_idx + s);
          const __half* B = (a >= 0 && a < p.lora.n_slots) ? p.lora.tabB[(size_t)a * p.lora.tab_stride + p.lora.seg[seg].proj_index] : nullptr;
          if (B != nullptr) adr[h] = (unsigned long long)(B + (size_t)j * ldb);
        }
      }
    };
    uint32_t slot = ring0;                                // ring slot consumed next
    const uint32_t ae = tc_smem_u32(a_empty), af = tc_smem_u32(a_full);
    const uint32_t lane_t = tmem + NR + ((uint32_t)(wq * 32) << 16);
    int sa = grp; uint32_t pa = 1;                        // stage of step i, parity of its "free" phase
    auto stage_free = [&](bool tested) {
      if (!__all_sync(0xffffffffu, tested)) {
        if (alive) alive = tc_wait(ae + 8 * sa, pa, status);
        alive = __all_sync(0xffffffffu, alive);
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    };
    auto stage_done = [&]() {
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(af + 8 * sa) : "memory");
    };
    // stages are dealt out by the running step count of the CTA
    auto next_stage = [&]() {
      sa += GR;
      if (sa >= NA) { sa -= NA; pa ^= 1u; }
    };
    fetch_tile(tile_of(first));
#pragma unroll 1
    for (int j = 0; j < WD; ++j) fetch_w();
    uint32_t p_done = 0;
    bool waited = false;
#pragma unroll 1
    for (int t = first; t < tiles; t += stride) {
    const Tile x = tile_of(t);
    const int u0 = x.u0, nsteps = x.u1 - x.u0, u_end = min(x.u1, L.KT);
    int i = grp;
#pragma unroll 1
    for (; u0 + i < u_end; i += GR) {
      const bool a_free = tc_test(ae + 8 * sa, pa);       // (its latency passes under the unpacking)
      asm volatile("cp.async.wait_group %0;" ::"n"(WD - 1) : "memory");
      __syncwarp();
      uint32_t w0[4], w1[4], sc0, sc1;
      asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                   : "=r"(w0[0]), "=r"(w0[1]), "=r"(w0[2]), "=r"(w0[3]) : "r"(slot + lane * 16) : "memory");
      asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                   : "=r"(w1[0]), "=r"(w1[1]), "=r"(w1[2]), "=r"(w1[3]) : "r"(slot + 512 + lane * 16) : "memory");
      asm volatile("ld.shared.u32 %0, [%1];" : "=r"(sc0) : "r"(slot + 1024 + g * 4) : "memory");
      asm volatile("ld.shared.u32 %0, [%1];" : "=r"(sc1) : "r"(slot + 1024 + 32 + g * 4) : "memory");
      slot = slot + TC_WSLOT == ring_end ? ring0 : slot + TC_WSLOT;
      uint32_t r0[16], r1[16];
      {
        auto unpack = [](const uint32_t (&w)[4], const auto& f, uint32_t (&r)[16]) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            uint32_t a[4];
            dequant8(w[j], f, a);
            r[4 * j] = a[0]; r[4 * j + 1] = a[2]; r[4 * j + 2] = a[1]; r[4 * j + 3] = a[3];
          }
        };
        if (__all_sync(0xffffffffu, (w4_odd(sc0) | w4_odd(sc1)) == 0u)) {
          unpack(w0, W4Scales<0>(sc0), r0);
          unpack(w1, W4Scales<0>(sc1), r1);
        } else {
          unpack(w0, W4Scales<2>(sc0), r0);
          unpack(w1, W4Scales<2>(sc1), r1);
        }
      }
      stage_free(a_free);
      tc_st_16x256b_x4(lane_t + sa * 32, r0);
      tc_st_16x256b_x4(lane_t + sa * 32 + (16u << 16), r1);
      fetch_w();                                          // refills the slot just read, while the stores finish
      stage_done();
      next_stage();
    }
#pragma unroll 1
    for (; i < nsteps; i += GR) {
      {
        // 64 (slot, rank index) pairs of the expand: lane = output feature, two rank
        // indices a column
        const int e = u0 + i - L.KT, sg = (e >= x.nE) + (e >= 2 * x.nE), seg = x.seg0 + sg, k0 = x.kb0 + (e - sg * x.nE) * 64;
        unsigned long long adr[2];
        expand_rows(seg, k0, adr);
        // [64 pairs][32 features] through the warp's ring (its weight steps are all done): 16-byte pieces in, columns out
        {
          const int piece = lane & 3, n = x.slab * TC_BM + ntile_of(wq, piece >> 1) * TILE_N + (piece & 1) * 8;
          int my_seg = -1, col = 0;
          if (n < p.N) map_col(p.mode, n, p.seg_n0, p.seg_n1, my_seg, col);
          asm volatile("cp.async.wait_group 0;" ::: "memory");
          __syncwarp();
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            const int k = c * 8 + (lane >> 2);
            const unsigned long long ad = __shfl_sync(0xffffffffu, adr[c >> 2], k & 31);
            const bool ok = my_seg == seg && ad != 0ull;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                         ::"r"(ring0 + (uint32_t)(k * 64 + piece * 16)), "l"(ok ? ad + (unsigned long long)col * 2 : (unsigned long long)p.w), "r"(ok ? 16 : 0) : "memory");
          }
          asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
          __syncwarp();
        }
        uint32_t v[2][16];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int c = 0; c < 16; ++c) {
            unsigned short b0, b1;
            const uint32_t src = ring0 + (uint32_t)((h * 32 + c * 2) * 64 + lane * 2);
            asm volatile("ld.shared.u16 %0, [%1];" : "=h"(b0) : "r"(src) : "memory");
            asm volatile("ld.shared.u16 %0, [%1];" : "=h"(b1) : "r"(src + 64) : "memory");
            v[h][c] = (uint32_t)b0 | ((uint32_t)b1 << 16);
          }
        __syncwarp();
        stage_free(false);
        tc_st_32x32b_x16(lane_t + sa * 32, v[0]);
        tc_st_32x32b_x16(lane_t + sa * 32 + 16, v[1]);
      }
      stage_done();
      next_stage();
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    const int slab = x.slab, m0 = x.m0;
    const bool more = S == 1 && t + stride < tiles;
    if (more) {                                            // the next tile's first weights, under the epilogue
      sa += nsteps + grp - i;                              // (from where step i would have been to step grp of the next tile)
      if (sa >= NA) { sa -= NA; pa ^= 1u; }
      else if (sa < 0) { sa += NA; pa ^= 1u; }
      fetch_tile(tile_of(t + stride));
      f_dst = slot = ring0;
#pragma unroll 1
      for (int j = 0; j < WD; ++j) fetch_w();
    }

    // ---- epilogue: lane = output feature, accumulator columns = rows
    const int lq = wq, half = grp;                         // GR warps share a lane quarter's columns
    const int n = slab * TC_BM + ntile_of(lq, lane >> 4) * TILE_N + (lane & 15);
    const bool n_ok = n < p.N;
    if (!waited) { asm volatile("griddepcontrol.wait;" ::: "memory"); waited = true; }   // (every earlier kernel's results)
    const int row0 = m0 + rank * CW;                       // rows this CTA finishes: row0 .. row0 + CW - 1
    if (tid < CW) {
      float inv = 1.f;
      if (EPI == EPI_RESID) {
        if (p.xg_out != nullptr && row0 + tid < p.M) inv = row_down(__ldcg(p.ssq_out_prev + p.ssq_hi + row0 + tid), p.N);
        s_ssq[0][tid] = s_ssq[1][tid] = 0ull;
      } else if (p.ssq_in != nullptr && row0 + tid < p.M) {
        inv = norm_factor(p.ssq_in + row0 + tid, p.ssq_in_prev + row0 + tid, p.ssq_hi, p.K, p.eps);
      }
      s_inv[tid] = inv;
      s_pos[tid] = 0;
      if (EPI == EPI_QKV && row0 + tid < p.M) {
        const int m = row0 + tid, st = stream_of(m), cached = p.suffix_len[st];
        s_pos[tid] = p.pos_base + cached + p.depth[m];
        s_dst[tid] = (size_t)st * p.kv_stream_stride + (size_t)(cached + m - st * p.rows_per_stream) * p.hd;
      }
    }
    constexpr int HC = CW / GR;                            // columns of a warp
    // columns handled at a time: 8 where the next tile's state is held beside the chunk's old rows or table entries (with 16 these
    // kernels spilled; llama3b, prompt of 1999 13.95 ms, 13.64 so, llama1b, of 512 1.530 and 1.509 ms)
    constexpr int CH_MAX = S == 1 && (EPI == EPI_RESID || EPI == EPI_QKV) ? 8 : 16, CH = HC < CH_MAX ? HC : CH_MAX;
    static_assert(HC % CH == 0 && CH >= 2 && (S == 1 || NR % (GR * 16) == 0), "a warp's columns: whole chunks, pairs of rows, whole loads");
    const int c_lo = half * HC;
    // (The epilogue is bound by the instructions it issues, 25 to 47 an output by way of an address and a bound for each: pointers
    // that step, one bound a chunk.  llama1b, two passes of 128 rows 2.49 -> 2.45 ms, llama3b, of 256 rows 7.67 -> 7.47, prompt of 100 on llama1b
    // 0.805 -> 0.777.)
    auto rows_of = [&](int c0) { return n_ok ? p.M - row0 - c0 : 0; };   // rows of the lane's feature from column c0 on (may be negative)
    float x_old[CH], gain = 1.f;
    auto prefetch_resid = [&](int c0) {
      const float* x = p.resid + (size_t)(row0 + c0) * p.N + n;
      const int rows = rows_of(c0);
#pragma unroll
      for (int j = 0; j < CH; ++j, x += p.N)
        if (j < rows) x_old[j] = __ldcg(x);
    };
    // EPI_QKV: segment and column of the lane's feature; a warp's lanes lie in one head
    int seg = 0, col = 0;
    if (EPI == EPI_QKV && n_ok) map_col(p.mode, n, p.seg_n0, p.seg_n1, seg, col);
    const int hh = p.hd >> 1, d = col & (p.hd - 1);
    const bool rope = EPI == EPI_QKV && __any_sync(0xffffffffu, n_ok && seg < 2);
    float2 cs[CH];
    auto prefetch_cs = [&](int c0) {                       // table entries of a chunk, all in flight (rows past the end: position 0)
      const float2* const tab = p.cs_table + (d & (hh - 1));
#pragma unroll
      for (int j = 0; j < CH; ++j) cs[j] = __ldg(tab + (unsigned)(s_pos[c0 + j] * hh));
    };
    if (EPI == EPI_RESID) {
      prefetch_resid(c_lo);
      if (p.xg_out != nullptr && n_ok) gain = __half2float(__ldg(p.gain_next + n));
    }
    // the tile's MMAs are done (also when a stage wait gave up earlier: wait, bounded, before touching anything)
    const bool done = tc_wait(tc_smem_u32(&done_bar), p_done, status);
    p_done ^= 1u;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (!more) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("bar.sync 1, %0;" ::"n"(TC_WARPS * 32) : "memory");
    if (EPI == EPI_QKV && rope) prefetch_cs(c_lo);
    float* const xch = reinterpret_cast<float*>(base);     // [S][CW][128] partial sums for the rows this CTA finishes
    if constexpr (S > 1) {                                 // (a cluster has one tile: its activation tiles are free now)
      asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
      const uint32_t my = tc_smem_u32(xch) + (uint32_t)((rank * CW) * TC_BM + lq * 32 + lane) * 4u;
#pragma unroll 1
      for (int c0 = half * (NR / GR); c0 < (half + 1) * (NR / GR); c0 += 16) {
        float v[16];
        tc_ld_32x32b_x16(tmem + ((uint32_t)(lq * 32) << 16) + (uint32_t)c0, v);
        constexpr int PER = CW < 16 ? CW : 16;              // columns in a row that go to the same CTA
#pragma unroll
        for (int j0 = 0; j0 < 16; j0 += PER) {
          uint32_t dst;
          asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"(my), "r"((c0 + j0) / CW));
          dst += (uint32_t)((c0 + j0) % CW) * (TC_BM * 4u);
#pragma unroll
          for (int j = 0; j < PER; ++j)
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dst + (uint32_t)j * (TC_BM * 4u)), "f"(v[j0 + j]) : "memory");
        }
      }
      asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
    const bool fine = __all_sync(0xffffffffu, done && alive);
#pragma unroll 1
    for (int c0 = c_lo; c0 < c_lo + HC && fine; c0 += CH) {
      float v[16];
      if constexpr (S > 1) {
#pragma unroll
        for (int j = 0; j < CH; ++j) v[j] = 0.f;
#pragma unroll
        for (int q = 0; q < S; ++q)
#pragma unroll
          for (int j = 0; j < CH; ++j) v[j] += xch[(size_t)(q * CW + c0 + j) * TC_BM + lq * 32 + lane];
      } else {
        if constexpr (CH == 8) tc_ld_32x32b_x8(tmem + ((uint32_t)(lq * 32) << 16) + (uint32_t)c0, v);
        else tc_ld_32x32b_x16(tmem + ((uint32_t)(lq * 32) << 16) + (uint32_t)c0, v);
      }
      float inv[CH];
      if (EPI == EPI_RESID || p.ssq_in != nullptr) {
        if constexpr (CH % 4 == 0) {
#pragma unroll
          for (int j = 0; j < CH; j += 4) *reinterpret_cast<float4*>(inv + j) = *reinterpret_cast<const float4*>(s_inv + c0 + j);
        } else {
#pragma unroll
          for (int j = 0; j < CH; ++j) inv[j] = s_inv[c0 + j];
        }
        if (EPI != EPI_RESID)
#pragma unroll
          for (int j = 0; j < CH; ++j) v[j] *= inv[j];
      }
      const int rows = rows_of(c0);
      if constexpr (EPI == EPI_F32) {
        float* o = p.out_f32 + (size_t)(row0 + c0) * p.ldo + n;
#pragma unroll
        for (int j = 0; j < CH; ++j, o += p.ldo)
          if (j < rows) *o = v[j];
      } else if constexpr (EPI == EPI_QKV) {
        // RoPE on q and k (pairs (i, i + hd/2): 16 lanes on), fp16, q to its matrix, k and v into the stream's cache
        if (rope) {
          const float sign = d < hh ? -1.f : 1.f;
#pragma unroll
          for (int j = 0; j < CH; ++j) {
            const float o = __shfl_xor_sync(0xffffffffu, v[j], 16);
            v[j] = v[j] * cs[j].x + (sign * o) * cs[j].y;
          }
          if (c0 + CH < c_lo + HC) prefetch_cs(c0 + CH);
        }
        if (seg == 0) {
          __half* dst = p.q_out + (size_t)(row0 + c0) * p.seg_n0 + col;
#pragma unroll
          for (int j = 0; j < CH; ++j, dst += p.seg_n0)
            if (j < rows) *dst = __float2half_rn(v[j]);
        } else {
          __half* const dst = (seg == 1 ? p.k_out : p.v_out) + (size_t)(col / p.hd) * p.kv_head_stride + d;
#pragma unroll
          for (int j = 0; j < CH; ++j)
            if (j < rows) dst[s_dst[c0 + j]] = __float2half_rn(v[j]);
        }
      } else if constexpr (EPI == EPI_SWIGLU) {
        // lanes 0-15 hold a gate tile's features, lanes 16-31 the up tile's: of every two rows the lower half takes the
        // first, the upper half the second
        const bool lo = lane < 16;
        const int F = p.N >> 1, second = lo ? 0 : 1;
        __half* dst = p.out_f16 + (size_t)(row0 + c0 + second) * F + (((n >> 5) << 4) | (n & 15));
#pragma unroll
        for (int j = 0; j < CH; j += 2, dst += 2 * F) {
          const float got = __shfl_xor_sync(0xffffffffu, lo ? v[j + 1] : v[j], 16);
          const float gt = lo ? v[j] : got, up = lo ? got : v[j + 1];
          if (j < rows - second) *dst = __float2half_rn(gt / (1.f + __expf(-gt)) * up);
        }
      } else {
        float xn[CH];
        float* x = p.resid + (size_t)(row0 + c0) * p.N + n;
        __half* xg = p.xg_out != nullptr ? p.xg_out + (size_t)(row0 + c0) * p.N + n : nullptr;
#pragma unroll
        for (int j = 0; j < CH; ++j, x += p.N) {
          xn[j] = j < rows ? x_old[j] + v[j] : 0.f;
          if (j < rows) *x = xn[j];
        }
        if (p.xg_out != nullptr) {
#pragma unroll
          for (int j = 0; j < CH; ++j, xg += p.N)
            if (j < rows) *xg = __float2half_rn(xn[j] * gain * inv[j]);
        }
        if (c0 + CH < c_lo + HC) prefetch_resid(c0 + CH);
        if (p.ssq_out != nullptr) {
          // sums of squares over the warp's 32 features for CH rows: a butterfly that halves the rows a lane keeps
          float q[CH];
#pragma unroll
          for (int j = 0; j < CH; ++j) q[j] = xn[j] * xn[j];
          int id = 0;
          int w = CH;
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            if (w > 1) {
              w >>= 1;
              const bool up = (lane & o) != 0;
#pragma unroll
              for (int j = 0; j < CH / 2; ++j) {
                if (j < w) {
                  const float got = __shfl_xor_sync(0xffffffffu, up ? q[j] : q[j + w], o);
                  q[j] = (up ? q[j + w] : q[j]) + got;
                }
              }
              id = id * 2 + (up ? 1 : 0);
            } else {
              q[0] += __shfl_xor_sync(0xffffffffu, q[0], o);
            }
          }
          constexpr int DUP = 32 / CH;                     // lanes that hold the same row's sum
          if ((lane & (DUP - 1)) == 0) {
            const bool large = ssq_is_large(q[0]);
            atomicAdd(&s_ssq[large][c0 + id], (unsigned long long)__float2ll_rn(large ? q[0] : q[0] * 4294967296.f));
          }
        }
      }
    }
    // the accumulator may be overwritten; the rows' sums of squares, complete, to where they are collected
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncwarp();
    if (lane == 0) tc_arrive(tc_smem_u32(&acc_free));
    asm volatile("bar.sync 1, %0;" ::"n"(TC_WARPS * 32) : "memory");
    if (EPI == EPI_RESID && p.ssq_out != nullptr && tid < CW && row0 + tid < p.M) {
      atomicAdd(p.ssq_out + row0 + tid, s_ssq[0][tid]);
      const unsigned long long more = s_ssq[1][tid], bits = (more != 0ull ? SSQ_LARGE : 0ull) | (s_inv[tid] != 1.f ? SSQ_SCALED : 0ull);
      if (more != 0ull) atomicAdd(p.ssq_out + p.ssq_hi + row0 + tid, more);
      if (bits != 0ull) ssq_mark(p.ssq_out + row0 + tid, bits);
    }
    if (!more) break;
    }
  }
  if constexpr (S > 1) {
    if (warp >= TC_WARPS) {                                // (the other warps took both barriers in the epilogue)
      asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
      asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == TC_WARPS + 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)C::COLS) : "memory");
}

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = []() -> PFN_cuTensorMapEncodeTiled_v12000 {
    void* sym = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return nullptr;
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(sym);
  }();
  return fn;
}

// rank-2 fp16 map over a row-major matrix [M][ld]: box = 64 columns x nrows rows, 128-byte swizzle, zero fill
static cudaError_t encode_row_map(const __half* base, int ld, int M, int nrows, CUtensorMap* map) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
  if (enc == nullptr) return cudaErrorNotSupported;
  const cuuint64_t dims[2] = {(cuuint64_t)ld, (cuuint64_t)M};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * sizeof(__half)};
  const cuuint32_t box[2] = {(cuuint32_t)TC_BK, (cuuint32_t)nrows};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<__half*>(base), dims, strides, box, estr,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <int NR, int S, int EPI, int GRP>
static cudaError_t tc_launch(const GemmArgs& a, int sm_count, int* status, cudaStream_t st) {
  CUtensorMap map, tmap;
  cudaError_t e = encode_row_map(a.h, a.K, a.M, NR, &map);
  if (e != cudaSuccess) return e;
  tmap = map;
  if (a.lora.text != nullptr) e = encode_row_map(a.lora.text, a.lora.nseg * 2 * a.lora.ke, a.M, NR, &tmap);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  // one CTA (or cluster) a tile; CTAs that have their K to themselves stay and take further tiles
  const int tiles = (a.N + TC_BM - 1) / TC_BM * ((a.M + NR - 1) / NR);
  if (S == 1 && tiles > sm_count * TcCfg<NR, GRP>::OCC) cfg.gridDim = dim3(1, (unsigned)(sm_count * TcCfg<NR, GRP>::OCC));
  else cfg.gridDim = dim3(S, (unsigned)((a.N + TC_BM - 1) / TC_BM), (unsigned)((a.M + NR - 1) / NR));
  cfg.blockDim = dim3(TcCfg<NR, GRP>::THREADS); cfg.dynamicSmemBytes = TcCfg<NR, GRP>::SMEM; cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = S; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = S > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, w4_gemm_tc_kernel<NR, S, EPI, GRP>, a, status, map, tmap);
}

#define TC_FOR_EACH(X) \
  X(32, 1, 2) X(32, 2, 2) X(32, 4, 2) X(32, 8, 2) X(64, 1, 2) X(64, 2, 2) X(64, 4, 2) X(64, 8, 2) \
  X(96, 1, 2) X(128, 1, 2) X(128, 2, 2) X(128, 4, 2) X(128, 8, 2) \
  X(64, 1, 4) X(64, 2, 4) X(64, 4, 4) X(64, 8, 4) \
  X(128, 1, 4) X(128, 2, 4) X(128, 4, 4) X(128, 8, 4) \
  X(192, 1, 4) X(256, 1, 4) X(256, 2, 4) X(256, 4, 4) X(256, 8, 4)
cudaError_t init_gemm_tc() {
  cudaError_t e;
#define TC_ATTR1(NR, S, EPI, GRP) \
  if ((e = full_carveout(w4_gemm_tc_kernel<NR, S, EPI, GRP>)) != cudaSuccess) return e; \
  if ((e = cudaFuncSetAttribute(w4_gemm_tc_kernel<NR, S, EPI, GRP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcCfg<NR, GRP>::SMEM)) != cudaSuccess) return e;
#define TC_ATTR(NR, S, GRP) TC_ATTR1(NR, S, EPI_F32, GRP) TC_ATTR1(NR, S, EPI_RESID, GRP) TC_ATTR1(NR, S, EPI_SWIGLU, GRP) TC_ATTR1(NR, S, EPI_QKV, GRP)
  TC_FOR_EACH(TC_ATTR)
#undef TC_ATTR
#undef TC_ATTR1
  return cudaSuccess;
}

bool tensor_maps_available() { return tensor_map_encoder() != nullptr; }

bool gemm_tc_eligible(const GemmArgs& a) {
  if (a.M < TC_MIN_ROWS || a.N % 16 || a.K % 64) return false;
  return reinterpret_cast<uintptr_t>(a.h) % 16 == 0 && tensor_map_encoder() != nullptr;   // TMA needs both
}

// CTAs that run at once with one on an SM: clusters do not fill the machine, 33 of four CTAs and 15 of eight on 148 SMs
// (cudaOccupancyMaxActiveClusters).
static int tc_resident(int split, int sm_count) { return sm_count - (split == 4 ? 16 : (split == 8 ? 28 : 0)); }

// Four dequantising groups (GR) where a CTA has an SM for itself: in a pass (the weights are in L2, asked for by the projection
// ahead) it is the unpacking that bounds up to 128 rows, two groups take 540 cycles for a step of 64 features while the MMAs take 255
// (128 rows).  llama3b, prompt of 300 3.64 -> 3.05 ms, llama1b 1.33 -> 1.17.  Not with adapters: their shrink kernel would no
// longer start beside the projection ahead (llama1b, two passes of 240 rows 3.02 -> 3.15 ms).  Not in a call of its own, whose weights
// come from HBM: over the best candidate with two it gained at most 2 % (21 projections, 9 .. 2000 rows), and the next call's CTAs find no room.
// Not where a cluster would have to wait for a second wave (8192 x 2048, 64 rows in clusters of eight: 16.7 us, 10.1 with two groups).
static bool tc_four_groups(TcCall call, int nr, int split, long long ctas, int sm_count) {
  return nr > 128 || ((nr == 64 || nr == 128) && call == TC_PASS && ctas <= tc_resident(split, sm_count));
}

// Rows per CTA and K split, by a model of the time in microseconds: that of a step of 64 features with one or two CTAs on an SM (or
// one with four groups), set-up and epilogue, what a further wave costs (less where the CTA stays), and the exchange of a split.
// pass: fitted to all candidates of ten projections of 2048 x 2048 .. 14336 x 4096 with 16 .. 2000 rows, four groups among them (prompts of
// 100 and 512 on llama1b 0.776 -> 0.764 and 1.553 -> 1.526 ms against the constants of lora).
// alone: fitted to all candidates with two groups at half of 462 pairs of a projection (512 x 512 .. 14336 x 4096) and a row count (9 ..
// 2000), steps' times held to rise with the rows.  Against the best candidate 0.3 % more on average on the fitted half, 0.6 % on the
// other, 14 % at worst; calls of their own with the constants of pass 9.4 %, and 92 % at worst.
// lora: the expand (left out of the model) and the shrink beside the projection ahead change the order; these are the constants with
// which llama3b's tree passes were fastest (two of 256 rows 7.43 ms, 8.04 with those of pass).  Splits in eight gain there even where
// the rest of them waits (14336 x 4096, 32 rows, 8 adapters of rank 16 24.4 us, 30.4 in four).
struct TcCosts { double step1[6], step2[6], step4[6], fixed, tail, tail4, exchange, exchange4, eight, wave1, wave1_f, wave, wave_f; };
TcPlan tc_plan(int M, int K, int N, TcCall call, int sm_count) {
  static const int sizes[6] = {32, 64, 96, 128, 192, 256};
  static const TcCosts costs[3] = {
      {{0.227, 0.242, 0.228, 0.286, 0.303, 0.320}, {0.393, 0.399, 0.484, 0.602, 0.0, 0.0}, {0.0, 0.274, 0.0, 0.244, 0.303, 0.320},
       4.37, 5.86, 5.15, 4.86, 2.67, 1.41, 1.4, 7.04, 4.86, 5.71},
      {{0.227, 0.242, 0.264, 0.286, 0.303, 0.320}, {0.393, 0.429, 0.484, 0.538, 0.0, 0.0}, {0.0, 0.0, 0.0, 0.0, 0.303, 0.320},
       3.34, 3.36, 3.36, 2.52, 2.52, 1.6, 1.4, 5.1, 4.8, 7.8},
      {{0.1957, 0.2, 0.2147, 0.2147, 0.2829, 0.3241}, {0.4481, 0.4481, 0.4997, 0.526, 0.0, 0.0}, {0.0, 0.0, 0.0, 0.0, 0.2829, 0.3241},
       2.11, 4.07, 3.08, 1.87, 2.33, 0.13, 0.78, 3.82, 0.0, 9.61}};
  static const int below[6] = {0, 32, 64, 64, 128, 128};   // alone: tiles that some smaller one with the same splits leaves without use
  const TcCosts& t = costs[call];
  const int slabs = (N + TC_BM - 1) / TC_BM, KT = K / TILE_K;
  double best = 1e30;
  TcPlan plan{32, 1, 2};
  for (int ri = 0; ri < 6; ++ri) {
    const int R = sizes[ri], max_split = R == 96 || R == 192 ? 1 : 8;
    if (ri > 0 && M <= (call == TC_ALONE ? below[ri] : sizes[ri - 1])) break;
    for (int S = 1; S <= max_split; S *= 2) {
      if (S > 1 && KT / S < 4) break;
      // (not counted with so few rows that the weights bound: 14336 x 2048, 32 rows 13.5 us in eight, 14.6 in four)
      const int sms = S < 8 || (call == TC_ALONE && M > 32) ? tc_resident(S, sm_count) : sm_count;
      const long long ctas = (long long)slabs * ((M + R - 1) / R) * S, per_wave = (long long)sms * (R > 128 ? 1 : 2);
      const long long full = ctas / per_wave, rest = ctas % per_wave;
      const bool four = tc_four_groups(call, R, S, ctas, sm_count);
      const double steps = (KT + S - 1) / S, f = R / 256.0, one = four ? t.step4[ri] : t.step1[ri];
      const double full_t = R > 128 ? one : t.step2[ri], rest_t = rest == 0 ? 0.0 : (rest > sms ? t.step2[ri] : one);
      const double more = (double)full + (rest > 0 ? 1 : 0) - 1.0;
      const double cost = steps * (full * full_t + rest_t) + t.fixed + (four ? t.tail4 : t.tail) * f + (S > 1 ? (four ? t.exchange4 : t.exchange) * f : 0.0) +
                          (S == 8 ? t.eight : 0.0) + more * (S == 1 ? t.wave1 + t.wave1_f * f : t.wave + t.wave_f * f);
      if (cost < best) { best = cost; plan = TcPlan{R, S, four ? 4 : 2}; }
    }
  }
  return plan;
}

// `status` may be nullptr
cudaError_t launch_gemm_tc(const GemmArgs& args, int sm_count, int* status, cudaStream_t st) {
  GemmArgs a = args;
  const unsigned T = (unsigned)(a.epi == EPI_QKV ? a.rows_per_stream : (a.lora.adapter_idx != nullptr ? a.lora.rows_per_stream : 1));
  a.stream_magic = T > 1 ? 0xffffffffu / T + 1u : 0u;      // exact for m, T below 65536
  const TcPlan plan = tc_plan(a.M, a.K, a.N, a.lora.adapter_idx != nullptr ? TC_LORA : (TcCall)a.call, sm_count);
#define TC_CASE(NR, S, GRP) \
  if (plan.rows == NR && plan.split == S && plan.groups == GRP) \
    return a.epi == EPI_F32 ? tc_launch<NR, S, EPI_F32, GRP>(a, sm_count, status, st) : a.epi == EPI_RESID ? tc_launch<NR, S, EPI_RESID, GRP>(a, sm_count, status, st) \
         : a.epi == EPI_SWIGLU ? tc_launch<NR, S, EPI_SWIGLU, GRP>(a, sm_count, status, st) : tc_launch<NR, S, EPI_QKV, GRP>(a, sm_count, status, st);
  TC_FOR_EACH(TC_CASE)
#undef TC_CASE
  return cudaErrorInvalidValue;
}

}  // namespace mlora
