// Squeeze GEMM on the 5th-generation tensor cores (sm_103a): the O(Dcut^15) contraction of
// arXiv:1906.06060 Sec. 2 (cost statement), written as C[m][n] = sum_k A[m][k] Bt[n][k].
//
// Precision: each FP32 operand is split into bf16 planes, x = hi + lo (2 planes) or
// x = hi + mid + lo (3 planes), each plane the bf16 rounding of what the previous ones left.
// The GEMM sums plane products ("passes"): with two planes hi*hi + hi*lo + lo*hi (3 passes) or
// all four products (4 passes, adds lo*lo), with three planes hh, hm, mh, hl, mm, lh (6
// passes), accumulating in FP32 in tensor memory. Per product the dropped terms and split
// residuals are O(2^-16) relative for 3 passes, O(2^-17) unbiased for 4 and O(2^-24) for 6. The
// dropped lo*lo of 3 passes is systematic when A and B are built from the same tensor.
// fp16 planes (two of them, 3 or 4 passes): each operand is scaled by an exact power of two 2^e
// that brings its largest entry just below 2^15, then split into fp16 hi + lo (11 significant
// bits each, O(2^-22) per product); the epilogue multiplies by 2^-(eA + eB). Same MMA cost as
// bf16 (kind::f16 takes either type; A and B always share one).
//
// Batched launches: a persistent launch can cover several independent products of one shape (a
// group of instances of a temperature scan): the tile list runs over the instances one after the
// other, the operand planes are 3D tensor maps whose third coordinate is the instance, and each
// instance has its own output, block descriptor and fp16 scale bounds.
//
// Accumulation: the tensor core's FP32 accumulate rounds toward zero, so a long chain of MMAs
// into one TMEM accumulator drifts systematically towards zero by about (chain length) x 2^-25
// relative - for K = 10^4 and 3 passes about 1e-4, far above what the free energy tolerates.
// The accumulator is therefore restarted for every 64-wide k-block (chain: npass x 4 MMAs, the
// small cross terms first so the large hi*hi products meet a small accumulator) and each
// k-block's partial sum is folded into an FP32 register accumulator with round-to-nearest adds.
//
// Kernel structure (one CTA per SM, persistent over output tiles, 384 threads):
//   warp 0      TMA producer: per k-block loads every 16-bit plane of the 128 x BK A tile and
//               of the 256 x BK B tile (BK*2-byte swizzle) into one stage of a shared-memory
//               ring, so the passes of a k-block reuse the same stage (BK = 64 or 32).
//   warp 1      MMA issuer: one thread issues tcgen05.mma.cta_group::1.kind::f16 (M=128,
//               N=256, K=16) for all passes of one k-block into one of two TMEM buffers (2 x 256
//               FP32 columns), releases the stage and hands the buffer over with tcgen05.commit.
//   warps 4-11  fold/epilogue: warp w reads TMEM lanes 32*(w%4).. (its hardware quadrant),
//               columns 128*((w-4)/4).. of the buffer, adds them into 128 FP32 registers per
//               thread and frees the buffer; after the last k-block it stores its 128 columns.
//
// CTA pairs (CG = 2, a thread-block cluster of two CTAs on two SMs, one 256 x 256 output tile):
// each CTA stages its own 128 A rows and half (128) of the tile's B rows per k-block, so a stage
// is 64 KB instead of 96 KB at BK = 64 (three stages fit instead of two) and each SM moves 2/3 of
// the shared-memory operand bytes per MMA flop. The first CTA's thread issues
// tcgen05.mma.cta_group::2 (M = 256): the tensor cores of both SMs read A from their own CTA and B
// from both, and each CTA's TMEM receives its 128 rows. The first CTA's producer issues the TMA
// copies of both CTAs (the second CTA's land in its shared memory through mapa addresses) and all
// bytes count on the first CTA's stage barriers, so stage hand-over never crosses SMs; the MMA
// commits free the stage there and reach the TMEM-full barriers of both CTAs (multicast); the
// fold warps of both report freed TMEM buffers to the first CTA. Measured reasons: a single CTA's
// 128 x 256 MMA chain, with operands resident and nothing else running, kept the tensor pipe busy
// about 2/3 of the time (pairs: about 3/4); and a pair whose second CTA issued its own copies,
// counted remotely on the first CTA's barrier, lost a quarter of its rate to the cross-SM hand-over (again with the
// stage freed in both CTAs by a multicast commit: 906 -> 1166 ms of GEMM in a steady step at bond dimension 10).
// Every mbarrier wait is bounded by a timeout; on expiry the CTA records ST_TIMEOUT, drains
// the copies and MMAs it issued (waits bounded by max(timeout, 1 s): issued work always
// completes, so a short caller limit never lets the CTA exit before it), frees TMEM and returns.
#include <cuda.h>

#include <algorithm>
#include <atomic>
#include <cstring>

#include "tc_ptx.cuh"

namespace hotrg {

namespace {

// k-block width BK (16-bit elements per tile row): 64 -> 128-byte swizzle, 32 -> 64-byte
// swizzle. A stage holds every plane of one k-block of the CTA's A rows (128) and B rows (256, or
// 128 for a CTA pair); as many stages as fit 216 KB, at most 6. The accumulator is folded once per
// k-block (or fold group).
template <int BK, int NPL, int CG>
struct Cfg {
  static constexpr uint32_t A_TILE = TC_BM * BK * 2;
  static constexpr uint32_t B_TILE = (TC_BN / CG) * BK * 2;
  static constexpr uint32_t STAGE_BYTES = NPL * (A_TILE + B_TILE);
  static constexpr int STAGES = (int)((216u * 1024u) / STAGE_BYTES) > 6 ? 6 : (int)((216u * 1024u) / STAGE_BYTES);
  // ring, barriers, and STORE_COLS columns of 32 rows (padded by one) per fold warp for ragged stores; the tile prefix is
  // static shared memory
  static constexpr size_t BASE = 1024 + STAGES * STAGE_BYTES + 256;
  static constexpr size_t LEFT = 227 * 1024 - sizeof(int) * (kMaxGemmBatch + 4) - BASE;
  static constexpr int STORE_COLS = LEFT >= (TC_FOLD_THREADS / 32) * 32 * 9 * sizeof(float) ? 8 : 4;
  static constexpr size_t SMEM = BASE + (TC_FOLD_THREADS / 32) * 32 * (STORE_COLS + 1) * sizeof(float);
  static_assert(SMEM - BASE <= LEFT, "a CTA's shared memory");
};

struct TmapSet {
  CUtensorMap a[3];
  CUtensorMap b[3];
};

// plane index of A and B for each pass, smallest products first, hi*hi last
//   npass 1: hh    npass 3: hl, lh, hh    npass 4: ll, hl, lh, hh (two planes, all products)
//   npass 6: lh, mm, hl, mh, hm, hh (three planes h=0, m=1, l=2)
__host__ __device__ constexpr int pass_plane_a(int npass, int ps) {
  return npass == 1 ? 0
       : npass == 3 ? (ps == 1 ? 1 : 0)
       : npass == 4 ? ((ps == 0 || ps == 2) ? 1 : 0)
       : (ps == 0 ? 2 : (ps == 1 || ps == 3) ? 1 : 0);
}
__host__ __device__ constexpr int pass_plane_b(int npass, int ps) {
  return npass == 1 ? 0
       : npass == 3 ? (ps == 0 ? 1 : 0)
       : npass == 4 ? ((ps == 0 || ps == 1) ? 1 : 0)
       : (ps == 2 ? 2 : (ps == 1 || ps == 4) ? 1 : 0);
}
static_assert(pass_plane_a(6, 0) == 2 && pass_plane_b(6, 0) == 0, "lh first");
static_assert(pass_plane_a(6, 5) == 0 && pass_plane_b(6, 5) == 0, "hh last");
static_assert(pass_plane_a(3, 2) == 0 && pass_plane_b(3, 2) == 0, "hh last");
static_assert(pass_plane_a(4, 0) == 1 && pass_plane_b(4, 0) == 1, "ll first");

struct TcParams {
  long long M, N, K;
  int num_m, num_n, num_kb, npass;
  int group_m;     // output tiles are rastered in groups of group_m M-tiles (L2 reuse of A and B)
  float* C;
  long long ldc;
  int* status;
  unsigned long long timeout_ns;
  int vec8;  // rows of C start on 32-byte boundaries
  const GemmBlocks* blk;  // null: one dense product over M x N x K
  uint32_t idesc;         // idesc_for(fp16 operands, CTA group)
  // fp16 operands carry power-of-two scales 2^eA, 2^eB (see Planes): the epilogue multiplies by
  // 2^-(eA + eB). Null amax: no scaling.
  const unsigned* amaxA;
  const unsigned* amaxB;
  float multA, multB;
  // batched launch: `batch` independent products of the same shape; instance i reads the operand
  // planes at z = i (A) and i / b_div (B) of the 3D tensor maps, writes C + i c_inst, takes the descriptor blk[i]
  // and the scale bounds amaxA[i], amaxB[i / b_div]
  int batch;
  long long c_inst;
  int b_div;  // B operand and B scale bound of instance i: i / b_div
  // wait probe: the producer issues no copies, so the first wait for a stage can never be satisfied
  // and must run out (nothing is in flight to drain)
  int stall;
};

template <int BK, int NPL, int NPASS, int FG, int CG>
__global__ void __launch_bounds__(TC_THREADS, 1)
    k_gemm_split(const __grid_constant__ TmapSet maps, TcParams p) {
  using C = Cfg<BK, NPL, CG>;
  static_assert(FG == 1 || FG <= C::STAGES - 1, "a fold group leaves one stage to the producer");
  static_assert(CG == 1 || CG == 2, "one CTA or a CTA pair");
  constexpr int TC_STAGES = C::STAGES;
  constexpr uint32_t A_TILE = C::A_TILE, B_TILE = C::B_TILE, STAGE_BYTES = C::STAGE_BYTES;
  constexpr int TC_BK = BK;
  constexpr int B_ROWS = TC_BN / CG;  // B rows this CTA stages per k-block
  static_assert(TC_STAGES >= 2, "ring needs two stages");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  // stage s: A planes 0..NPL-1 then B planes 0..NPL-1
  auto a_tile = [&](int stage, int pl) { return smem + stage * STAGE_BYTES + pl * A_TILE; };
  auto b_tile = [&](int stage, int pl) { return smem + stage * STAGE_BYTES + NPL * A_TILE + pl * B_TILE; };
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + TC_STAGES * STAGE_BYTES);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * TC_STAGES + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const uint32_t full0 = smem_u32(bars);
  const uint32_t empty0 = full0 + 8 * TC_STAGES;
  const uint32_t tfull0 = empty0 + 8 * TC_STAGES;
  const uint32_t tempty0 = tfull0 + 16;
  const uint32_t final_bar = tempty0 + 16;
  // CTA pair: rank 0 issues the MMAs and owns the stage-full and TMEM-empty barriers both CTAs
  // signal; every CTA walks the same tiles (one per cluster)
  const uint32_t rank = CG == 2 ? cluster_rank() : 0u;
  const bool leader = rank == 0;
  const int cta0 = (int)blockIdx.x / CG, ncta = (int)gridDim.x / CG;

  __shared__ int s_prefix[kMaxGemmBatch + 1];
  __shared__ int s_total;
  if (p.blk) {
    // tiles of every instance (block-sparse: the descriptors differ per instance), then their first tiles below
    for (int i = threadIdx.x; i < p.batch; i += TC_THREADS) {
      Blk b[2];
      const int nb = load_blocks<BK, CG>(p, i, b);
      s_prefix[i] = b[0].tiles + (nb > 1 ? b[1].tiles : 0);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    Blk b[2];
    if (p.blk) {
      int t = 0;
      for (int i = 0; i < p.batch; ++i) {
        const int n = s_prefix[i];
        s_prefix[i] = t;
        t += n;
      }
      s_prefix[p.batch] = t;
      s_total = t;
    } else {
      load_blocks<BK, CG>(p, 0, b);
      s_total = b[0].tiles * p.batch;
    }
    for (int s = 0; s < TC_STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(tfull0 + 8 * b, 1);
      mbar_init(tempty0 + 8 * b, CG * TC_FOLD_THREADS / 32);
    }
    mbar_init(final_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0 && lane < 2 * NPL) {
    const CUtensorMap* m = lane < NPL ? &maps.a[lane] : &maps.b[lane - NPL];
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
  }
  if (warp == 1) {
    if constexpr (CG == 1) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                   "r"(TMEM_COLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    } else {
      // one warp of each CTA of the pair allocates collectively: the same columns in both
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                   "r"(TMEM_COLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
  }
  tc_fence_before();
  if constexpr (CG == 1) __syncthreads();
  else cluster_sync();  // the peer's copies and arrivals target barriers initialised above
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  const int total = s_total;

  if (warp < TC_FOLD_WARP0) {
  regs_give<TC_ROLE_REGS>();
  if (warp == 0) {
    if (lane == 0 && leader) {
      int stage = 0;
      uint32_t phase = 0;
      long long issued = 0;  // stages this thread filled
      bool ok = !p.stall;
      for (int tile = cta0; tile < total && ok; tile += ncta) {
        int inst, mt, nt;
        Blk bk;
        locate<BK, CG>(p, s_prefix, tile, inst, bk, mt, nt);
        const int arow = bk.m0 + mt * TC_BM * CG + (int)rank * TC_BM;
        const int brow = bk.n0 + nt * TC_BN + (int)rank * B_ROWS;
        const int binst = inst / p.b_div;
        for (int kb = 0; kb < bk.num_kb; ++kb) {
          if (!mbar_wait(empty0 + 8 * stage, phase ^ 1, abort_flag, p.timeout_ns)) { ok = false; break; }
          const uint32_t fb = full0 + 8 * stage;
          const int kx = bk.k0 + kb * TC_BK;
          if constexpr (CG == 1) {
            mbar_expect_tx(fb, STAGE_BYTES);
#pragma unroll
            for (int pl = 0; pl < NPL; ++pl) {
              tma_load_3d(smem_u32(a_tile(stage, pl)), &maps.a[pl], fb, kx, arow, inst);
              tma_load_3d(smem_u32(b_tile(stage, pl)), &maps.b[pl], fb, kx, brow, binst);
            }
          } else {
            // this CTA fills the stage in both CTAs of the pair (the second CTA's copies land at the
            // same offsets of its shared memory); all bytes count on this CTA's barrier
            mbar_expect_tx(fb, 2 * STAGE_BYTES);
#pragma unroll
            for (int pl = 0; pl < NPL; ++pl) {
              const uint32_t sa = smem_u32(a_tile(stage, pl)), sb = smem_u32(b_tile(stage, pl));
              tma_load_3d_pair(sa, &maps.a[pl], fb, kx, arow, inst);
              tma_load_3d_pair(sb, &maps.b[pl], fb, kx, brow, binst);
              tma_load_3d_pair(mapa_rank(sa, 1), &maps.a[pl], fb, kx, arow + TC_BM, inst);
              tma_load_3d_pair(mapa_rank(sb, 1), &maps.b[pl], fb, kx, brow + B_ROWS, binst);
            }
          }
          ++issued;
          if (++stage == TC_STAGES) { stage = 0; phase ^= 1; }
        }
      }
      // Drain, on every exit path: the last min(STAGES, issued) loads must land before the CTA (or
      // either CTA of a pair: the second waits at the final cluster barrier) exits - a consumer that
      // gave up may never have waited for them. Each stage holds at most one load in flight, and
      // issued copies always complete, so these waits use a floor of one second whatever the
      // caller's limit (after a normal run they return at once).
      for (long long i = (issued > TC_STAGES ? issued - TC_STAGES : 0); i < issued; ++i)
        mbar_wait(full0 + 8 * (int)(i % TC_STAGES), (uint32_t)((i / TC_STAGES) & 1), abort_flag,
                  drain_ns(p.timeout_ns), false);
    }
  } else if (warp == 1) {
    if (lane == 0 && leader) {
      int stage = 0;
      uint32_t phase = 0;
      int buf = 0;
      uint32_t bphase = 0;
      bool ok = true;
      for (int tile = cta0; tile < total && ok; tile += ncta) {
        int inst_, mt_, nt_;
        Blk bk_;
        locate<BK, CG>(p, s_prefix, tile, inst_, bk_, mt_, nt_);
        const int num_kb = bk_.num_kb;
        // Descriptors differ only in their start-address field (bits 0-13, address >> 4), so each
        // one is a base descriptor plus the tile's byte offset >> 4 (all offsets are multiples of
        // 16 bytes and the shared window is < 256 KB, so the field never carries over). Passes,
        // planes and the fold group are compile-time: a group's MMAs unroll into straight-line
        // issue code with constant offsets. A pair's MMA reads the same offsets in both CTAs.
        const uint64_t desc_base = smem_desc<BK>(smem_u32(smem));
        const uint32_t idesc = p.idesc;
        constexpr uint32_t B_OFF = NPL * A_TILE;
        for (int kb0 = 0; kb0 < num_kb && ok; kb0 += FG) {
          const int g = min(FG, num_kb - kb0);  // k-blocks in this fold group
          if (!mbar_wait(tempty0 + 8 * buf, bphase ^ 1, abort_flag, p.timeout_ns)) { ok = false; break; }
          uint32_t so[FG];  // byte offsets of the group's stages
          {
            int st = stage;
            uint32_t ph = phase;
#pragma unroll
            for (int i = 0; i < FG; ++i) {
              so[i] = (uint32_t)st * STAGE_BYTES;
              if (i < g && ok && !mbar_wait(full0 + 8 * st, ph, abort_flag, p.timeout_ns)) ok = false;
              if (++st == TC_STAGES) { st = 0; ph ^= 1; }
            }
          }
          if (!ok) break;
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + (uint32_t)(buf * TC_BN);
#pragma unroll
          for (int ps = 0; ps < NPASS; ++ps) {
#pragma unroll
            for (int i = 0; i < FG; ++i) {
              if (i < g) {
                const uint64_t da = desc_base + ((so[i] + (uint32_t)pass_plane_a(NPASS, ps) * A_TILE) >> 4);
                const uint64_t db = desc_base + ((so[i] + B_OFF + (uint32_t)pass_plane_b(NPASS, ps) * B_TILE) >> 4);
#pragma unroll
                for (int k = 0; k < TC_BK / 16; ++k)
                  mma_f16<CG>(d_tmem, da + (uint64_t)(k * 2), db + (uint64_t)(k * 2), idesc,
                              (ps == 0 && i == 0 && k == 0) ? 0u : 1u);
              }
            }
          }
          for (int i = 0; i < g; ++i) {
            mma_commit_local<CG>(empty0 + 8 * stage);  // frees the stage (its copies are issued here)
            if (++stage == TC_STAGES) { stage = 0; phase ^= 1; }
          }
          mma_commit<CG>(tfull0 + 8 * buf);
          if (++buf == 2) { buf = 0; bphase ^= 1; }
        }
      }
      // all MMAs issued by this thread complete before TMEM is released (issued MMAs always
      // complete: the wait has the drain's floor, not the caller's limit)
      mma_commit_local<CG>(final_bar);
      mbar_wait(final_bar, 0, abort_flag, drain_ns(p.timeout_ns), false);
    }
  }
  } else {
    regs_take<TC_FOLD_REGS>();
    const int q = warp & 3;          // TMEM lane quadrant this warp may access
    const int half = (warp - TC_FOLD_WARP0) >> 2;  // which 128 of the 256 columns
    // where this warp reports a freed TMEM buffer: the MMA-issuing CTA's barriers (contiguous in
    // its shared memory, so buffer b's barrier is 8 b bytes further in either address window)
    const uint32_t tempty_dst = CG == 2 && !leader ? mapa_rank(tempty0, 0) : tempty0;
    int buf = 0;
    uint32_t bphase = 0;
    bool ok = true;
    for (int tile = cta0; tile < total && ok; tile += ncta) {
      int num_kb;
      {
        // only the k-block count stays live through the k loop (the accumulator holds 128
        // registers); the tile is located again for the store
        int inst, mt, nt;
        Blk bk;
        locate<BK, CG>(p, s_prefix, tile, inst, bk, mt, nt);
        num_kb = bk.num_kb;
      }
      float acc[128];
#pragma unroll
      for (int j = 0; j < 128; ++j) acc[j] = 0.f;
      for (int kb = 0; kb < num_kb; kb += FG) {
        // one lane waits for the fold group's MMAs, the warp follows it
        int w = 1;
        if (lane == 0) w = mbar_wait(tfull0 + 8 * buf, bphase, abort_flag, p.timeout_ns) ? 1 : 0;
        w = __shfl_sync(0xffffffffu, w, 0);
        if (!w) { ok = false; break; }
        tc_fence_after();
        const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * TC_BN + half * 128);
#pragma unroll
        for (int c = 0; c < 4; c += 2) {
          uint32_t r0[32], r1[32];
          tmem_ld32(taddr + c * 32, r0);
          tmem_ld32(taddr + (c + 1) * 32, r1);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            acc[c * 32 + j] += __uint_as_float(r0[j]);
            acc[(c + 1) * 32 + j] += __uint_as_float(r1[j]);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {  // one arrive per warp
          const uint32_t bar = tempty_dst + 8 * buf;
          if constexpr (CG == 1) mbar_arrive(bar);
          else if (leader) mbar_arrive(bar);
          else mbar_arrive_remote(bar);
        }
        if (++buf == 2) { buf = 0; bphase ^= 1; }
      }
      if (!ok) break;
      int inst, mt, nt;
      Blk bk;
      locate<BK, CG>(p, s_prefix, tile, inst, bk, mt, nt);
      if (p.amaxA) {
        // undo the operands' power-of-two scales (exact): the exponents the operand builders used
        const float unscale =
            pow2f(-(f16_scale_exponent(plane_bound(p.amaxA + inst, p.multA)) +
                    f16_scale_exponent(plane_bound(p.amaxB + inst / p.b_div, p.multB))));
#pragma unroll
        for (int j = 0; j < 128; ++j) acc[j] *= unscale;
      }
      const long long row = (long long)bk.m0 + (long long)mt * TC_BM * CG + (long long)rank * TC_BM + q * 32 + lane;
      const long long col0 = (long long)bk.n0 + (long long)nt * TC_BN + half * 128;
      const long long row_end = (long long)bk.m0 + bk.mc, col_end = (long long)bk.n0 + bk.nc;
      float* const cbase = p.C + (long long)inst * p.c_inst;
      // Whole rows of 128 columns at 32-byte aligned addresses: each thread stores its row, 32 bytes a time (whole
      // sectors). Otherwise (ragged columns, an odd row stride, a block that starts off the boundary) the warp passes a few
      // columns at a time through shared memory and stores 32 bytes of four rows at once: one thread per row would store
      // single floats, 32 sectors an instruction (2401 x 16807 x 2401, FP16X3: 632 us).
      if (p.vec8 && (bk.n0 & 7) == 0 && col0 + 128 <= col_end) {
        if (row < row_end) {
          float* dst = cbase + row * p.ldc + col0;
#pragma unroll
          for (int j = 0; j < 128; j += 8)
            asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst + j), "f"(acc[j]),
                         "f"(acc[j + 1]), "f"(acc[j + 2]), "f"(acc[j + 3]), "f"(acc[j + 4]), "f"(acc[j + 5]),
                         "f"(acc[j + 6]), "f"(acc[j + 7])
                         : "memory");
        }
      } else if (row - lane < row_end && col0 < col_end) {
        const int nrow = (int)min(32LL, row_end - (row - lane));
        constexpr int SC = C::STORE_COLS;  // columns at a time; rows padded by one (no bank conflicts)
        float* const stg = reinterpret_cast<float*>(smem + TC_STAGES * STAGE_BYTES + 256) + (warp - TC_FOLD_WARP0) * (32 * (SC + 1));
        float* const put = stg + lane * (SC + 1);
        const float* const get = stg + lane / SC * (SC + 1) + lane % SC;
        float* dst = cbase + (row - lane + lane / SC) * p.ldc + col0 + lane % SC;
        const int left = (int)min(128LL, col_end - col0) - lane % SC;
#pragma unroll
        for (int c = 0; c < 128; c += SC) {
          __syncwarp();
#pragma unroll
          for (int u = 0; u < SC; ++u) put[u] = acc[c + u];
          __syncwarp();
          if (c < left) {
            float* d = dst + c;
#pragma unroll 2
            for (int r = 0; r < 32; r += 32 / SC, d += 32 / SC * p.ldc)
              if (r + lane / SC < nrow) *d = get[r * (SC + 1)];
          }
        }
      }
    }
  }
  if constexpr (CG == 1) {
    __syncthreads();
    if (threadIdx.x == 0 && *abort_flag) atomic_status(p.status, ST_TIMEOUT);
    if (warp == 1) {
      tc_fence_after();
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS)
                   : "memory");
    }
  } else {
    __syncwarp();
    // every role of both CTAs is done: the pair's copies have landed (the first CTA's drain) and its
    // MMAs have completed, so neither CTA's shared or tensor memory is still in use
    cluster_sync();
    if (threadIdx.x == 0 && *abort_flag) atomic_status(p.status, ST_TIMEOUT);
    if (warp == 1) {
      tc_fence_after();
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS)
                   : "memory");
    }
  }
}

// Split planes of rows x cols floats: a block takes rows in turn, a thread two adjacent columns at a time (two 4-byte
// loads, whatever the rows' alignment; a 4-byte store per plane). Bound by its traffic: 4 bytes in, 2 per plane out (one
// element per thread with a 64-bit division each: 140 us at 16807 x 2401, two planes, for 47 us of traffic).
__global__ void __launch_bounds__(256) k_split_rows(const float* __restrict__ X, long long ldx, int rows, int cols,
                                                    Planes<__nv_bfloat16> out, long long ld) {
  const float sc = plane_scale(out);
  for (int r = blockIdx.x; r < rows; r += gridDim.x) {
    const float* x = X + (long long)r * ldx;
    const long long o = (long long)r * ld;
#pragma unroll 4
    for (int c = 2 * threadIdx.x; c < cols; c += 512) {
      __nv_bfloat16 q0[3], q1[3];
      split_planes(out, x[c], sc, q0);
      split_planes(out, c + 1 < cols ? x[c + 1] : 0.f, sc, q1);  // (rows of the planes are padded to 64 columns)
#pragma unroll
      for (int k = 0; k < 3; ++k)
        if (k < out.nparts) {
          __nv_bfloat162 q;
          q.x = q0[k];
          q.y = q1[k];
          *reinterpret_cast<__nv_bfloat162*>(out.p[k] + o + c) = q;
        }
    }
  }
}

// ------------------------------------------------------------------ host: tensor maps
// 3D map of `batch` planes of rows x cols (row stride ld, instance stride inst elements), boxes of
// box_rows x bk x 1.
bool make_map(CUtensorMap* m, const __nv_bfloat16* ptr, long long rows, long long cols, long long ld, int batch,
              long long inst, int box_rows, int bk, bool f16) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return false;
  cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)batch};
  cuuint64_t strides[2] = {(cuuint64_t)ld * 2, (cuuint64_t)inst * 2};
  cuuint32_t box[3] = {(cuuint32_t)bk, (cuuint32_t)box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return enc(m, f16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3,
             const_cast<__nv_bfloat16*>(ptr), dims, strides, box,
             estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             bk == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Encodes the tensor maps and launches one kernel variant. The maps' box sizes, the stage slot
// sizes and the expected transaction bytes all derive from the same compile-time BK, NPL and CG,
// so a TMA copy can never be larger than the stage slot it lands in. Persistent launch: as many
// CTAs (CG = 2: clusters of two) as can be resident at once, one per SM, and no more than the
// tiles (tiles < 0: counted on the device).
template <int BK, int NPL, int NPASS, int FG, int CG>
int launch_variant(long long tiles, const Planes<__nv_bfloat16>& A, long long lda, const Planes<__nv_bfloat16>& B,
                   long long ldb, long long a_inst, long long b_inst, const TcParams& p, cudaStream_t s) {
  using Cf = Cfg<BK, NPL, CG>;
  static_assert(Cf::STAGE_BYTES == NPL * (TC_BM + TC_BN / CG) * BK * 2, "stage holds exactly the boxes");
  TmapSet maps;
  std::memset(&maps, 0, sizeof(maps));
  for (int i = 0; i < NPL; ++i)
    if (!make_map(&maps.a[i], A.p[i], p.M, p.K, lda, p.batch, a_inst, TC_BM, BK, A.fmt == 1) ||
        !make_map(&maps.b[i], B.p[i], p.N, p.K, ldb, p.batch / p.b_div, b_inst, TC_BN / CG, BK, B.fmt == 1))
      return HOTRG_EDEVICE;
  auto kern = k_gemm_split<BK, NPL, NPASS, FG, CG>;
  // the dynamic shared-memory limit is a per-device attribute of the kernel: set it once on each
  // device this variant launches on; so is the number of resident CTAs or clusters
  static std::atomic<int> resident[kMaxDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return HOTRG_EDEVICE;
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CG;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.blockDim = dim3(TC_THREADS);
  cfg.dynamicSmemBytes = Cf::SMEM;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = CG > 1 ? 1 : 0;
  int n = resident[dev].load();
  if (n <= 0) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cf::SMEM) != cudaSuccess)
      return HOTRG_EDEVICE;
    if (CG == 1) {
      n = num_sms();
    } else {
      cfg.gridDim = dim3((unsigned)(CG * std::max(1, num_sms() / CG)));
      if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n <= 0) {
        cudaGetLastError();
        return HOTRG_EDEVICE;
      }
    }
    // the register shares need what they were planned with
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, kern) != cudaSuccess || fa.numRegs < TC_LAUNCH_REGS) return HOTRG_EDEVICE;
    resident[dev].store(n);
  }
  const long long units = tiles >= 0 && tiles < n ? (tiles > 0 ? tiles : 1) : n;
  cfg.gridDim = dim3((unsigned)(units * CG));
  if (cudaLaunchKernelEx(&cfg, kern, maps, p) != cudaSuccess) {
    cudaGetLastError();
    return HOTRG_EDEVICE;
  }
  return HOTRG_OK;
}

}  // namespace

int launch_gemm_split(const Planes<__nv_bfloat16>& A, long long lda, const Planes<__nv_bfloat16>& B,
                      long long ldb, float* C, long long ldc, long long M, long long N, long long K,
                      int npass, int* status, double timeout_s, cudaStream_t s, int bk, int group_m,
                      int fold_group, const GemmBlocks* blk, const GemmBatch* bat, bool stall, int cta_group) {
  if (bk != 32 && bk != 64) return HOTRG_EINVAL;
  if (cta_group == 0) cta_group = M > TC_BM ? 2 : 1;
  if (cta_group != 1 && cta_group != 2) return HOTRG_EINVAL;
  if (group_m < 1 || group_m > 64 || fold_group < 1) return HOTRG_EINVAL;
  if (M < TC_BM || N < TC_BN || K < 64 || (npass != 1 && npass != 3 && npass != 4 && npass != 6))
    return HOTRG_EINVAL;
  const int nplanes = npass == 1 ? 1 : (npass == 6 ? 3 : 2);
  if (nplanes == 3) bk = 32;  // three 64-wide planes do not fit two ring stages: resolved first
  if (nplanes == 1) bk = 64;  // single-plane GEMMs use 64-wide stages
  if (A.nparts < nplanes || B.nparts < nplanes) return HOTRG_EINVAL;
  // fp16 planes: both operands (one MMA type), two planes at most, each with its scale bound
  if (A.fmt != B.fmt || A.fmt < 0 || A.fmt > 1) return HOTRG_EINVAL;
  if (A.fmt == 1 && (nplanes > 2 || !A.amax || !B.amax)) return HOTRG_EINVAL;
  if ((lda % 8) || (ldb % 8) || lda < K || ldb < K || ldc < N) return HOTRG_EINVAL;
  if (M > 0x7fffffffLL || N > 0x7fffffffLL || K > 0x7fffffffLL) return HOTRG_EINVAL;
  auto al16 = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15) == 0; };
  for (int i = 0; i < nplanes; ++i)
    if (!al16(A.p[i]) || !al16(B.p[i])) return HOTRG_EINVAL;
  // batched launch: instances' planes apart by at least a whole plane, 16-byte aligned
  const int batch = bat ? bat->batch : 1;
  const long long a_inst = bat ? bat->a_inst : M * lda, b_inst = bat ? bat->b_inst : N * ldb;
  if (batch < 1 || batch > kMaxGemmBatch) return HOTRG_EINVAL;
  if (batch > 1 && (a_inst < M * lda || b_inst < N * ldb || (a_inst % 8) || (b_inst % 8) || bat->c_inst < M * ldc ||
                    bat->b_div < 1 || batch % bat->b_div))
    return HOTRG_EINVAL;
  TcParams p;
  p.M = M;
  p.N = N;
  p.K = K;
  p.num_m = (int)((M + TC_BM - 1) / TC_BM);
  p.num_n = (int)((N + TC_BN - 1) / TC_BN);
  p.num_kb = (int)((K + bk - 1) / bk);
  p.npass = npass;
  p.group_m = group_m;
  p.C = C;
  p.ldc = ldc;
  p.status = status;
  p.timeout_ns = (unsigned long long)(timeout_s * 1e9);
  p.vec8 = (ldc % 8) == 0 && (reinterpret_cast<uintptr_t>(C) & 31) == 0 && (!bat || bat->c_inst % 8 == 0);
  p.blk = blk;
  p.idesc = idesc_for(A.fmt == 1, cta_group);
  p.amaxA = A.fmt == 1 ? A.amax : nullptr;
  p.amaxB = A.fmt == 1 ? B.amax : nullptr;
  p.multA = A.amax_mult;
  p.multB = B.amax_mult;
  p.batch = batch;
  p.c_inst = bat ? bat->c_inst : 0;
  p.b_div = bat ? bat->b_div : 1;
  p.stall = stall ? 1 : 0;
  // output tiles: 128 x 256 per CTA, 256 x 256 per CTA pair
  const long long tiles = (long long)((M + (long long)TC_BM * cta_group - 1) / ((long long)TC_BM * cta_group)) *
                          p.num_n * batch;
  if (tiles > 0x7fffffffLL) return HOTRG_EINVAL;
  // supported variants (fold groups beyond a variant's maximum are clamped to it)
  const int fg = std::max(1, std::min(fold_group, max_fold_group(npass, bk)));
  // with device-side blocks the tile count is known only on the device
  const long long t = blk ? -1 : tiles;
  int rc = HOTRG_EINVAL;
#define HOTRG_GEMM_VARIANT(BK_, NPL_, NP_, FG_)                                                        \
  if (bk == BK_ && nplanes == NPL_ && npass == NP_ && fg == FG_)                                      \
    rc = cta_group == 2 ? launch_variant<BK_, NPL_, NP_, FG_, 2>(t, A, lda, B, ldb, a_inst, b_inst, p, s) \
                        : launch_variant<BK_, NPL_, NP_, FG_, 1>(t, A, lda, B, ldb, a_inst, b_inst, p, s);
  HOTRG_GEMM_VARIANT(64, 1, 1, 1)
  HOTRG_GEMM_VARIANT(64, 1, 1, 2)
  HOTRG_GEMM_VARIANT(64, 2, 3, 1)
  HOTRG_GEMM_VARIANT(64, 2, 4, 1)
  HOTRG_GEMM_VARIANT(32, 2, 3, 1)
  HOTRG_GEMM_VARIANT(32, 2, 3, 2)
  HOTRG_GEMM_VARIANT(32, 2, 4, 1)
  HOTRG_GEMM_VARIANT(32, 2, 4, 2)
  HOTRG_GEMM_VARIANT(32, 3, 6, 1)
  HOTRG_GEMM_VARIANT(32, 3, 6, 2)
#undef HOTRG_GEMM_VARIANT
  if (rc) return rc;
  count_launches(1);
  return HOTRG_OK;
}

int max_fold_group(int npass, int bk) {
  if (npass == 6) return 2;        // 32-wide stages, three planes, 3-stage ring
  if (npass == 1) return 2;        // 64-wide stages, one plane, 4-stage ring
  return bk == 64 ? 1 : 2;         // two planes: 2-stage ring at 64, 4-stage ring at 32
}

void launch_split_rows(const float* X, long long ldx, long long rows, long long cols,
                       const Planes<__nv_bfloat16>& out, long long ld, cudaStream_t s) {
  const int g = (int)std::min(rows, 152LL * 16);
  k_split_rows<<<g, 256, 0, s>>>(X, ldx, (int)rows, (int)cols, out, ld);
  count_launches(1);
}

}  // namespace hotrg
