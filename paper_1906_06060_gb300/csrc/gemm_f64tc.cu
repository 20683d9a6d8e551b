// FP64 squeeze products on the 5th-generation tensor cores: C[m][n] = sum_k A[m][k] Bt[n][k] in double precision
// from exact integer slices (the error-free splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012).
//
// GB300 has no fast FP64 unit (1.25 TFLOP/s nominal, 4 flop per clock and SM), its fp16 tensor cores run at
// 8192 flop per clock and SM. Column k of A is scaled by a power of two c(k), the size of the largest entry of Bt's
// column k, and column k of Bt by 1 / c(k): the product is the same. Then every row of an operand is scaled by a power of
// two 2^-e that brings its largest entry below 1 and rounded to a 63-bit fixed-point number, which is cut into 8 balanced
// digits of 8 bits,
//   x 2^-e = sum_i q_i 2^-(7 + 8 i),  -128 <= q_i <= 128,
// each stored as an fp16 integer (exact). The product is the sum over the digit pairs with i + j <= 7 (36 products),
// grouped by level s = i + j:
//   C[m][n] 2^-(eA + eB) = sum_s L_s 2^-(14 + 8 s),  L_s = sum_{i <= s} sum_k qA_i qB_{s-i}.
// Exactness: |qA qB| <= 2^14, so a chain of 16 x 64 products stays within 2^24 and the tensor cores' FP32 accumulator
// holds it exactly; every chain is added into an int32 register accumulator (|L_s| <= (s + 1) K 2^14 < 2^31 for
// K <= 16320). Levels 7 and 6 are folded into level 5 with a rounding shift each, and the six level sums are combined
// exactly and rounded once.
// Error of C[m][n]: one rounding of the result, and what the carries, the rows' last bits and the dropped digit pairs are
// worth, at most (2^-53 + K 2^-58) R and typically 2^-55 R with R = max_k |A[m][k] c(k)| max_k |Bt[n][k] / c(k)|. It is an
// error relative to R, where that of an FP64 sum (up to K 2^-53) is relative to sum_k |A[m][k] Bt[n][k]|. The two are of
// one size within a factor of K for rows that share their decay, and, by the column scales, where A's columns grow as
// Bt's decay (a tensor in an unbalanced gauge of its bonds); an output whose rows are large in different columns from
// those of their neighbours can be far below R and keeps fewer bits than an FP64 sum would give it. (Seven digits and 28
// products, 13 - 22 % faster, drop sqrt(6 K) 2^-57: at K = 4100 on rows that decay, further off than an FP64 product, so
// they are not taken.) Measured over random rows, flat and decaying, in the 2-norm:
// 5e-17 to 7e-17, one rounding, where FP64 products have 3e-16 to 1.1e-15. Rows holding NaN or infinity give NaN.
//
// Work: 36 tensor products of 2 M N K flops against one on the FP64 units at 1/2000 of the rate.
// Kernel structure, ring and bounded waits as k_gemm_split (gemm_tc.cu): warp 0 copies, warp 1 issues MMAs, warps
// 4-11 fold. Per output tile the levels run one after the other, least significant first, each over all k-blocks; a
// ring stage holds one digit tile of A and one of B. A finished level sum goes to a per-CTA scratch area in global
// memory (L2), one 16-byte access per thread and four columns, coalesced; the last level combines them in registers.
#include "tc_ptx.cuh"

namespace hotrg {

namespace {

constexpr int NSL = kSliceCount;      // digits per entry
constexpr int kSliceBits = 8 * NSL - 1;  // bits of the fixed-point rows
constexpr int CHAIN = 16;             // 64-wide k steps per accumulator chain
constexpr int SC_PLANES = 6;          // level sums parked in scratch: levels 5 (with 6), 4, 3, 2, 1, 0
constexpr int kExpNaN = 0x40000000;   // row exponent of a row with a non-finite entry
constexpr int SBK = 64;

template <int CG>
struct SCfg {
  static constexpr uint32_t A_TILE = TC_BM * SBK * 2;
  static constexpr uint32_t B_TILE = (TC_BN / CG) * SBK * 2;
  static constexpr uint32_t STAGE_BYTES = A_TILE + B_TILE;
  static constexpr int STAGES = CG == 2 ? 6 : 4;
  static constexpr size_t SMEM = 1024 + STAGES * STAGE_BYTES + 256;
};

struct SliceMaps {
  CUtensorMap a, b;
};

struct SliceParams {
  long long M, N, K;
  int num_kb, group_m, batch, b_div;  // Bt of product i: instance i / b_div
  double* C;
  long long ldc, c_inst;
  const int* ea;  // row exponents of A and of Bt, instance strides ea_inst, eb_inst
  const int* eb;
  long long ea_inst, eb_inst;
  int4* scratch;
  int* status;
  unsigned long long timeout_ns;
  const GemmBlocks* blk;
  uint32_t idesc;
  int accumulate;  // C += instead of C =
  int vec;         // entries per store: 4 (32-byte aligned rows) or 1
  int stall;       // wait probe: bit r: CTA r of the pair (or the CTA) issues no copies
};

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y, int z,
                                            int w) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], "
      "[%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y), "r"(z), "r"(w)
      : "memory");
}
// the same from either CTA of a pair: `dst` in its own shared memory, the bytes count on the first CTA's barrier `bar`
__device__ __forceinline__ void tma_load_4d_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y,
                                                 int z, int w) {
  asm volatile(
      "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, "
      "{%3, %4, %5, %6}], [%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y), "r"(z), "r"(w)
      : "memory");
}

// (hi 2^24 + lo) 2^e as a double, rounded once (to nearest, ties to even), in integer arithmetic: the FP64 unit's two
// operations a clock would make the tile's 32768 conversions and scalings cost more than its copies. |hi| < 2^45,
// |lo| < 2^47.
__device__ __forceinline__ double assemble(long long hi, long long lo, int e) {
  const bool wide = hi > (1LL << 38) || hi < -(1LL << 38);
  if (wide || e < -900 || e > 900)  // beyond 64 bits, or near the ends of the exponent range
    return ldexp(fma((double)hi, 16777216.0, (double)lo), e);
  const long long v = (hi << 24) + lo;  // |v| < 2^62 + 2^47
  const unsigned long long u = v < 0 ? 0ULL - (unsigned long long)v : (unsigned long long)v;
  const int lz = __clzll((long long)u);
  const unsigned long long m = u << (lz & 63);
  const unsigned long long kept = m >> 11;  // 53 bits, the leading one included: it adds 1 to the exponent field below
  const unsigned rest = (unsigned)m & 0x7FFu;
  const unsigned up = (rest + (unsigned)(kept & 1)) > 0x400u;
  const unsigned long long bits = ((unsigned long long)(unsigned)(1023 + 62 - lz + e) << 52) + kept + up;
  return __longlong_as_double((long long)(u ? bits | ((unsigned long long)v & 0x8000000000000000ULL) : 0ULL));
}

// Where a fold thread's 128 entries of a finished tile (its row, columns col0 ...) go.
struct TileOut {
  double* dst = nullptr;  // null: nothing to do
  const int* eb;
  int ea, ncol;  // ncol: columns of the 128 inside the block
  bool v4;
};

// Results of columns [j0, j0 + 4 JG) from the level sums in the scratch area (this thread's own stores). All loads are in
// flight together: the loop is bound by their latency.
template <int JG>
__device__ __forceinline__ void finish_columns(const SliceParams& p, const TileOut& o, const int4* park, int j0) {
  int4 l[JG][SC_PLANES];
#pragma unroll
  for (int g = 0; g < JG; ++g)
#pragma unroll
    for (int k = 0; k < SC_PLANES; ++k) l[g][k] = park[(k * 32 + j0 / 4 + g) * TC_FOLD_THREADS];
#pragma unroll
  for (int g = 0; g < JG; ++g) {
    const int j = j0 + 4 * g;
    auto value = [&](int u) -> double {
      if (j + u >= o.ncol) return 0.0;
      auto at = [&](int k) { return (long long)(u == 0 ? l[g][k].x : u == 1 ? l[g][k].y : u == 2 ? l[g][k].z : l[g][k].w); };
      const int ebj = o.eb[j + u];
      if (o.ea == kExpNaN || ebj == kExpNaN) return nan("");
      return assemble((at(5) << 16) + (at(4) << 8) + at(3), (at(2) << 16) + (at(1) << 8) + at(0), o.ea + ebj - 54);
    };
    double v[4] = {value(0), value(1), value(2), value(3)};
    if (o.v4) {
      if (p.accumulate) {
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] += o.dst[j + u];
      }
      asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(o.dst + j), "d"(v[0]), "d"(v[1]), "d"(v[2]), "d"(v[3])
                   : "memory");
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (j + u < o.ncol) o.dst[j + u] = p.accumulate ? o.dst[j + u] + v[u] : v[u];
    }
  }
}

template <int CG>
__global__ void __launch_bounds__(TC_THREADS, 1)
    k_gemm_slices(const __grid_constant__ SliceMaps maps, SliceParams p) {
  using C = SCfg<CG>;
  constexpr int STAGES = C::STAGES;
  constexpr uint32_t A_TILE = C::A_TILE, STAGE_BYTES = C::STAGE_BYTES;
  constexpr int B_ROWS = TC_BN / CG;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const uint32_t full0 = smem_u32(bars);
  const uint32_t empty0 = full0 + 8 * STAGES;
  const uint32_t tfull0 = empty0 + 8 * STAGES;
  const uint32_t tempty0 = tfull0 + 16;
  const uint32_t final_bar = tempty0 + 16;
  const uint32_t rank = CG == 2 ? cluster_rank() : 0u;
  const bool leader = rank == 0;
  const int cta0 = (int)blockIdx.x / CG, ncta = (int)gridDim.x / CG;

  __shared__ int s_prefix[kMaxGemmBatch + 1];
  __shared__ int s_total;
  if (p.blk) {
    for (int i = threadIdx.x; i < p.batch; i += TC_THREADS) {
      Blk b[2];
      const int nb = load_blocks<SBK, CG>(p, i, b);
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
      load_blocks<SBK, CG>(p, 0, b);
      s_total = b[0].tiles * p.batch;
    }
    for (int s = 0; s < STAGES; ++s) {
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
  if (warp == 0 && lane < 2) {
    const CUtensorMap* m = lane ? &maps.b : &maps.a;
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
  }
  if (warp == 1) {
    if constexpr (CG == 1) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                   "r"(TMEM_COLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                   "r"(TMEM_COLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
  }
  tc_fence_before();
  if constexpr (CG == 1) __syncthreads();
  else cluster_sync();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const int total = s_total;

  if (warp < TC_FOLD_WARP0) {
  regs_give<TC_ROLE_REGS>();
  if (warp == 0) {
    // every CTA copies its own tiles (128 rows of A, its share of the B rows); a pair's bytes all count on the first
    // CTA's barriers, and a stage is freed in both CTAs by the commit of the MMAs that read it
    if (lane == 0 && !(p.stall >> rank & 1)) {
      int stage = 0;
      uint32_t phase = 0;
      long long issued = 0;
      bool ok = true;
      for (int tile = cta0; tile < total && ok; tile += ncta) {
        int inst, mt, nt;
        Blk bk;
        locate<SBK, CG>(p, s_prefix, tile, inst, bk, mt, nt);
        const int arow = bk.m0 + mt * TC_BM * CG + (int)rank * TC_BM;
        const int brow = bk.n0 + nt * TC_BN + (int)rank * B_ROWS;
        const int binst = inst / p.b_div;
        for (int s = NSL - 1; s >= 0 && ok; --s)
          for (int kb = 0; kb < bk.num_kb && ok; ++kb) {
            const int kx = bk.k0 + kb * SBK;
            for (int i = 0; i <= s; ++i) {
              if (!mbar_wait(empty0 + 8 * stage, phase ^ 1, abort_flag, p.timeout_ns)) { ok = false; break; }
              const uint32_t fb = full0 + 8 * stage;
              const uint32_t sa = smem_u32(smem + stage * STAGE_BYTES), sb = sa + A_TILE;
              if (leader) mbar_expect_tx(fb, CG * STAGE_BYTES);
              if constexpr (CG == 1) {
                tma_load_4d(sa, &maps.a, fb, kx, arow, i, inst);
                tma_load_4d(sb, &maps.b, fb, kx, brow, s - i, binst);
              } else {
                const uint32_t fb0 = mapa_rank(fb, 0);
                tma_load_4d_pair(sa, &maps.a, fb0, kx, arow, i, inst);
                tma_load_4d_pair(sb, &maps.b, fb0, kx, brow, s - i, binst);
              }
              ++issued;
              if (++stage == STAGES) { stage = 0; phase ^= 1; }
            }
          }
      }
      // drain the copies in flight (see k_gemm_split; of a given-up pair: below)
      if (leader) {
        for (long long i = (issued > STAGES ? issued - STAGES : 0); i < issued; ++i)
          mbar_wait(full0 + 8 * (int)(i % STAGES), (uint32_t)((i / STAGES) & 1), abort_flag, drain_ns(p.timeout_ns),
                    CG == 2);
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && leader) {
      int stage = 0, buf = 0;
      uint32_t phase = 0, bphase = 0;
      bool ok = true;
      const uint64_t desc_base = smem_desc<SBK>(smem_u32(smem));
      for (int tile = cta0; tile < total && ok; tile += ncta) {
        int inst_, mt_, nt_;
        Blk bk;
        locate<SBK, CG>(p, s_prefix, tile, inst_, bk, mt_, nt_);
        for (int s = NSL - 1; s >= 0 && ok; --s) {
          const int steps = bk.num_kb * (s + 1);
          for (int t0 = 0; t0 < steps && ok; t0 += CHAIN) {
            const int g = min(CHAIN, steps - t0);
            if (!mbar_wait(tempty0 + 8 * buf, bphase ^ 1, abort_flag, p.timeout_ns)) { ok = false; break; }
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + (uint32_t)(buf * TC_BN);
            for (int t = 0; t < g; ++t) {
              if (!mbar_wait(full0 + 8 * stage, phase, abort_flag, p.timeout_ns)) { ok = false; break; }
              tc_fence_after();
              const uint64_t da = desc_base + ((uint32_t)stage * STAGE_BYTES >> 4);
              const uint64_t db = da + (A_TILE >> 4);
#pragma unroll
              for (int k = 0; k < SBK / 16; ++k)
                mma_f16<CG>(d_tmem, da + (uint64_t)(k * 2), db + (uint64_t)(k * 2), p.idesc, (t | k) ? 1u : 0u);
              mma_commit<CG>(empty0 + 8 * stage);
              if (++stage == STAGES) { stage = 0; phase ^= 1; }
            }
            if (!ok) break;
            mma_commit<CG>(tfull0 + 8 * buf);
            if (++buf == 2) { buf = 0; bphase ^= 1; }
          }
        }
      }
      mma_commit_local<CG>(final_bar);
      mbar_wait(final_bar, 0, abort_flag, drain_ns(p.timeout_ns), false);
    }
  }
  } else {
    regs_take<TC_FOLD_REGS>();
    const int q = warp & 3, half = (warp - TC_FOLD_WARP0) >> 2;
    const int ftid = (int)threadIdx.x - 32 * TC_FOLD_WARP0;
    int4* const park = p.scratch + (size_t)blockIdx.x * (SC_PLANES * 32 * TC_FOLD_THREADS) + ftid;
    const uint32_t tempty_dst = CG == 2 && !leader ? mapa_rank(tempty0, 0) : tempty0;
    int buf = 0;
    uint32_t bphase = 0;
    bool ok = true;
    // a finished tile's results are formed four columns at a time between the chains of the next tile, up to its first
    // parked level: formed at once, they held the MMAs up (683 -> 647 us at 1000 x 10000 x 1000, 2812 -> 2711 at 2048 x
    // 16384 x 2048, pairs)
    TileOut done;
    int next = 0;  // columns of `done` formed so far
    for (int tile = cta0; tile < total && ok; tile += ncta) {
      int num_kb;
      {
        int inst, mt, nt;
        Blk bk;
        locate<SBK, CG>(p, s_prefix, tile, inst, bk, mt, nt);
        num_kb = bk.num_kb;
      }
      int per = 0;  // column groups to form per chain
      if (done.dst) {
        int before = 0;
        for (int s = NSL - 1; s >= 5; --s) before += (num_kb * (s + 1) + CHAIN - 1) / CHAIN;
        per = (32 + before - 1) / max(1, before);
      }
      auto finish_some = [&](int groups) {
        if (done.dst)
          for (int g = 0; g < groups && next < done.ncol; ++g, next += 4) finish_columns<1>(p, done, park, next);
        __syncwarp();
      };
      int acc[128];
#pragma unroll
      for (int j = 0; j < 128; ++j) acc[j] = 0;
      for (int s = NSL - 1; s >= 0 && ok; --s) {
        const int chains = (num_kb * (s + 1) + CHAIN - 1) / CHAIN;
        for (int t = 0; t < chains; ++t) {
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
              acc[c * 32 + j] += __float2int_rn(__uint_as_float(r0[j]));
              acc[(c + 1) * 32 + j] += __float2int_rn(__uint_as_float(r1[j]));
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) {
            const uint32_t bar = tempty_dst + 8 * buf;
            if constexpr (CG == 1) mbar_arrive(bar);
            else if (leader) mbar_arrive(bar);
            else mbar_arrive_remote(bar);
          }
          if (++buf == 2) { buf = 0; bphase ^= 1; }
          if (s >= 5) finish_some(per);
        }
        if (!ok) break;
        if (s == 5) finish_some(32);  // (the scratch area is written from here on)
        if (s > 5) {
          // carry into the next level's unit, rounded
#pragma unroll
          for (int j = 0; j < 128; ++j) acc[j] = (acc[j] + 128) >> 8;
        } else {
          int4* dst = park + (size_t)(5 - s) * 32 * TC_FOLD_THREADS;
#pragma unroll
          for (int j = 0; j < 128; j += 4) {
            dst[(j / 4) * TC_FOLD_THREADS] =
                make_int4(acc[j], acc[j + 1], acc[j + 2], acc[j + 3]);
            acc[j] = acc[j + 1] = acc[j + 2] = acc[j + 3] = 0;
          }
        }
      }
      if (!ok) break;
      int inst, mt, nt;
      Blk bk;
      locate<SBK, CG>(p, s_prefix, tile, inst, bk, mt, nt);
      const long long row = (long long)bk.m0 + (long long)mt * TC_BM * CG + (long long)rank * TC_BM + q * 32 + lane;
      const long long col0 = (long long)bk.n0 + (long long)nt * TC_BN + half * 128;
      const long long row_end = (long long)bk.m0 + bk.mc, col_end = (long long)bk.n0 + bk.nc;
      done.dst = nullptr;
      next = 0;
      if (row < row_end && col0 < col_end) {
        done.ea = p.ea[(long long)inst * p.ea_inst + row];
        done.eb = p.eb + (long long)(inst / p.b_div) * p.eb_inst + col0;
        done.dst = p.C + (long long)inst * p.c_inst + row * p.ldc + col0;
        done.ncol = (int)min(128LL, col_end - col0);
        done.v4 = p.vec == 4 && (bk.n0 & 3) == 0 && done.ncol == 128;
      }
    }
    // the last tile (a given-up kernel leaves no result worth storing)
    if (ok && done.dst)
      for (int j0 = 0; j0 < done.ncol; j0 += 16) finish_columns<4>(p, done, park, j0);
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
    // A warp that gave up, or saw that its CTA did, tells the other CTA: after the barrier both know, and neither issues
    // copies any more.
    if (lane == 0 && *abort_flag) store_remote(mapa_rank(smem_u32(tmem_slot + 1), rank ^ 1u), 1);
    __syncwarp();
    cluster_sync();
    if (*abort_flag) {
      // Copies of a stage that only one of the CTAs filled complete no phase of its barrier, so nothing signals that the
      // last ones have landed: 2 ms, a thousand times what a copy takes, before either CTA may leave.
      for (const unsigned long long t0 = globaltimer_ns(); globaltimer_ns() - t0 < 2000000ull;) {}
      __syncwarp();
      cluster_sync();
      if (threadIdx.x == 0) atomic_status(p.status, ST_TIMEOUT);
    }
    if (warp == 1) {
      tc_fence_after();
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS)
                   : "memory");
    }
  }
}

// ---------------------------------------------------------------------------- slicing
// Column fields: fields[k] = max over the rows of X (`rows` x K, row stride ldx, instances x_inst apart) of the exponent
// field of X[.][k], an integer >= 1 for a non-zero finite entry, so 0 for a column without one; `fields` starts at zero.
// A thread per column, the rows over blockIdx.y. Bound by reading X once; the column scales cost 0.4 % of a 4D FP64 step
// (bond dimensions 5 x 6 x 4 x 5: 5.71 -> 5.73 ms), 1.5 % of a gradient (4D, bond dimension 5: 75.0 -> 76.1, where the
// tangents' operands are built twice). Zero-field operands (L != null, instance blockIdx.z): a
// column holds entries only in the rows of its class' column group.
__device__ __forceinline__ int exponent_field(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }
__device__ __forceinline__ bool is_zero(double x) { return (__double_as_longlong(x) << 1) == 0; }
constexpr int FIELD_COLS = 128;
__global__ void __launch_bounds__(FIELD_COLS) k_column_fields(const double* __restrict__ X, long long ldx, long long rows,
                                                              int K, int* fields, const Z2Layout* __restrict__ L,
                                                              long long x_inst, long long f_inst) {
  X += (long long)blockIdx.z * x_inst;
  fields += (long long)blockIdx.z * f_inst;
  const int k = blockIdx.x * FIELD_COLS + threadIdx.x;
  long long r = 0, end = k < K ? rows : 0;
  if (L && k < K) {
    L += blockIdx.z;
    const int ck = k >= L->kstart[1] ? 1 : 0;
    r = ck ? L->goff[1] : 0;
    end = k - L->kstart[ck] >= L->ncls[ck] ? r : ck ? rows : L->goff[1];
  }
  int top = 0;
#pragma unroll 4
  for (r += blockIdx.y; r < end; r += gridDim.y) {
    const double x = X[r * ldx + k];
    const int f = exponent_field(x);
    if (!is_zero(x) && f < 0x7FF) top = max(top, max(f, 1));
  }
  if (top) atomicMax(fields + k, top);
}

// One warp per row: the row's largest exponent field gives its scale, then every entry becomes NSL fp16 digits, all in
// integer arithmetic (in FP64 operations, ten an entry at two a clock and SM, a 10^4 x 10^3 operand took 160 us; its
// traffic is worth 32). Rows are read twice (the second time from L1 / L2), two columns a lane; digits are stored four
// bytes a lane, coalesced.
// Column scales: entry k counts as x 2^s(k) in Bt's rows and x 2^-s(k) in A's, s from the column fields of Bt (s cancels in
// every product of the two; it exists only as an integer added to exponent fields). `side` = -1: a row of Bt, 1: of A. In
// a column of zeros of Bt, A's entries count as zeros.
// Zero-field operands (L != null): row r of slot blockIdx.y (instance blockIdx.y / nb) belongs to a parity class that
// holds entries only in the columns [kstart, kstart + ncls) of its k class; the columns up to the next multiple of 64 get
// zeros (the GEMM's k-blocks run over them). k class of a row of Bt: its column group; of A: its row class ^ pi[slot].
constexpr int SLICE_WARPS = 4;
__device__ __forceinline__ long long fixed_point(double x, int top) {
  // x 2^(kSliceBits - e) with e = top - 1022, rounded half away from zero: the mantissa moved by the fields' difference
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int f = (int)(b >> 52) & 0x7FF;
  const unsigned long long m = (b & 0xFFFFFFFFFFFFFULL) | (f ? 1ULL << 52 : 0ULL);
  const int sh = top - max(f, 1) - (kSliceBits - 53);
  const unsigned long long v = sh <= 0 ? m << -sh : (sh > 54 ? 0ULL : (m + (1ULL << (sh - 1))) >> sh);
  return (long long)b < 0 ? -(long long)v : (long long)v;
}
// what column k's field adds to the exponent field of its entries; `dropped`: the entry counts as zero
__device__ __forceinline__ int column_shift(int field, int side, bool& dropped) {
  dropped = side > 0 && field == 0;
  return side * (max(field, 1) - 1023);
}
__global__ void __launch_bounds__(32 * SLICE_WARPS) k_slice_rows(const double* __restrict__ X, long long ldx,
                                                                 long long rows, int K, __half* out, long long ld,
                                                                 long long plane, int* __restrict__ exps,
                                                                 const Z2Layout* __restrict__ L,
                                                                 const int* __restrict__ pi, int side, long long x_inst,
                                                                 long long o_inst, long long e_inst, int nb,
                                                                 const int* __restrict__ fields, long long f_inst) {
  const int lane = threadIdx.x % 32;
  const long long row = (long long)blockIdx.x * SLICE_WARPS + threadIdx.x / 32;
  if (row >= rows) return;
  X += (long long)blockIdx.y * x_inst + row * ldx;
  out += (long long)blockIdx.y * o_inst + row * ld;
  fields += (blockIdx.y / nb) * f_inst;
  int kc = K, kpad = K;
  if (L) {
    L += blockIdx.y / nb;
    const int ck = side < 0 ? (row >= L->goff[1] ? 1 : 0) : ((row >= L->ncls[0] ? 1 : 0) ^ pi[blockIdx.y]);
    X += L->kstart[ck];
    out += L->kstart[ck];
    fields += L->kstart[ck];
    kc = L->ncls[ck];
    kpad = (kc + 63) / 64 * 64;
  }
  constexpr int kNone = -(1 << 20);  // no entry but zeros
  int top = kNone;
  bool finite = true;
#pragma unroll 4
  for (int k = lane; k < kc; k += 32) {
    const double x = X[k];
    const int f = exponent_field(x);
    bool dropped;
    const int shift = column_shift(fields[k], side, dropped);
    finite = finite && f < 0x7FF;
    if (!dropped && !is_zero(x)) top = max(top, max(f, 1) + shift);
  }
  for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
  finite = __all_sync(0xffffffffu, finite);
  if (top == kNone) top = 1022;
  if (lane == 0) exps[(long long)blockIdx.y * e_inst + row] = finite ? top - 1022 : kExpNaN;
#pragma unroll 2
  for (int k = 2 * lane; k < kpad; k += 64) {
    long long v[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      v[u] = 0;
      if (finite && k + u < kc) {
        bool dropped;
        const int shift = column_shift(fields[k + u], side, dropped);
        if (!dropped) v[u] = fixed_point(X[k + u], top - shift);
      }
    }
    const bool both = k + 1 < kpad;
#pragma unroll
    for (int i = NSL - 1; i >= 0; --i) {
      unsigned h = 0;  // 1024 + (d + 128) is an fp16 whose low bits hold d + 128
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int dgt = i ? (int)(signed char)(v[u] & 255) : (int)v[u];
        if (i) v[u] = (v[u] - dgt) >> 8;
        h |= (unsigned)(0x6400 + dgt + 128) << (16 * u);
      }
      const __half2 q = __hsub2(*reinterpret_cast<const __half2*>(&h), __half2half2(__ushort_as_half(0x6480)));
      __half* dst = out + (long long)i * plane + k;
      if (both) *reinterpret_cast<__half2*>(dst) = q;
      else dst[0] = __low2half(q);
    }
  }
}

bool slice_map(CUtensorMap* m, const __half* ptr, long long rows, long long cols, long long ld, long long plane, int batch,
               long long inst, int box_rows) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return false;
  cuuint64_t dims[4] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)NSL, (cuuint64_t)batch};
  cuuint64_t strides[3] = {(cuuint64_t)ld * 2, (cuuint64_t)plane * 2, (cuuint64_t)inst * 2};
  cuuint32_t box[4] = {SBK, (cuuint32_t)box_rows, 1, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, const_cast<__half*>(ptr), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int CG>
int launch_slices_variant(long long tiles, const SliceOperand& A, const SliceOperand& B, const SliceParams& p,
                          cudaStream_t s) {
  using Cf = SCfg<CG>;
  SliceMaps maps;
  std::memset(&maps, 0, sizeof(maps));
  if (!slice_map(&maps.a, A.p, p.M, p.K, A.ld, A.plane, p.batch, A.inst, TC_BM) ||
      !slice_map(&maps.b, B.p, p.N, p.K, B.ld, B.plane, p.batch / p.b_div, B.inst, TC_BN / CG))
    return HOTRG_EDEVICE;
  auto kern = k_gemm_slices<CG>;
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
  // the scratch area holds kSliceCtas CTAs
  const long long units = std::max(1LL, std::min({tiles, (long long)n, (long long)(kSliceCtas / CG)}));
  cfg.gridDim = dim3((unsigned)(units * CG));
  if (cudaLaunchKernelEx(&cfg, kern, maps, p) != cudaSuccess) {
    cudaGetLastError();
    return HOTRG_EDEVICE;
  }
  return HOTRG_OK;
}

long long slice_tiles(long long M, long long N, int cg) {
  return ((M + TC_BM * cg - 1) / (TC_BM * cg)) * ((N + TC_BN - 1) / TC_BN);
}

}  // namespace

bool slices_take(long long M, long long N, long long K) {
  return M >= TC_BM && N >= TC_BN && K >= 64 && K <= 16320 && M <= 0x7fffffffLL && N <= 0x7fffffffLL;
}

size_t slice_scratch_bytes(long long M, long long N, int batch) {
  // at most kSliceCtas CTAs, and at most one (or a pair) per tile of up to two blocks per instance
  const long long t = std::min<long long>(kSliceCtas, 4 * slice_tiles(M, N, 1) * batch);
  return (size_t)t * SC_PLANES * 128 * TC_FOLD_THREADS * sizeof(int);
}

void launch_column_fields(const double* X, long long ldx, long long rows, long long K, int* fields, long long f_inst,
                          int batch, long long x_inst, cudaStream_t s, const Z2Layout* L) {
  const int gx = (int)((K + FIELD_COLS - 1) / FIELD_COLS);
  // about 16 blocks an SM, at least 8 rows a block
  const long long gy = std::max(1LL, std::min((rows + 7) / 8, 152LL * 16 / ((long long)gx * batch)));
  k_column_fields<<<dim3((unsigned)gx, (unsigned)gy, (unsigned)batch), FIELD_COLS, 0, s>>>(X, ldx, rows, (int)K, fields, L,
                                                                                          x_inst, f_inst);
  count_launches(1);
}

void launch_slice_rows(const double* X, long long ldx, long long rows, long long K, const SliceOperand& out, int batch,
                       long long x_inst, const int* fields, long long f_inst, int side, cudaStream_t s, int nb,
                       const Z2Layout* L, const int* pi) {
  k_slice_rows<<<dim3((unsigned)((rows + SLICE_WARPS - 1) / SLICE_WARPS), (unsigned)batch), 32 * SLICE_WARPS, 0, s>>>(
      X, ldx, rows, (int)K, out.p, out.ld, out.plane, out.exps, L, pi, side, x_inst, out.inst, out.exp_inst, nb, fields,
      f_inst);
  count_launches(1);
}

int launch_gemm_slices(const SliceOperand& A, const SliceOperand& B, double* C, long long ldc, long long M, long long N,
                       long long K, int* scratch, int* status, double timeout_s, cudaStream_t s, const GemmBlocks* blk,
                       const GemmBatch* bat, bool accumulate, int cta_group, int stall) {
  if (!slices_take(M, N, K)) return HOTRG_EINVAL;
  if (cta_group == 0) {
    // pairs (half the B copies per SM: 647 against 708 us at 1000 x 10000 x 1000) where their 256-row tiles pad no more
    // rows than 128-row ones (else slower by what they pad: 768 against 640 rows at M = 625)
    const long long m = blk ? (M + 1) / 2 : M;
    cta_group = (m + 255) / 256 * 2 == (m + 127) / 128 ? 2 : 1;
  }
  const int batch = bat ? bat->batch : 1;
  if (batch < 1 || batch > kMaxGemmBatch || (A.ld % 8) || (B.ld % 8) || A.ld < K || B.ld < K || ldc < N)
    return HOTRG_EINVAL;
  if ((reinterpret_cast<uintptr_t>(A.p) | reinterpret_cast<uintptr_t>(B.p)) & 15) return HOTRG_EINVAL;
  if ((A.plane % 8) || (B.plane % 8) || (A.inst % 8) || (B.inst % 8)) return HOTRG_EINVAL;
  SliceParams p;
  p.M = M;
  p.N = N;
  p.K = K;
  p.num_kb = (int)((K + SBK - 1) / SBK);
  p.group_m = 16;
  p.batch = batch;
  p.b_div = bat ? bat->b_div : 1;
  if (p.b_div < 1 || batch % p.b_div) return HOTRG_EINVAL;
  p.C = C;
  p.ldc = ldc;
  p.c_inst = bat ? bat->c_inst : 0;
  p.ea = A.exps;
  p.eb = B.exps;
  p.ea_inst = A.exp_inst;
  p.eb_inst = B.exp_inst;
  p.scratch = reinterpret_cast<int4*>(scratch);
  p.status = status;
  p.timeout_ns = (unsigned long long)(timeout_s * 1e9);
  p.blk = blk;
  p.accumulate = accumulate ? 1 : 0;
  p.stall = stall;
  p.vec = (ldc % 4) == 0 && (reinterpret_cast<uintptr_t>(C) & 31) == 0 && (p.c_inst % 4) == 0 ? 4 : 1;
  p.idesc = idesc_for(true, cta_group);
  long long t = slice_tiles(M, N, cta_group) * batch;
  if (t > 0x3fffffffLL) return HOTRG_EINVAL;
  if (blk) t *= 2;  // the two blocks' tiles are counted on the device
  const int rc = cta_group == 2 ? launch_slices_variant<2>(t, A, B, p, s) : launch_slices_variant<1>(t, A, B, p, s);
  if (rc) return rc;
  count_launches(1);
  return HOTRG_OK;
}

}  // namespace hotrg
