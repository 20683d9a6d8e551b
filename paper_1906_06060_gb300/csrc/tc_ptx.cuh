// Shared parts of the tcgen05 GEMM kernels (gemm_tc.cu: split-precision products; gemm_f64tc.cu: FP64 products
// from exact integer slices): inline-PTX wrappers (mbarrier, TMA, tcgen05, clusters), the output tile list, and the
// host's tensor-map encoder. Everything is local to the including file.
#pragma once
#include <cuda.h>

#include <algorithm>
#include <atomic>
#include <cstring>

#include "kernels.h"

namespace hotrg {

namespace {

constexpr int TC_BM = 128, TC_BN = 256;
constexpr int kMaxDevices = 64;
// Warpgroup 0: warp 0 copies, warp 1 issues MMAs (warps 2 and 3 idle); warpgroups 1 and 2 (warps 4-11): fold. The fold
// warps hold 128 sums a thread beside the tensor-memory loads in flight: they take registers over from warpgroup 0
// (setmaxnreg; the shares add up to what the launch allocates, 168 x 384).
constexpr int TC_THREADS = 384;
constexpr int TC_FOLD_WARP0 = 4;
constexpr int TC_FOLD_THREADS = 256;
constexpr int TC_LAUNCH_REGS = 168;
constexpr int TC_ROLE_REGS = 56, TC_FOLD_REGS = 224;
static_assert(128 * TC_ROLE_REGS + TC_FOLD_THREADS * TC_FOLD_REGS <= TC_LAUNCH_REGS * TC_THREADS, "register shares");
constexpr uint32_t TMEM_COLS = 2 * TC_BN;

// kind::f16 instruction descriptor: D = F32 (bits 4-5 = 1), A and B format (bits 7-9, 10-12:
// 1 = BF16, 0 = F16; A and B always of the same type), both K-major, N >> 3 at bits 17-22,
// M >> 4 at bits 24-28 (M = 128 for one CTA, 256 for a CTA pair: 128 rows in each).
constexpr uint32_t idesc_for(bool f16, int cg) {
  return (1u << 4) | (f16 ? 0u : (1u << 7) | (1u << 10)) | ((uint32_t)(TC_BN >> 3) << 17) |
         ((uint32_t)((TC_BM * cg) >> 4) << 24);
}

// One output block of the product as the kernel sees it (clamped to the operand extents).
struct Blk {
  int m0, mc, n0, nc, k0, num_m, num_n, num_kb, tiles;
};

// The (at most two) blocks of instance `inst`: from its device descriptor of a block-sparse
// product (clamped to the operand extents), or the single dense block. Output tiles are
// (128 CG) x 256: a CTA pair (CG = 2) computes 256 rows.
template <int BK, int CG, class Par>
__device__ __forceinline__ int load_blocks(const Par& p, int inst, Blk* b) {
  int nb = 1;
  if (p.blk) {
    const GemmBlocks* g = p.blk + inst;
    nb = min(max(g->nb, 0), 2);
    for (int i = 0; i < nb; ++i) {
      const long long m0 = max(g->m0[i], 0), n0 = max(g->n0[i], 0), k0 = max(g->k0[i], 0);
      b[i].m0 = (int)min(m0, p.M);
      b[i].n0 = (int)min(n0, p.N);
      b[i].k0 = (int)min(k0, p.K);
      b[i].mc = (int)min((long long)max(g->mc[i], 0), p.M - b[i].m0);
      b[i].nc = (int)min((long long)max(g->nc[i], 0), p.N - b[i].n0);
      const int kc = (int)min((long long)max(g->kc[i], 0), p.K - b[i].k0);
      b[i].num_kb = (kc + BK - 1) / BK;
    }
  } else {
    b[0].m0 = b[0].n0 = b[0].k0 = 0;
    b[0].mc = (int)p.M;
    b[0].nc = (int)p.N;
    b[0].num_kb = p.num_kb;
  }
  for (int i = 0; i < nb; ++i) {
    b[i].num_m = (b[i].mc + TC_BM * CG - 1) / (TC_BM * CG);
    b[i].num_n = (b[i].nc + TC_BN - 1) / TC_BN;
    b[i].tiles = b[i].num_m * b[i].num_n;
  }
  return nb;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait. Returns false if another role aborted or this wait exceeded timeout_ns.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                       unsigned long long timeout_ns, bool honour_abort = true) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = globaltimer_ns();
  for (;;) {
#pragma unroll 1
    for (int i = 0; i < 32; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (honour_abort && *abort_flag) return false;
    if (globaltimer_ns() - t0 > timeout_ns) {
      *abort_flag = 1;
      return false;
    }
  }
}
// Limit of the waits for work this CTA already issued (TMA copies, MMAs), which always
// completes: at least one second, so that a short caller limit cannot let the CTA exit (and
// release TMEM or shared memory) while that work is still in flight.
__device__ __forceinline__ unsigned long long drain_ns(unsigned long long timeout_ns) {
  return timeout_ns > 1000000000ull ? timeout_ns : 1000000000ull;
}
// 3D tiled load: x along K (a multiple of BK: 16-byte aligned starts), y the tile's first row, z the
// instance of a batched launch (0 otherwise)
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y,
                                            int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], "
      "[%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y), "r"(z)
      : "memory");
}
// The same load for a CTA pair: `dst` is a shared::cluster address in either CTA (mapa for the other one), the bytes count
// on the first CTA's barrier `bar` (a shared::cluster address).
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y,
                                                 int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, "
      "{%3, %4, %5}], [%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y), "r"(z)
      : "memory");
}
// shared::cluster address of this CTA's shared-memory location `a` in cluster CTA `rank`
__device__ __forceinline__ uint32_t mapa_rank(uint32_t a, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// store to another CTA's shared memory (shared::cluster address)
__device__ __forceinline__ void store_remote(uint32_t a, int v) {
  asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
// every thread of both CTAs of the cluster (release / acquire at cluster scope)
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// arrive on a barrier of another CTA of the cluster (shared::cluster address)
__device__ __forceinline__ void mbar_arrive_remote(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// No "memory" clobber: the MMA reads shared memory the async proxy filled and writes TMEM; its
// order against the mbarrier waits and tcgen05.commit around it is kept because all of these are
// volatile asm statements, which the compiler does not reorder among themselves.
// CG = 2: issued by the pair's first CTA; A rows and B rows come from both CTAs' shared memory
// (the same offsets), each CTA's tensor memory receives its 128 rows of D.
template <int CG>
__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                        uint32_t accumulate) {
  if constexpr (CG == 1)
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
  else
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}
// Arrive on `bar` once the MMAs this thread issued so far have completed. CG = 2: on the barrier
// at the same offset in both CTAs of the pair.
template <int CG>
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  if constexpr (CG == 1)
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
  else
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
            bar),
        "h"((uint16_t)3)
        : "memory");
}
// the same, on this CTA's barrier only
template <int CG>
__device__ __forceinline__ void mma_commit_local(uint32_t bar) {
  if constexpr (CG == 1)
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
  else
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}
// Shared-memory matrix descriptor, K-major operand staged by TMA with a BK*2-byte swizzle:
// start address >> 4 (bits 0-13), leading byte offset 16 B (unused for these layouts, bits
// 16-29), stride byte offset = 8 rows x BK*2 bytes between 8-row groups (bits 32-45), version 1
// (bits 46-47), base offset 0 (tiles are 1024-B aligned), layout SWIZZLE_128B = 2 or
// SWIZZLE_64B = 4 (bits 61-63). Consecutive K=16 slices are 32 bytes apart inside a row.
template <int BK>
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= ((uint64_t)(BK == 64 ? 1024 : 512) >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)(BK == 64 ? 2 : 4) << 61;
  return d;
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
        "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
        "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
        "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
template <int N>
__device__ __forceinline__ void regs_give() {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N>
__device__ __forceinline__ void regs_take() {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}
__device__ __forceinline__ void tmem_ld_wait() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void raster(int tile, int num_m, int num_n, int group_m, int& mt, int& nt) {
  const int per_group = group_m * num_n;
  const int g = tile / per_group;
  const int first_m = g * group_m;
  const int gsz = min(num_m - first_m, group_m);
  const int local = tile - g * per_group;
  mt = first_m + local % gsz;
  nt = local / gsz;
}

// Tile -> (instance, block, M-tile, N-tile). Instances' tiles are numbered one after the other
// (prefix[i] = first tile of instance i, for block-sparse launches), and inside an instance the
// blocks' tiles one after the other.
template <int BK, int CG, class Par>
__device__ __forceinline__ void locate(const Par& p, const int* prefix, int tile, int& inst, Blk& bk, int& mt,
                                       int& nt) {
  Blk b[2];
  int local;
  if (!p.blk) {
    load_blocks<BK, CG>(p, 0, b);
    inst = tile / b[0].tiles;
    local = tile - inst * b[0].tiles;
    bk = b[0];
  } else {
    int lo = 0, hi = p.batch;  // prefix[lo] <= tile < prefix[hi]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (prefix[mid] <= tile) lo = mid;
      else hi = mid;
    }
    inst = lo;
    local = tile - prefix[lo];
    const int nb = load_blocks<BK, CG>(p, inst, b);
    const int bi = (nb > 1 && local >= b[0].tiles) ? 1 : 0;
    if (bi) local -= b[0].tiles;
    bk = b[bi];
  }
  raster(local, bk.num_m, bk.num_n, p.group_m, mt, nt);
}

// ------------------------------------------------------------------ host
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  }
  return fn;
}

// SM count of the current device (cached per device)
int num_sms() {
  static std::atomic<int> cache[kMaxDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    cudaGetLastError();
    return 1;
  }
  int n = cache[dev].load();
  if (n <= 0) {
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
      cudaGetLastError();
      n = 1;
    }
    cache[dev].store(n);
  }
  return n;
}

}  // namespace

}  // namespace hotrg
