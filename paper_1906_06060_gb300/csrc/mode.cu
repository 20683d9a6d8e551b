// Mode products of one HOTRG step (a leg of the tensor contracted with one slice of an isometry): a kernel per bond
// dimension, in a file of its own because they take as long to compile as the rest of the tensor kernels.
#include <type_traits>

#include "kernels.h"

namespace hotrg {

namespace {

// V neighbouring entries (one, or two in FP32)
template <class T, class Acc, int V>
__device__ __forceinline__ void load_run(const T* p, Acc* x) {
  if constexpr (V == 2) {
    const float2 q = *reinterpret_cast<const float2*>(p);
    x[0] = q.x;
    x[1] = q.y;
  } else {
    x[0] = (Acc)*p;
  }
}
template <class T, class Acc, int V>
__device__ __forceinline__ void store_run(T* p, const Acc* x) {
  if constexpr (V == 2) *reinterpret_cast<float2*>(p) = make_float2(x[0], x[1]);
  else *p = (T)x[0];
}

// One thread per V neighbouring "bases" (input indices with digit b = 0): it reads the DB inputs along leg b of each
// once and writes all DB outputs, so every input element is read from memory once.
// TWO: out also accumulates the same product of a second input with a second matrix (the
// tangent of a mode product: dX = M_U(dT) + M_dU(T)).
// DB = bond dimension at compile time: all loads of a thread go out together, a row of the matrix comes as 16-byte
// broadcasts and every one of its weights meets its own accumulator. With the dimension at run time (one weight read
// from shared memory per FMA, 64-bit divisions) the kernel ran at 3.0 TB/s in FP32 at D = 10 (266 us) and at a quarter
// of the FP64 units' rate at D = 6 (2.1 ms for the 42 products of a 6^4 step, now 0.9; FP32 at D = 10 now 123 us, 6.5 TB/s).
// V = 2 (FP32, even strides): half the shared-memory reads per FMA.
template <class Tin, class Tout, bool TWO, int DB, int V>
__global__ void __launch_bounds__(256) k_mode_unprimed(const Tin* __restrict__ in, Tout* __restrict__ out,
                                                       long long total, long long stride_b,
                                                       const double* __restrict__ U, int kk,
                                                       const Tin* __restrict__ in2, const double* __restrict__ U2,
                                                       unsigned* amax, long long in_inst, long long out_slot,
                                                       long long u_inst) {
  using Acc = AccT<Tout>;
  constexpr int PAD = 16 / (int)sizeof(Acc);
  constexpr int PARTS = DB > 8 ? 2 : 1, JB = (DB + PARTS - 1) / PARTS;  // outputs in one or two parts (registers)
  constexpr int WS = (JB + PAD - 1) / PAD * PAD;
  // chunk blockIdx.y of instance blockIdx.z (the input comes from L2 for every chunk but the first)
  const int slot = blockIdx.z * gridDim.y + blockIdx.y;
  in += blockIdx.z * in_inst;
  if (TWO) in2 += blockIdx.z * in_inst;
  out += slot * out_slot;
  U += blockIdx.z * u_inst;
  kk += blockIdx.y;
  if (amax) amax += slot;
  __shared__ __align__(16) Acc W[PARTS * DB * WS];
  __shared__ __align__(16) Acc W2[TWO ? PARTS * DB * WS : PAD];
  for (int t = threadIdx.x; t < DB * DB; t += blockDim.x) {
    const int i = t / DB, j = t % DB, w = (j / JB * DB + i) * WS + j % JB;
    W[w] = (Acc)U[(long long)kk * DB * DB + t];
    if (TWO) W2[w] = (Acc)U2[(long long)kk * DB * DB + t];
  }
  __syncthreads();
  const long long nbase = total / (DB * V);
  const bool small = total < (1LL << 31);
  float m = 0.f;  // max |out| of this thread (with amax: the bound of an fp16 operand's source)
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < nbase;
       t += (long long)gridDim.x * blockDim.x) {
    const long long hi = small ? (long long)((unsigned)(t * V) / (unsigned)stride_b) : t * V / stride_b;
    const long long base = t * V + hi * stride_b * (DB - 1);
    Acc x[DB][V], x2[TWO ? DB : 1][V];
#pragma unroll
    for (int i = 0; i < DB; ++i) {
      load_run<Tin, Acc, V>(in + base + i * stride_b, x[i]);
      if (TWO) load_run<Tin, Acc, V>(in2 + base + i * stride_b, x2[TWO ? i : 0]);
    }
#pragma unroll 1
    for (int part = 0; part < PARTS; ++part) {
      const Acc *w = W + part * DB * WS, *w2 = W2 + (TWO ? part * DB * WS : 0);
      Acc acc[JB][V];
#pragma unroll
      for (int j = 0; j < JB; ++j)
#pragma unroll
        for (int v = 0; v < V; ++v) acc[j][v] = 0;
#pragma unroll
      for (int i = 0; i < DB; ++i)
#pragma unroll
        for (int j = 0; j < JB; ++j)
#pragma unroll
          for (int v = 0; v < V; ++v) {
            acc[j][v] += w[i * WS + j] * x[i][v];
            if (TWO) acc[j][v] += w2[i * WS + j] * x2[TWO ? i : 0][v];
          }
#pragma unroll
      for (int j = 0; j < JB; ++j) {
        if (PARTS * JB > DB && part * JB + j >= DB) break;
        store_run<Tout, Acc, V>(out + base + (part * JB + j) * stride_b, acc[j]);
        if (amax)
#pragma unroll
          for (int v = 0; v < V; ++v) m = fmaxf(m, abs_up((Tout)acc[j][v]));
      }
    }
  }
  if (amax) {
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(amax, __float_as_uint(m));
  }
}

template <class Tin, class Tout, int DB>
void mode_unprimed(const Tin* in, long long in_inst, Tout* out, long long out_slot, long long total,
                          long long stride_b, const double* U, long long u_inst, int kk, int ng, int nb, cudaStream_t s,
                          const Tin* in2, const double* U2, unsigned* amax) {
  const long long nbase = total / DB;
  if constexpr (std::is_same<Tin, float>::value && std::is_same<Tout, float>::value) {
    // pairs of entries: every row of stride_b entries and every slot starts on an 8-byte boundary
    const bool even = stride_b % 2 == 0 && in_inst % 2 == 0 && out_slot % 2 == 0 &&
                      ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 7) == 0;
    if (even && !in2) {
      k_mode_unprimed<Tin, Tout, false, DB, 2><<<dim3(grid_for(nbase / 2, 256), nb, ng), 256, 0, s>>>(
          in, out, total, stride_b, U, kk, nullptr, nullptr, amax, in_inst, out_slot, u_inst);
      return;
    }
  }
  const dim3 grid(grid_for(nbase, 256), nb, ng);
  if (in2)
    k_mode_unprimed<Tin, Tout, true, DB, 1><<<grid, 256, 0, s>>>(in, out, total, stride_b, U, kk, in2, U2, amax, in_inst,
                                                                 out_slot, u_inst);
  else
    k_mode_unprimed<Tin, Tout, false, DB, 1><<<grid, 256, 0, s>>>(in, out, total, stride_b, U, kk, nullptr, nullptr, amax,
                                                                  in_inst, out_slot, u_inst);
}

}  // namespace

template <class Tin, class Tout>
void launch_mode_unprimed(const Tin* in, long long in_inst, Tout* out, long long out_slot, Geom g, int b, const double* U,
                          long long u_inst, int kk, int ng, int nb, cudaStream_t s, const Tin* in2, const double* U2,
                          unsigned* amax) {
  const long long total = g.P * g.P;
  if (amax) cudaMemsetAsync(amax, 0, sizeof(unsigned) * ng * nb, s);
  switch (g.D[b]) {
#define HOTRG_MODE_DB(C)                                                                                               \
  case C:                                                                                                              \
    mode_unprimed<Tin, Tout, C>(in, in_inst, out, out_slot, total, g.Sn[b] * g.P, U, u_inst, kk, ng, nb, s, in2, U2,   \
                                amax);                                                                                 \
    break;
    HOTRG_MODE_DB(1) HOTRG_MODE_DB(2) HOTRG_MODE_DB(3) HOTRG_MODE_DB(4) HOTRG_MODE_DB(5) HOTRG_MODE_DB(6)
    HOTRG_MODE_DB(7) HOTRG_MODE_DB(8) HOTRG_MODE_DB(9) HOTRG_MODE_DB(10) HOTRG_MODE_DB(11) HOTRG_MODE_DB(12)
    HOTRG_MODE_DB(13) HOTRG_MODE_DB(14) HOTRG_MODE_DB(15) HOTRG_MODE_DB(16)
#undef HOTRG_MODE_DB
  }
  count_launches(1);
}

#define HOTRG_MODE(TI, TO)                                                                                            \
  template void launch_mode_unprimed<TI, TO>(const TI*, long long, TO*, long long, Geom, int, const double*, long long, \
                                             int, int, int, cudaStream_t, const TI*, const double*, unsigned*);
HOTRG_MODE(double, double)
HOTRG_MODE(double, float)
HOTRG_MODE(float, float)
#undef HOTRG_MODE

}  // namespace hotrg
