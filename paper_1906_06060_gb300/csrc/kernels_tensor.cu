// Element-wise, reduction and re-layout kernels of one HOTRG step (arXiv:1906.06060, Sec. 2).
// The squeeze GEMM itself lives in gemm_tc.cu (tensor cores) and gemm_simt.cu (FP64).
#include <atomic>
#include <type_traits>

#include "kernels.h"

namespace hotrg {

static std::atomic<long long> g_launches{0};
void count_launches(int n) { g_launches.fetch_add(n, std::memory_order_relaxed); }
long long launches_total() { return g_launches.load(std::memory_order_relaxed); }

namespace {

constexpr int kNormBlocks = 1024;

// ---------------------------------------------------------------------------- max |x|
// *out = max(*out, max |x|) over rows x cols entries with row stride ld, as the bits of a
// non-negative float (their unsigned order is the order of the values). NaN entries are skipped.
template <class T>
__global__ void __launch_bounds__(256) k_absmax(const T* __restrict__ x, long long rows, long long cols,
                                                long long ld, unsigned* out, long long x_inst) {
  x += (long long)blockIdx.y * x_inst;
  out += blockIdx.y;
  float m = 0.f;
  // contiguous rows as one, else a row per block at a time (no index division: 110 us at 16807 x 2401 with one)
  const bool flat = ld == cols;
  const long long n = flat ? rows * cols : cols, nr = flat ? 1 : rows;
  const long long i0 = threadIdx.x + (flat ? (long long)blockIdx.x * 256 : 0), step = flat ? (long long)gridDim.x * 256 : 256;
  for (long long r = flat ? 0 : blockIdx.x; r < nr; r += gridDim.x) {
    const T* xr = x + r * ld;
#pragma unroll 8
    for (long long i = i0; i < n; i += step) m = fmaxf(m, abs_up(xr[i]));
  }
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, __float_as_uint(m));
}

// ---------------------------------------------------------------------------- T^(0)
// T[idx] = sum_s V_s prod_{legs} W[s, leg]; W[s,0] = sqrt(cosh b), W[s,1] = s sqrt(sinh b),
// V_s = e^{b h s}; bit l of idx (from the most significant) is the index of leg l.
__global__ void k_init_tensor(double* T, long long inst_stride, int d, const double* beta,
                              const double* hfield, int spin_insertion) {
  const int nlegs = 2 * d;
  const int total = 1 << nlegs;
  const int inst = blockIdx.y;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= total) return;
  const double b = beta[inst], h = hfield[inst];
  const double wc = sqrt(cosh(b)), ws = sqrt(sinh(b));
  double acc = 0.0;
  for (int si = 0; si < 2; ++si) {
    const double s = si ? -1.0 : 1.0;
    double v = exp(s * b * h);
    for (int l = 0; l < nlegs; ++l) {
      const int bit = (idx >> (nlegs - 1 - l)) & 1;
      v *= bit ? s * ws : wc;
    }
    acc += spin_insertion ? s * v : v;
  }
  T[inst * inst_stride + idx] = acc;
}

// ---------------------------------------------------------------------------- T^(0) tangents
// dT[idx] = d T^(0)[idx] / d beta (which = 0) or d / d h (which = 1). With n1 legs at index 1 and
// n0 = 2d - n1 at index 0, prod W = cosh^{n0/2} (s sinh^{1/2})^{n1} and
//   d/d beta [V_s prod W] = V_s prod W (h s + n0 tanh(b)/2 + n1 coth(b)/2),
//   d/d h    [V_s prod W] = V_s prod W (b s).
__global__ void k_init_tangent(double* dT, long long inst_stride, int d, const double* beta, const double* hfield,
                               int which) {
  const int nlegs = 2 * d;
  const int total = 1 << nlegs;
  const int inst = blockIdx.y;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= total) return;
  const double b = beta[inst], h = hfield[inst];
  const double wc = sqrt(cosh(b)), ws = sqrt(sinh(b));
  const int n1 = __popc(idx);
  const int n0 = nlegs - n1;
  double acc = 0.0;
  for (int si = 0; si < 2; ++si) {
    const double s = si ? -1.0 : 1.0;
    double v = exp(s * b * h);
    for (int l = 0; l < nlegs; ++l) {
      const int bit = (idx >> (nlegs - 1 - l)) & 1;
      v *= bit ? s * ws : wc;
    }
    const double f = which == 0 ? h * s + 0.5 * n0 * tanh(b) + 0.5 * n1 / tanh(b) : b * s;
    acc += v * f;
  }
  dT[inst * inst_stride + idx] = acc;
}

// ---------------------------------------------------------------------------- norms
template <int BS>
__device__ double block_sum(double v, double* sh) {
  sh[threadIdx.x] = v;
  __syncthreads();
  for (int w = BS / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  double r = sh[0];
  __syncthreads();
  return r;
}

__global__ void __launch_bounds__(256) k_sumsq_partial(const double* __restrict__ x, long long x_inst, long long n,
                                                       double* __restrict__ partial) {
  __shared__ double sh[256];
  x += (long long)blockIdx.y * x_inst;
  partial += (long long)blockIdx.y * kNormBlocks;
  double s = 0.0;
  for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < n; i += (long long)kNormBlocks * 256) {
    const double v = x[i];
    s = fma(v, v, s);
  }
  const double t = block_sum<256>(s, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = t;
}

__global__ void k_step_advance(int* dstep) { *dstep += 1; }

__global__ void __launch_bounds__(256) k_norm_finish(const double* __restrict__ partial, double* c_out,
                                                     double* lnc_log, long long log_inst, double* L, const int* dstep,
                                                     int* status) {
  const int step = *dstep;
  partial += (long long)blockIdx.x * kNormBlocks;
  c_out += blockIdx.x;
  lnc_log += (long long)blockIdx.x * log_inst;
  L += blockIdx.x;
  __shared__ double sh[256];
  double s = 0.0;
  for (int i = threadIdx.x; i < kNormBlocks; i += 256) s += partial[i];
  const double t = block_sum<256>(s, sh);
  if (threadIdx.x == 0) {
    const double c = sqrt(t);
    if (!(c > 0.0) || !isfinite(c)) atomic_status(status, ST_NUMERIC);
    const double lc = log(c);
    *c_out = c;
    lnc_log[step] = lc;
    *L += ldexp(lc, -step);
  }
}

// partial[b] = sum over this block's share of x[i] (y1[i] + y2[i]) (y2 may be null): fixed grid.
__global__ void __launch_bounds__(256) k_dot_partial(const double* __restrict__ x, const double* __restrict__ y1,
                                                     const double* __restrict__ y2, long long n,
                                                     double* __restrict__ partial) {
  __shared__ double sh[256];
  double s = 0.0;
  for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < n; i += (long long)kNormBlocks * 256) {
    const double y = y2 ? y1[i] + y2[i] : y1[i];
    s = fma(x[i], y, s);
  }
  const double t = block_sum<256>(s, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = t;
}

// dlnc = <T, D> / c^2 for the tangent D of an unnormalised tensor T with norm c; dL += 2^-n dlnc.
__global__ void __launch_bounds__(256) k_tangent_finish(const double* __restrict__ partial, const double* c,
                                                        double* dlnc, double* dL, const int* dstep) {
  __shared__ double sh[256];
  double s = 0.0;
  for (int i = threadIdx.x; i < kNormBlocks; i += 256) s += partial[i];
  const double t = block_sum<256>(s, sh);
  if (threadIdx.x == 0) {
    const double cv = *c;
    const double v = t / (cv * cv);
    *dlnc = v;
    *dL += ldexp(v, -*dstep);
  }
}

// dTn = (D1 + D2) / c - dlnc T / c : the tangent of T / ||T||.
// D1 and dTn may be the same buffer (each element is read before it is written, by one thread).
__global__ void k_tangent_update(const double* __restrict__ T, const double* D1,
                                 const double* __restrict__ D2, double* dTn, long long n,
                                 const double* c, const double* dlnc) {
  const double inv = 1.0 / *c, g = *dlnc;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const double d = D2 ? D1[i] + D2[i] : D1[i];
    dTn[i] = (d - g * T[i]) * inv;
  }
}

// d(ln Z/N) = dL + 2^-n Tr dT / Tr T for every instance (one CTA each).
__global__ void __launch_bounds__(256) k_trace_tangent(const double* __restrict__ T, const double* __restrict__ dT,
                                                       long long t_stride, long long P, const double* dL,
                                                       const int* dstep, double* out) {
  __shared__ double sh[256];
  T += (long long)blockIdx.x * t_stride;
  dT += (long long)blockIdx.x * t_stride;
  double a = 0.0, b = 0.0;
  for (long long u = threadIdx.x; u < P; u += 256) {
    a += T[u * P + u];
    b += dT[u * P + u];
  }
  const double ta = block_sum<256>(a, sh);
  const double tb = block_sum<256>(b, sh);
  if (threadIdx.x == 0) out[blockIdx.x] = dL[blockIdx.x] + ldexp(tb / ta, -*dstep);
}

// out[i] = Tr S_i / Tr T_i for every instance (one CTA each): Eqs. (energy), (spin).
__global__ void __launch_bounds__(256) k_trace_ratio(const double* __restrict__ S, const double* __restrict__ T,
                                                     long long t_stride, long long P, double* out) {
  __shared__ double sh[256];
  S += (long long)blockIdx.x * t_stride;
  T += (long long)blockIdx.x * t_stride;
  double a = 0.0, b = 0.0;
  for (long long u = threadIdx.x; u < P; u += 256) {
    a += S[u * P + u];
    b += T[u * P + u];
  }
  const double ta = block_sum<256>(a, sh);
  const double tb = block_sum<256>(b, sh);
  if (threadIdx.x == 0) out[blockIdx.x] = ta / tb;
}

__global__ void k_scale(const double* __restrict__ src, long long src_inst, double* __restrict__ dst, long long dst_inst,
                        long long n, const double* __restrict__ c) {
  src += (long long)blockIdx.y * src_inst;
  dst += (long long)blockIdx.y * dst_inst;
  const double cv = c[blockIdx.y];
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    dst[i] = src[i] / cv;
}

// ---------------------------------------------------------------------------- trace, X^(n)
// out3[0] = Tr T, out3[1] = L + 2^-step ln Tr T, out3[2] = X^(n) along axis.
__global__ void __launch_bounds__(256) k_trace_x(const double* __restrict__ T, long long t_stride, Geom g,
                                                 int axis, const double* L, const int* dstep, double* out3) {
  __shared__ double sh[256];
  const int step = *dstep;
  T += (long long)blockIdx.x * t_stride;
  L += blockIdx.x;
  out3 += 3 * blockIdx.x;
  __shared__ double A[kMaxBond * kMaxBond];
  const long long P = g.P;
  double s = 0.0;
  for (long long u = threadIdx.x; u < P; u += 256) s += T[u * P + u];
  const double tr = block_sum<256>(s, sh);
  // A_{ij} = sum over the other slots (equal on both halves) with slot `axis` = i / j.
  const int Da = g.D[axis];
  const long long Sa = g.Sn[axis];
  const long long nrest = P / Da;
  for (int e = threadIdx.x; e < Da * Da; e += 256) {
    const int i = e / Da, j = e % Da;
    double acc = 0.0;
    for (long long r = 0; r < nrest; ++r) {
      // r enumerates the other slots: split r around slot `axis`
      const long long hi = r / Sa, lo = r % Sa;
      const long long base = hi * Sa * Da + lo;
      acc += T[(base + i * Sa) * P + base + j * Sa];
    }
    A[e] = acc;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double trA = 0.0, trA2 = 0.0;
    for (int i = 0; i < Da; ++i) trA += A[i * Da + i];
    for (int i = 0; i < Da; ++i)
      for (int j = 0; j < Da; ++j) trA2 += A[i * Da + j] * A[j * Da + i];
    // a non-positive trace is reported by the free-energy query, not here
    out3[0] = tr;
    out3[1] = tr > 0.0 ? *L + ldexp(log(tr), -step) : nan("");
    out3[2] = trA * trA / trA2;
  }
}

// ---------------------------------------------------------------------------- transpose
template <class Tout>
__global__ void __launch_bounds__(256) k_transpose(const double* __restrict__ T, Tout* __restrict__ Tt,
                                                   long long P, long long t_inst, long long tt_inst) {
  __shared__ double tile[32][33];
  T += blockIdx.z * t_inst;
  Tt += blockIdx.z * tt_inst;
  const long long r0 = (long long)blockIdx.y * 32, c0 = (long long)blockIdx.x * 32;
  for (int k = threadIdx.y; k < 32; k += 8) {
    const long long r = r0 + k, c = c0 + threadIdx.x;
    if (r < P && c < P) tile[k][threadIdx.x] = T[r * P + c];
  }
  __syncthreads();
  for (int k = threadIdx.y; k < 32; k += 8) {
    const long long r = c0 + k, c = r0 + threadIdx.x;  // Tt[r][c] = T[c][r]
    if (r < P && c < P) Tt[r * P + c] = (Tout)tile[threadIdx.x][k];
  }
}

// ---------------------------------------------------------------------------- B operand
// Bt[(j*P + n)][k] = sum_x U3[j][k_c3][x] Tt[n][k | c3 := x]
// TWO: the row also accumulates sum_x U3b[j][k_c3][x] Tt2[n][k | c3 := x] (the tangent of the
// B operand: dBt = B_U3(dTt) + B_dU3(Tt)).
// A thread holds the Dc source entries of its (n, k) and forms the rows of all its j from them (block z: j0 = z jper up to
// jper rows). One output a thread read its source entries again for every j and one weight per FMA (with 64-bit index divisions 1.25 ms
// for an 8^4 tensor, 10.3 for the zero-field 10^4; 0.50 and 4.8 this way).
template <class Tin, class Tout, bool TWO>
__global__ void __launch_bounds__(256) k_build_bt(const Tin* __restrict__ Tt, Planes<Tout> out,
                                                  long long ld, long long P,
                                                  long long Sc, int Dc, const double* __restrict__ U3,
                                                  int chi3, const Tin* __restrict__ Tt2,
                                                  const double* __restrict__ U3b, long long tt_inst, long long out_inst,
                                                  long long u_inst, int jper) {
  using Acc = AccT<Tout>;
  Tt += blockIdx.y * tt_inst;
  if (TWO) Tt2 += blockIdx.y * tt_inst;
  if (U3) U3 += blockIdx.y * u_inst;
  out.advance(blockIdx.y, out_inst);
  extern __shared__ __align__(16) unsigned char smraw[];
  Acc* W = reinterpret_cast<Acc*>(smraw);  // [chi3][Dc][bt_row(Dc)], then the same for U3b
  const int ws = bt_row<Acc>(Dc), nW = chi3 * Dc * ws;
  Acc* W2 = W + nW;
  load_bt_weights(W, U3, chi3, Dc);
  if (TWO) load_bt_weights(W2, U3b, chi3, Dc);
  __syncthreads();
  const long long total = P * P;
  const int j0 = blockIdx.z * jper, j1 = min(chi3, j0 + jper);
  for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    const BtIndex e(idx, P, total);
    const unsigned k = e.k;
    const long long n = e.row;
    if (Sc == 0) {
      for (int j = j0; j < j1; ++j) store_planes(out, (j * P + n) * ld + k, (Acc)Tt[idx]);
      continue;
    }
    const unsigned kc = (k / (unsigned)Sc) % (unsigned)Dc;
    const long long base = idx - (long long)kc * Sc;
    Acc x[kMaxBond], x2[TWO ? kMaxBond : 1];
#pragma unroll
    for (int i = 0; i < kMaxBond; ++i)
      if (i < Dc) {
        x[i] = (Acc)Tt[base + i * Sc];
        if (TWO) x2[TWO ? i : 0] = (Acc)Tt2[base + i * Sc];
      }
    for (int j = j0; j < j1; ++j) {
      Acc acc = bt_dot((Acc)0, W + (j * Dc + (int)kc) * ws, x, Dc);
      if constexpr (TWO) acc = bt_dot(acc, W2 + (j * Dc + (int)kc) * ws, x2, Dc);
      store_planes(out, (j * P + n) * ld + k, acc);
    }
  }
}

// ---------------------------------------------------------------------------- A operand
// Y[m][k] = X[R(k) + C(m)], R(k) = sum_{b!=a} k_b Sn_b P + k_a Sn_a, C(m) = sum_{b!=a} m_b Sn_b + m_a Sn_a P.
// Tiles of 32 columns x (32 kYMT) rows; when a is the fastest slot the source is contiguous along k
// (no transpose), otherwise along m (transpose through shared memory, one 32 x 32 tile at a time).
// Warp 0 decomposes the tile's 32 k, warps 1..kYMT its rows, at the same time, in 32-bit index
// arithmetic (P < 2^31); the fp16 scale of the planes is read once per thread.
constexpr int kYMT = 4;
template <class Tin, class Tout>
__global__ void __launch_bounds__(256) k_build_y(const Tin* __restrict__ X, Planes<Tout> out, long long ld,
                                                 Geom g, int a, long long x_slot, long long out_slot) {
  using Acc = AccT<Tout>;
  X += blockIdx.z * x_slot;
  out.advance(blockIdx.z, out_slot);
  __shared__ Acc tile[32][33];
  __shared__ long long Rk[32], Cm[32 * kYMT];
  const int P = (int)g.P;
  const long long PP = g.P;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int m0 = blockIdx.y * 32 * kYMT, k0 = blockIdx.x * 32;
  if (ty == 0) {
    const int k = k0 + tx;
    long long rk = 0;
    for (int b = 0; b < g.d; ++b) {
      const int sb = (int)g.Sn[b];
      const long long kb = (k / sb) % g.D[b];
      rk += b == a ? kb * sb : kb * sb * PP;
    }
    Rk[tx] = rk;
  } else if (ty <= kYMT) {
    const int r = (ty - 1) * 32 + tx;
    const int m = m0 + r;
    long long cm = 0;
    for (int b = 0; b < g.d; ++b) {
      const int sb = (int)g.Sn[b];
      const long long mb = (m / sb) % g.D[b];
      cm += b == a ? mb * sb * PP : mb * sb;
    }
    Cm[r] = cm;
  }
  __syncthreads();
  const float sc = plane_scale(out);
  const int k = k0 + tx;
  if (a == g.d - 1) {
    // contiguous along k: the thread's 4 kYMT loads first, then the stores
    Acc v[4 * kYMT];
#pragma unroll
    for (int q = 0; q < 4 * kYMT; ++q) {
      const int m = m0 + ty + 8 * q;
      v[q] = (m < P && k < P) ? (Acc)X[Rk[tx] + Cm[ty + 8 * q]] : (Acc)0;
    }
#pragma unroll
    for (int q = 0; q < 4 * kYMT; ++q) {
      const int m = m0 + ty + 8 * q;
      if (m < P && k < P) store_planes_sc(out, (long long)m * ld + k, v[q], sc);
    }
  } else {
    for (int t = 0; t < kYMT; ++t) {
      for (int r = ty; r < 32; r += 8) {  // r indexes k, tx indexes m
        const int kr = k0 + r, m = m0 + t * 32 + tx;
        if (m < P && kr < P) tile[r][tx] = (Acc)X[Rk[r] + Cm[t * 32 + tx]];
      }
      __syncthreads();
      for (int r = ty; r < 32; r += 8) {  // r indexes m, tx indexes k
        const int m = m0 + t * 32 + r;
        if (m < P && k < P) store_planes_sc(out, (long long)m * ld + k, tile[tx][r], sc);
      }
      __syncthreads();
    }
  }
}

// ---------------------------------------------------------------------------- pair contraction
template <class Tin, class Tout>
__global__ void __launch_bounds__(256) k_pair_contract(const Tin* __restrict__ in, Tout* __restrict__ out,
                                                       View v, long long total, int kaxis, int Di, int Dj,
                                                       long long si, long long sj,
                                                       const double* __restrict__ U, int chi,
                                                       long long in_base, long long out_base) {
  using Acc = AccT<Tout>;
  extern __shared__ unsigned char smraw[];
  Acc* W = reinterpret_cast<Acc*>(smraw);  // [chi][Di][Dj]
  const int nW = chi * Di * Dj;
  for (int t = threadIdx.x; t < nW; t += blockDim.x) W[t] = U ? (Acc)U[t] : (Acc)1;
  __syncthreads();
  for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    long long rem = idx, ioff = in_base, ooff = out_base;
    int kp = 0;
    for (int ax = v.ndim - 1; ax >= 0; --ax) {
      const long long c = rem % v.shape[ax];
      rem /= v.shape[ax];
      ioff += c * v.in_stride[ax];
      ooff += c * v.out_stride[ax];
      if (ax == kaxis) kp = (int)c;
    }
    const Acc* w = W + (long long)kp * Di * Dj;
    Acc acc = 0;
    for (int i = 0; i < Di; ++i) {
      const Tin* src = in + ioff + i * si;
      for (int j = 0; j < Dj; ++j) acc += w[i * Dj + j] * (Acc)src[j * sj];
    }
    out[ooff] = (Tout)acc;
  }
}

// All chi outputs of one "rest" index per thread: out[o + k' sk] = sum_{i,j} U[k'][i][j] in[r + i si + j sj]
// (r, o: offsets of the rest index in the input and output views). Every input element is read
// once; W is held in shared memory as [i][j][k'], rows padded to 16 bytes, so a warp reads it by broadcast.
// TWO: out also accumulates the same contraction of in2 with U2 (the tangent of an epilogue
// contraction: dR' = C_U(dR) + C_dU(R)).
// CHI = chi at compile time (exact accumulators, no predicated-off FMAs). NJ = Dj at compile time for the FP32
// steady-state shape (chi = Dj; a row of loads is issued before its FMAs), 0: any Dj, four loads at a time. The FP64
// instances are bound by the FP64 units (chi FMAs per input entry at two a clock and SM).
template <class Tin, class Tout, bool TWO, int CHI, int NJ>
__global__ void __launch_bounds__(256) k_pair_contract_all(const Tin* __restrict__ in, Tout* __restrict__ out,
                                                           View v, long long total, int Di, int Dj,
                                                           long long si, long long sj, long long sk,
                                                           const double* __restrict__ U, long long out_base,
                                                           const Tin* __restrict__ in2,
                                                           const double* __restrict__ U2, SlotStrides st) {
  using Acc = AccT<Tout>;
  constexpr int PAD = 16 / (int)sizeof(Acc);
  constexpr int WS = (CHI + PAD - 1) / PAD * PAD;
  constexpr int U4 = NJ > 0 ? NJ : 4;  // loads issued together
  extern __shared__ __align__(16) unsigned char smraw[];
  Acc* W = reinterpret_cast<Acc*>(smraw);  // [Di*Dj][WS], then the same for U2
  const long long in_off = (blockIdx.z * gridDim.y + blockIdx.y) * st.in_slot;
  out_base += blockIdx.z * st.out_inst + blockIdx.y * st.out_chunk;
  in += in_off;
  if (TWO) in2 += in_off;
  U += blockIdx.z * st.u_inst;
  const int nij = Di * Dj;
  Acc* W2 = W + (long long)WS * nij;
  for (int t = threadIdx.x; t < WS * nij; t += blockDim.x) {
    const int k = t / nij, ij = t % nij;
    W[ij * WS + k] = k < CHI ? (Acc)U[t] : (Acc)0;
    if (TWO) W2[ij * WS + k] = k < CHI ? (Acc)U2[t] : (Acc)0;
  }
  __syncthreads();
  for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    long long ioff = 0, ooff = out_base;
    if (total <= 0xffffffffLL) {
      unsigned rem = (unsigned)idx;
      for (int ax = v.ndim - 1; ax >= 0; --ax) {
        const unsigned n = (unsigned)v.shape[ax], q = rem / n, c = rem - q * n;
        rem = q;
        ioff += c * v.in_stride[ax];
        ooff += c * v.out_stride[ax];
      }
    } else {
      long long rem = idx;
      for (int ax = v.ndim - 1; ax >= 0; --ax) {
        const long long c = rem % v.shape[ax];
        rem /= v.shape[ax];
        ioff += c * v.in_stride[ax];
        ooff += c * v.out_stride[ax];
      }
    }
    Acc acc[CHI];
#pragma unroll
    for (int k = 0; k < CHI; ++k) acc[k] = 0;
    for (int pass = 0; pass < (TWO ? 2 : 1); ++pass) {
      const Tin* base_in = pass ? in2 : in;
      const Acc* Wp = pass ? W2 : W;
      for (int i = 0; i < Di; ++i) {
        const Tin* src = base_in + ioff + i * si;
        for (int j0 = 0; j0 < (NJ > 0 ? NJ : Dj); j0 += U4) {
          Acc x[U4];
#pragma unroll
          for (int u = 0; u < U4; ++u) x[u] = (NJ > 0 || j0 + u < Dj) ? (Acc)src[(j0 + u) * sj] : (Acc)0;
#pragma unroll
          for (int u = 0; u < U4; ++u) {
            if (NJ == 0 && j0 + u >= Dj) break;
            const Acc* w = Wp + (i * Dj + j0 + u) * WS;
#pragma unroll
            for (int k = 0; k < CHI; ++k) acc[k] += w[k] * x[u];
          }
        }
      }
    }
#pragma unroll
    for (int k = 0; k < CHI; ++k) out[ooff + k * sk] = (Tout)acc[k];
  }
}

}  // namespace

// ============================================================================ launchers
void launch_init_tensor(double* T, long long inst_stride, int batch, int d, const double* beta,
                        const double* h, cudaStream_t s, int spin_insertion) {
  const int total = 1 << (2 * d);
  dim3 grid((total + 255) / 256, batch);
  k_init_tensor<<<grid, 256, 0, s>>>(T, inst_stride, d, beta, h, spin_insertion);
  count_launches(1);
}

void launch_step_advance(int* dstep, cudaStream_t s) {
  k_step_advance<<<1, 1, 0, s>>>(dstep);
  count_launches(1);
}

void launch_norm_log(const double* x, long long x_inst, int batch, long long n, double* partial, double* c_out,
                     double* lnc_log, long long log_inst, double* L, const int* dstep, int* status, cudaStream_t s) {
  k_sumsq_partial<<<dim3(kNormBlocks, batch), 256, 0, s>>>(x, x_inst, n, partial);
  count_launches(1);
  k_norm_finish<<<batch, 256, 0, s>>>(partial, c_out, lnc_log, log_inst, L, dstep, status);
  count_launches(1);
}

void launch_init_tangent(double* dT, long long inst_stride, int batch, int d, const double* beta, const double* h,
                         int which, cudaStream_t s) {
  const int total = 1 << (2 * d);
  k_init_tangent<<<dim3((total + 255) / 256, batch), 256, 0, s>>>(dT, inst_stride, d, beta, h, which);
  count_launches(1);
}

void launch_tangent_norm(const double* T, const double* D1, const double* D2, double* dTn, long long n,
                         const double* c, double* partial, double* dlnc, double* dL, const int* dstep,
                         cudaStream_t s) {
  k_dot_partial<<<kNormBlocks, 256, 0, s>>>(T, D1, D2, n, partial);
  count_launches(1);
  k_tangent_finish<<<1, 256, 0, s>>>(partial, c, dlnc, dL, dstep);
  count_launches(1);
  k_tangent_update<<<grid_for(n, 256), 256, 0, s>>>(T, D1, D2, dTn, n, c, dlnc);
  count_launches(1);
}

void launch_trace_tangent(const double* T, const double* dT, long long t_stride, int batch, long long P,
                          const double* dL, const int* dstep, double* out, cudaStream_t s) {
  k_trace_tangent<<<batch, 256, 0, s>>>(T, dT, t_stride, P, dL, dstep, out);
  count_launches(1);
}

void launch_trace_ratio(const double* S, const double* T, long long t_stride, int batch, long long P, double* out,
                        cudaStream_t s) {
  k_trace_ratio<<<batch, 256, 0, s>>>(S, T, t_stride, P, out);
  count_launches(1);
}

void launch_scale(const double* src, long long src_inst, double* dst, long long dst_inst, int batch, long long n,
                  const double* c, cudaStream_t s) {
  k_scale<<<dim3(grid_for(n, 256), batch), 256, 0, s>>>(src, src_inst, dst, dst_inst, n, c);
  count_launches(1);
}

void launch_trace_x(const double* T, long long t_stride, int batch, Geom g, int axis, const double* L,
                    const int* dstep, double* out3, cudaStream_t s) {
  k_trace_x<<<batch, 256, 0, s>>>(T, t_stride, g, axis, L, dstep, out3);
  count_launches(1);
}

template <class T>
void launch_absmax(const T* x, long long rows, long long cols, long long ld, unsigned* out, cudaStream_t s, int batch,
                   long long x_inst) {
  cudaMemsetAsync(out, 0, sizeof(unsigned) * batch, s);
  k_absmax<T><<<dim3(grid_for(rows * cols, 256), batch), 256, 0, s>>>(x, rows, cols, ld, out, x_inst);
  count_launches(1);
}
template void launch_absmax<float>(const float*, long long, long long, long long, unsigned*, cudaStream_t, int, long long);
template void launch_absmax<double>(const double*, long long, long long, long long, unsigned*, cudaStream_t, int,
                                    long long);

template <class Tout>
void launch_transpose(const double* T, long long t_inst, Tout* Tt, long long tt_inst, long long P, int ng,
                      cudaStream_t s) {
  dim3 grid((unsigned)((P + 31) / 32), (unsigned)((P + 31) / 32), (unsigned)ng);
  k_transpose<Tout><<<grid, dim3(32, 8), 0, s>>>(T, Tt, P, t_inst, tt_inst);
  count_launches(1);
}

template <class Tin, class Tout>
void launch_build_bt(const Tin* Tt, long long tt_inst, const Planes<Tout>& out, long long out_inst, long long ld, Geom g,
                     int c3, const double* U3, long long u_inst, int chi3, int ng, cudaStream_t s, const Tin* Tt2,
                     const double* U3b) {
  using Acc = AccT<Tout>;
  const long long Sc = c3 >= 0 ? g.Sn[c3] : 0;
  const int Dc = c3 >= 0 ? g.D[c3] : 1;
  const int nchi = c3 >= 0 ? chi3 : 1;
  const bool two = Tt2 && c3 >= 0;
  const size_t smem = sizeof(Acc) * (size_t)nchi * Dc * bt_row<Acc>(Dc) * (two ? 2 : 1);
  const long long total = g.P * g.P;
  const int jper = bt_rows_per_thread(total * ng, nchi);
  const dim3 grid(grid_for(total, 256), ng, (nchi + jper - 1) / jper);
  if (two)
    k_build_bt<Tin, Tout, true><<<grid, 256, smem, s>>>(Tt, out, ld, g.P, Sc, Dc, U3, nchi, Tt2, U3b, tt_inst, out_inst,
                                                        u_inst, jper);
  else
    k_build_bt<Tin, Tout, false><<<grid, 256, smem, s>>>(Tt, out, ld, g.P, Sc, Dc, c3 >= 0 ? U3 : nullptr, nchi, nullptr,
                                                         nullptr, tt_inst, out_inst, u_inst, jper);
  count_launches(1);
}

template <class Tin, class Tout>
void launch_build_y(const Tin* X, long long x_slot, const Planes<Tout>& out, long long out_slot, long long ld, Geom g,
                    int a, int nz, cudaStream_t s) {
  dim3 grid((unsigned)((g.P + 31) / 32), (unsigned)((g.P + 32 * kYMT - 1) / (32 * kYMT)), (unsigned)nz);
  k_build_y<Tin, Tout><<<grid, dim3(32, 8), 0, s>>>(X, out, ld, g, a, x_slot, out_slot);
  count_launches(1);
}

template <class Tin, class Tout>
void launch_pair_contract(const Tin* in, Tout* out, const View& v, int kaxis, int Di, int Dj,
                          long long si, long long sj, const double* U, int chi, long long in_base,
                          long long out_base, cudaStream_t s) {
  using Acc = AccT<Tout>;
  long long total = 1;
  for (int i = 0; i < v.ndim; ++i) total *= v.shape[i];
  const int nchi = U ? chi : 1;
  const size_t smem = sizeof(Acc) * (size_t)nchi * Di * Dj;
  k_pair_contract<Tin, Tout><<<grid_for(total, 256), 256, smem, s>>>(in, out, v, total, kaxis, Di, Dj,
                                                                      si, sj, U, nchi, in_base, out_base);
  count_launches(1);
}

template <class Tin, class Tout, bool TWO, int CHI, int NJ>
static void pair_contract_all(const Tin* in, Tout* out, const View& rest, int Di, int Dj, long long si, long long sj,
                              long long sk, const double* U, long long out_base, const SlotStrides& st, cudaStream_t s,
                              const Tin* in2, const double* U2) {
  using Acc = AccT<Tout>;
  constexpr int PAD = 16 / (int)sizeof(Acc);
  // axes that run on from one another in both tensors become one: the index of an output costs a division an axis
  View v;
  v.ndim = 0;
  long long total = 1;
  for (int i = 0; i < rest.ndim; ++i) {
    total *= rest.shape[i];
    if (rest.shape[i] == 1) continue;
    const int l = v.ndim - 1;
    if (l >= 0 && v.in_stride[l] == rest.in_stride[i] * rest.shape[i] &&
        v.out_stride[l] == rest.out_stride[i] * rest.shape[i] && (long long)v.shape[l] * rest.shape[i] < (1LL << 31)) {
      v.shape[l] *= rest.shape[i];
    } else {
      ++v.ndim;
      v.shape[l + 1] = rest.shape[i];
    }
    v.in_stride[v.ndim - 1] = rest.in_stride[i];
    v.out_stride[v.ndim - 1] = rest.out_stride[i];
  }
  const size_t smem = sizeof(Acc) * (size_t)((CHI + PAD - 1) / PAD * PAD) * Di * Dj * (TWO ? 2 : 1);
  k_pair_contract_all<Tin, Tout, TWO, CHI, NJ><<<dim3(grid_for(total, 256), st.nb, st.ng), 256, smem, s>>>(
      in, out, v, total, Di, Dj, si, sj, sk, U, out_base, in2, U2, st);
  count_launches(1);
}

template <class Tin, class Tout>
void launch_pair_contract_all(const Tin* in, Tout* out, const View& rest, int Di, int Dj, long long si,
                              long long sj, long long sk, const double* U, int chi, long long out_base,
                              const SlotStrides& st, cudaStream_t s, const Tin* in2, const double* U2) {
  switch (chi) {
#define HOTRG_PCA(C)                                                                                               \
  case C:                                                                                                          \
    if (in2)                                                                                                       \
      pair_contract_all<Tin, Tout, true, C, 0>(in, out, rest, Di, Dj, si, sj, sk, U, out_base, st, s, in2, U2);      \
    else if (std::is_same<Tin, float>::value && C >= 6 && Dj == C)                                                 \
      pair_contract_all<Tin, Tout, false, C, std::is_same<Tin, float>::value && C >= 6 ? C : 0>(                   \
          in, out, rest, Di, Dj, si, sj, sk, U, out_base, st, s, nullptr, nullptr);                                \
    else                                                                                                           \
      pair_contract_all<Tin, Tout, false, C, 0>(in, out, rest, Di, Dj, si, sj, sk, U, out_base, st, s, nullptr,      \
                                                nullptr);                                                          \
    return;
    HOTRG_PCA(1) HOTRG_PCA(2) HOTRG_PCA(3) HOTRG_PCA(4) HOTRG_PCA(5) HOTRG_PCA(6) HOTRG_PCA(7) HOTRG_PCA(8)
    HOTRG_PCA(9) HOTRG_PCA(10) HOTRG_PCA(11) HOTRG_PCA(12) HOTRG_PCA(13) HOTRG_PCA(14) HOTRG_PCA(15) HOTRG_PCA(16)
#undef HOTRG_PCA
    default:
      return;
  }
}

// The two-input contractions and B-operand builds in FP64 can need more than the default 48 KB
// of dynamic shared memory (2 x 16 x 256 doubles): raise the limit once, outside any capture.
template <class Tin, class Tout>
static void raise_two_input_limit(int big) {
#define HOTRG_PCA_ATTR(C) \
  cudaFuncSetAttribute(k_pair_contract_all<Tin, Tout, true, C, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
  HOTRG_PCA_ATTR(12) HOTRG_PCA_ATTR(13) HOTRG_PCA_ATTR(14) HOTRG_PCA_ATTR(15) HOTRG_PCA_ATTR(16)
#undef HOTRG_PCA_ATTR
}

void prepare_kernel_attributes() {
  // 2 x round_up(chi, 2) x Di Dj doubles: above 48 KB from chi = 12 on (12 x 256 x 2 x 8 bytes = 48 KB)
  const int big = (int)(2 * sizeof(double) * kMaxBond * kMaxGram);
  raise_two_input_limit<double, double>(big);
  raise_two_input_limit<float, float>(big);
  raise_two_input_limit<float, double>(big);
  cudaFuncSetAttribute(k_build_bt<double, double, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
  cudaFuncSetAttribute(k_build_bt<float, __nv_bfloat16, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
}

// explicit instantiations: FP64 path (double everywhere) and BF16X3 path (float intermediates)
template void launch_transpose<double>(const double*, long long, double*, long long, long long, int, cudaStream_t);
template void launch_transpose<float>(const double*, long long, float*, long long, long long, int, cudaStream_t);
#define HOTRG_BT(TI, TO)                                                                                          \
  template void launch_build_bt<TI, TO>(const TI*, long long, const Planes<TO>&, long long, long long, Geom, int,   \
                                        const double*, long long, int, int, cudaStream_t, const TI*, const double*);
HOTRG_BT(double, double)
HOTRG_BT(float, __nv_bfloat16)
#undef HOTRG_BT
#define HOTRG_Y(TI, TO)                                                                                               \
  template void launch_build_y<TI, TO>(const TI*, long long, const Planes<TO>&, long long, long long, Geom, int, int, \
                                       cudaStream_t);
HOTRG_Y(double, double)
HOTRG_Y(float, __nv_bfloat16)
HOTRG_Y(double, __nv_bfloat16)
#undef HOTRG_Y
template void launch_pair_contract<double, double>(const double*, double*, const View&, int, int, int, long long, long long, const double*, int, long long, long long, cudaStream_t);
template void launch_pair_contract<float, float>(const float*, float*, const View&, int, int, int, long long, long long, const double*, int, long long, long long, cudaStream_t);
template void launch_pair_contract<float, double>(const float*, double*, const View&, int, int, int, long long, long long, const double*, int, long long, long long, cudaStream_t);
#define HOTRG_PCA(TI, TO)                                                                                              \
  template void launch_pair_contract_all<TI, TO>(const TI*, TO*, const View&, int, int, long long, long long, long long, \
                                                 const double*, int, long long, const SlotStrides&, cudaStream_t,       \
                                                 const TI*, const double*);
HOTRG_PCA(double, double)
HOTRG_PCA(float, float)
HOTRG_PCA(float, double)
#undef HOTRG_PCA

}  // namespace hotrg
