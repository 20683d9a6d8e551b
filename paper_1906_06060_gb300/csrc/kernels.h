// Host-side launchers of the libhotrg kernels. All launch on the given stream and return
// immediately; errors surface through cudaGetLastError() and the device status word.
#pragma once
#include "common.cuh"

namespace hotrg {

// Number of kernels the launchers below have enqueued in this process (diagnostics: lets a
// caller count the library's launches inside a timed region).
void count_launches(int n);
long long launches_total();

// ---- kernels_tensor.cu --------------------------------------------------------------------
// T^(0) (Sec. 2) for `batch` instances: T + i*stride gets beta[i], h[i] (device arrays). With
// spin_insertion, the impure tensor S^(0) (the summand carries the spin s).
void launch_init_tensor(double* T, long long inst_stride, int batch, int d, const double* beta,
                        const double* h, cudaStream_t s, int spin_insertion = 0);
// *dstep += 1 (device-side step counter read by the kernels below, so that a captured step
// can be replayed for any step number).
void launch_step_advance(int* dstep, cudaStream_t s);
// For `batch` tensors x + i x_inst: c = ||x||_F (deterministic) into c_out[i], lnc_log[i log_inst + n] = ln c, L[i] +=
// 2^-n ln c with n = *dstep; status on a bad norm. partial: 1024 doubles per tensor.
void launch_norm_log(const double* x, long long x_inst, int batch, long long n, double* partial, double* c_out,
                     double* lnc_log, long long log_inst, double* L, const int* dstep, int* status, cudaStream_t s);
// Tangents of the flow (fixed isometries). dT = d T^(0) / d beta (which = 0) or d / d h (which = 1).
void launch_init_tangent(double* dT, long long inst_stride, int batch, int d, const double* beta, const double* h,
                         int which, cudaStream_t s);
// For an unnormalised tensor T with norm *c and tangent D = D1 + D2 (D2 may be null):
// dlnc = <T, D> / c^2, dL += 2^-n dlnc (n = *dstep), dTn = (D - dlnc T) / c (tangent of T / c).
void launch_tangent_norm(const double* T, const double* D1, const double* D2, double* dTn, long long n,
                         const double* c, double* partial, double* dlnc, double* dL, const int* dstep,
                         cudaStream_t s);
// out[i] = dL[i] + 2^-n Tr dT_i / Tr T_i for every instance.
void launch_trace_tangent(const double* T, const double* dT, long long t_stride, int batch, long long P,
                          const double* dL, const int* dstep, double* out, cudaStream_t s);
// out[i] = Tr S_i / Tr T_i (Eqs. (energy), (spin)) for every instance.
void launch_trace_ratio(const double* S, const double* T, long long t_stride, int batch, long long P, double* out,
                        cudaStream_t s);
// *out = max |x| over a rows x cols array with row stride ld (upper bound as a float; the bits
// of that non-negative float are written, after zeroing *out on the stream).
// `batch` arrays x + i x_inst, out[i].
template <class T>
void launch_absmax(const T* x, long long rows, long long cols, long long ld, unsigned* out, cudaStream_t s,
                   int batch = 1, long long x_inst = 0);
// dst + i dst_inst = (src + i src_inst) / c[i], i < batch
void launch_scale(const double* src, long long src_inst, double* dst, long long dst_inst, int batch, long long n,
                  const double* c, cudaStream_t s);
// Tr T (Eq. (tTr)) and ln Z/N = L + 2^-n ln Tr (n = *dstep); X^(n) along `axis` (Eq. (x)).
// One CTA per instance: T + i*t_stride, L + i, out3 + 3 i.
void launch_trace_x(const double* T, long long t_stride, int batch, Geom g, int axis, const double* L,
                    const int* dstep, double* out3, cudaStream_t s);
// The launchers below cover ng instances (and, per instance, nb chunks of a squeeze) in one launch: instance j reads at
// j x its instance stride, slot z = j nb + chunk at z x its slot stride (elements). See squeeze() in hotrg.cu.

// For chunk c of instance j: out_z[..u_b=j..] = sum_i U_j[kk + c][i][j] in_j[..u_b=i..] on unprimed leg b (U: [chi][Db][Db]
// fp64); with in2 (one instance), plus the same product of in2 with U2. With amax, amax[z] = max |out_z| (the bits of a
// non-negative float, as launch_absmax writes them).
template <class Tin, class Tout>
void launch_mode_unprimed(const Tin* in, long long in_inst, Tout* out, long long out_slot, Geom g, int b, const double* U,
                          long long u_inst, int kk, int ng, int nb, cudaStream_t s, const Tin* in2 = nullptr,
                          const double* U2 = nullptr, unsigned* amax = nullptr);
// Tt_j[p][u] = T_j[u][p] (P x P), converted to Tout.
template <class Tout>
void launch_transpose(const double* T, long long t_inst, Tout* Tt, long long tt_inst, long long P, int ng, cudaStream_t s);
// B operand, K-major: Bt[(j*P + n)][k] = sum_x U3[j][k_c3][x] Tt[n][k | c3 := x], j < chi3.
// c3 < 0: Bt = Tt. Mixed: 2 or 3 16-bit planes (instance i's scale bound at amax + i); FP64: one double plane. With Tt2
// (c3 >= 0, one instance), plus the same sum over Tt2 with U3b.
template <class Tin, class Tout>
void launch_build_bt(const Tin* Tt, long long tt_inst, const Planes<Tout>& out, long long out_inst, long long ld, Geom g,
                     int c3, const double* U3, long long u_inst, int chi3, int ng, cudaStream_t s,
                     const Tin* Tt2 = nullptr, const double* U3b = nullptr);
// A operand of slot z, K-major: Y[m][k] = X[u = (k_b, m_a)][p = (m_b, k_a)] for a step along `a` (scale bound at
// amax + z).
template <class Tin, class Tout>
void launch_build_y(const Tin* X, long long x_slot, const Planes<Tout>& out, long long out_slot, long long ld, Geom g,
                    int a, int nz, cudaStream_t s);
// Strided copy (see View).
template <class Tin, class Tout>
void launch_pair_contract(const Tin* in, Tout* out, const View& v, int kaxis, int Di, int Dj,
                          long long si, long long sj, const double* U, int chi, long long in_base,
                          long long out_base, cudaStream_t s);
// The slots of an epilogue contraction: slot z = j nb + c reads at z in_slot and writes at j out_inst + c out_chunk with
// the isometry at j u_inst.
struct SlotStrides {
  int ng, nb;
  long long in_slot, out_inst, out_chunk, u_inst;
};
// Pair contraction out[o] = sum_{i,j} U[k'][i][j] in[...], one thread per index of `rest` (the output axes without k'),
// computing all chi outputs out[o + k' sk]; every input element is read once. With in2 (same layout), plus the same
// contraction of in2 with U2.
template <class Tin, class Tout>
void launch_pair_contract_all(const Tin* in, Tout* out, const View& rest, int Di, int Dj, long long si,
                              long long sj, long long sk, const double* U, int chi, long long out_base,
                              const SlotStrides& st, cudaStream_t s, const Tin* in2 = nullptr,
                              const double* U2 = nullptr);
// Raise the dynamic shared-memory limit of the two-input kernels (call once, before any capture).
void prepare_kernel_attributes();

// ---- gram.cu -------------------------------------------------------------------------------
// Q[(i,al)][(i~,al~)] = sum over all other legs of T[..i..al..] T[..i~..al~..]; legs l1, l2 are
// positions 0..2d-1 in the natural layout. partial: scratch of partial_doubles; the sum over the columns runs in as many
// splits (batch nr^2 doubles each) as it holds, at most those that gram_partial_doubles provides for.
// Instance i reads T + i*t_stride and writes Q + i*q_stride.
size_t gram_partial_doubles(int nr_max, int batch);  // scratch for `partial`
// With TA: rows from TA (same layout and strides as T), columns from T: Q(TA, T).
// With z2ev ([batch][kMaxD] even-value counts, values ordered even-parity first), the zero-field
// block structure is used: a quarter of the work (see gram.cu).
void launch_half_gram(const double* T, long long t_stride, int batch, Geom g, int l1, int l2,
                      double* partial, size_t partial_doubles, double* Q, long long q_stride, cudaStream_t s,
                      const double* TA = nullptr, const int* z2ev = nullptr);
// G[(b1 b2)][(b1~ b2~)] = sum_{al,al~} Q1[(b1,al)][(b1~,al~)] Q2[(b2,al)][(b2~,al~)] per instance
void launch_gram_combine(const double* Q1, const double* Q2, long long q_stride, int batch, int Db,
                         int Da, double* G, long long g_stride, cudaStream_t s);
// dG = sum (H1 + H1^T) Q2 + Q1 (H2 + H2^T), H = Q(dT, T): the tangent of the Gram matrix.
void launch_gram_combine_tangent(const double* Q1, const double* Q2, const double* H1, const double* H2,
                                 long long q_stride, int batch, int Db, int Da, double* dG, long long g_stride,
                                 cudaStream_t s);

// ---- eig.cu --------------------------------------------------------------------------------
// Where the sorted eigenvalues go: base + i*inst_stride + (*step - 1)*step_stride for instance
// i (nothing is written when the step is outside 1..max_steps).
struct EigOut {
  double* base;
  long long inst_stride, step_stride;
  const int* step;
  int max_steps;
};
// Symmetric eigendecomposition of G (n x n, n <= 256) by cyclic Jacobi, one cluster of up to 16 CTAs per instance;
// eigenvalues sorted descending, the leading chi eigenvectors, sign-fixed, into U[k][0..n).
// work: batch * 2*n*n doubles. Sets ST_NOCONV on the sweep limit.
// Several axes in one launch (blockIdx.y = axis): per axis its Gram matrices G (+ instance x
// g_stride), size n, kept count chi, the axis and Db for the zero-field ordering, the eigenvalue
// log base (+ instance x out.inst_stride + (step - 1) x out.step_stride), U (+ instance x u_stride)
// and a work area of batch x 2 n^2 doubles.
struct EigAxis {
  const double* G;
  int n, chi, z2_axis, Db;
  double* evals;
  double* U;
  double* work;
};
struct EigAxes {
  int nt;
  int max_sweeps;  // sweep limit (ST_NOCONV when reached)
  long long g_stride, u_stride;
  EigOut out;  // strides, step counter and step limit (its base is unused here)
  EigAxis ax[kMaxD];
};
void launch_eig_axes(const EigAxes& ea, int batch, int* status, cudaStream_t s, const int* z2_ev = nullptr,
                     int* z2_ev_new = nullptr);
// z2_ev (non-null): zero-field flow: [batch][kMaxD] even counts of the legs; the kept vectors of
// axis z2_axis (Db x Db fused index) are written even-parity first (each group in descending
// eigenvalue order), z2_ev_new[i][z2_axis] = number of even ones; a vector that is not
// parity-pure sets ST_Z2.
void launch_eig(const double* G, long long g_stride, int batch, int n, int chi, const EigOut& o,
                double* U, long long u_stride, double* work, int* status, cudaStream_t s,
                const int* z2_ev = nullptr, int* z2_ev_new = nullptr, int z2_axis = 0, int Db = 0,
                int max_sweeps = 40);
// First-order change of the kept eigenvectors for a change dG of G, from the eigensystem that
// launch_eig left in `work` (call before the next launch_eig reuses it):
//   dU_k = sign_k sum_{j >= chi} V_j (V_j^T dG V_k) / (lambda_k - lambda_j),  k < chi,
// with sign_k the sign convention applied to U_k. Rotations inside the kept space are left out:
// they are a gauge change of the new bond under which the flow's ln Z is invariant. A cut with
// lambda_k == lambda_j (k < chi <= j) has no derivative: dU gets NaN.
void launch_eig_tangent(const double* work, const double* U, long long u_stride, const double* dG,
                        long long g_stride, int batch, int n, int chi, double* dU, cudaStream_t s);
void prepare_eig_attributes();  // shared-memory limit of the tangent kernel (once, before any capture)

// ---- gemm_simt.cu --------------------------------------------------------------------------
// C[m][n] = sum_k A[m][k] Bt[n][k] in FP64 (CUDA cores).
// With blk (device memory, see GemmBlocks below), only the listed output blocks are computed, each
// over its own k range; M, N are then the extents of A's and Bt's rows.
// With bat (a batched launch, see GemmBatch), `batch` such products, instance i at A + i a_inst,
// Bt + i b_inst, C + i c_inst with blocks blk[i].
struct GemmBlocks;
struct GemmBatch;
void launch_gemm_f64(const double* A, long long lda, const double* Bt, long long ldb, double* C,
                     long long ldc, long long M, long long N, long long K, cudaStream_t s,
                     const GemmBlocks* blk = nullptr, const GemmBatch* bat = nullptr);

// ---- gemm_f64tc.cu --------------------------------------------------------------------------
// FP64 products on the tensor cores from exact integer slices. An operand: kSliceCount planes of fp16 digits (`plane`
// elements apart, rows of `ld`, instances `inst` apart) and the exponent of every row (instances exp_inst apart).
constexpr int kSliceCount = 8;
constexpr int kSliceProducts = kSliceCount * (kSliceCount + 1) / 2;  // digit pairs a product runs
constexpr int kSliceCtas = 152;  // CTAs of a launch at most (one per SM): the scratch area is sized for them
struct SliceOperand {
  __half* p = nullptr;
  long long ld = 0, plane = 0, inst = 0;
  int* exps = nullptr;
  long long exp_inst = 0;
};
// Whether a product of this shape can run on slices: at least one 128 x 256 tile and K up to 16320 (the int32 sums).
bool slices_take(long long M, long long N, long long K);
// Bytes of the level-sum scratch of a launch over `batch` products of at most M x N.
size_t slice_scratch_bytes(long long M, long long N, int batch);
struct Z2Layout;
// Column scales of a product, from its Bt (`rows` x K doubles, row stride ldx; `batch` instances x_inst apart):
// fields[k] = max(fields[k], largest exponent field in column k), instances f_inst apart, zeroed by the caller. With L
// (zero-field operands) only the entries of the parity classes.
void launch_column_fields(const double* X, long long ldx, long long rows, long long K, int* fields, long long f_inst,
                          int batch, long long x_inst, cudaStream_t s, const Z2Layout* L = nullptr);
// Digits and row exponents of `rows` x K doubles (row stride ldx; `batch` slots x_inst apart) with the column scales of
// slot z's instance z / nb. side: -1 for Bt, 1 for A. With L (zero-field operands: instance z / nb's layout, slot z's
// chunk parity) only the columns of each row's parity class, see k_slice_rows.
void launch_slice_rows(const double* X, long long ldx, long long rows, long long K, const SliceOperand& out, int batch,
                       long long x_inst, const int* fields, long long f_inst, int side, cudaStream_t s, int nb = 1,
                       const Z2Layout* L = nullptr, const int* pi = nullptr);
// C[m][n] (+)= sum_k A[m][k] Bt[n][k]; blk and bat as for launch_gemm_f64. cta_group: 1 or 2 CTAs per tile (the same
// results), 0: by shape. stall (test of the bounded waits): bit r: CTA r of a pair (or the CTA of a tile) issues no copies.
// Returns 0 or a hotrg_status.
int launch_gemm_slices(const SliceOperand& A, const SliceOperand& B, double* C, long long ldc, long long M, long long N,
                       long long K, int* scratch, int* status, double timeout_s, cudaStream_t s,
                       const GemmBlocks* blk = nullptr, const GemmBatch* bat = nullptr, bool accumulate = false,
                       int cta_group = 0, int stall = 0);

// ---- gemm_tc.cu ----------------------------------------------------------------------------
// C[m][n] = sum over passes p of sum_k A_{a(p)}[m][k] Bt_{b(p)}[n][k], bf16 operand planes on
// tcgen05, FP32 accumulation in TMEM. npass = 1: (hi,hi); 3: + (hi,lo), (lo,hi) with 2 planes;
// 4: + (lo,lo); 6: (hi,hi), (hi,mid), (mid,hi), (hi,lo), (mid,mid), (lo,hi) with 3 planes.
// bk = 64 or 32: the k-block width (the accumulator restarts and is folded once per k-block);
// group_m: output tiles are visited in groups of group_m M-tiles (L2 reuse); fold_group: k-blocks
// per accumulator fold (at most ring stages - 1 when > 1).
// Returns 0 or a hotrg_status (tensor-map encode failure, bad alignment or sizes).
// Block-sparse form (blk != null, device memory read by the kernel at start): only the output
// blocks listed are computed. Block b: rows [m0, m0+mc) of A and C, rows [n0, n0+nc) of Bt
// (columns of C), k range [k0, k0+kc), where both operands must hold zeros from k0+kc up to the
// next multiple of bk. M, N, K are then the operands' extents (rows of A, rows of Bt, row
// length) and bound every copy; nothing outside the blocks is written.
struct GemmBlocks {
  int nb;
  int m0[2], mc[2], n0[2], nc[2], k0[2], kc[2];
};
// Largest number of instances one batched GEMM launch takes (its tile prefix lives in shared memory).
constexpr int kMaxGemmBatch = 256;
// Batched launch (up to kMaxGemmBatch instances): `batch` independent products of the same shape in one
// persistent launch; plane k of instance i starts at A.p[k] + i a_inst (elements, multiple of 8,
// at least M lda), likewise C (c_inst) and, by b_div, B (b_inst); with blk, instance i's blocks are blk[i];
// fp16 scale bounds at A.amax + i and B.amax + i / b_div. Products i / b_div with the same value share one B operand (the
// chunks of an instance): B of product i is at (i / b_div) b_inst.
struct GemmBatch {
  int batch = 1, b_div = 1;
  long long a_inst = 0, b_inst = 0, c_inst = 0;
};
int launch_gemm_split(const Planes<__nv_bfloat16>& A, long long lda, const Planes<__nv_bfloat16>& B,
                      long long ldb, float* C, long long ldc, long long M, long long N, long long K,
                      int npass, int* status, double timeout_s, cudaStream_t s, int bk = 64,
                      int group_m = 16, int fold_group = 1, const GemmBlocks* blk = nullptr,
                      const GemmBatch* bat = nullptr, bool stall = false, int cta_group = 0);
// stall (test of the bounded waits): the kernel's producer issues no copies, so every CTA's first
// wait for a stage runs out after timeout_s and the launch ends with ST_TIMEOUT in *status.
// cta_group: 1 = one CTA per 128 x 256 output tile, 2 = a CTA pair (cluster of two) per 256 x 256
// tile with tcgen05 cta_group::2 MMAs, each CTA staging half the B rows; 0 = pairs from 129 rows on (the faster form at every
// measured shape: 8^4 chunks 1555 against 1929 us, 7^4 329 against 402, 10^4 28.9 against 34.4 ms, 5^4 43 against 45 us).
// Largest fold group the kernel variant for (npass, bk) accepts.
int max_fold_group(int npass, int bk);
void launch_split_rows(const float* X, long long ldx, long long rows, long long cols,
                       const Planes<__nv_bfloat16>& out, long long ld, cudaStream_t s);

// ---- z2.cu ---------------------------------------------------------------------------------
// Parity-blocked layout of the zero-field squeeze's operands for one instance (see z2.cu).
struct Z2Layout {
  int d;
  int D[kMaxD], e[kMaxD];      // bond dimensions and even-value counts of the current legs
  int ncls[2];                 // natural P-indices of even / odd total parity
  int kstart[2];               // operand column where each parity class starts (64-aligned)
  int patoff[16];              // rank of the first index of each leg-parity pattern
  int bs[16][kMaxD];           // row-major strides inside each pattern's box
  int chi3, e3;                // the new c3 index: range and number of even values
  int goff[2];                 // first output column of each group (parity of (j, n))
  int jstart[2][kMaxBond + 1]; // offset of new index j inside each group
};
// Layouts of every instance (ev, ev_new: [batch][kMaxD] even counts before / after the step).
void launch_z2_layout(const int* ev, const int* ev_new, int batch, Geom g, int c3, int chi3, Z2Layout* out,
                      cudaStream_t s);
// Index tables of ng instances: rank[P], kcol[P] (instance stride p_inst) and colpos[chi3 * P] (stride c_inst).
struct Z2Tables {
  int *rank, *kcol, *colpos;
  long long p_inst, c_inst;
  Z2Tables from(int j) const { return {rank + j * p_inst, kcol + j * p_inst, colpos + j * c_inst, p_inst, c_inst}; }
};
void launch_z2_tables(const Z2Layout* L, long long P, int chi3, const Z2Tables& t, int ng, cudaStream_t s);
// For every slot z = j nb + c: the chunk's parity pi[z] (new indices k0 of axis b0 and k1 of b1 fixed, nfix of them, the
// last of them advanced by c; ev_new: [ng][kMaxD]) and its two GEMM blocks blk[z]; flops[0] += their 2 M N K, flops[1] +=
// that times npass.
void launch_z2_chunk(const Z2Layout* L, const int* ev_new, int ng, int nb, int nfix, int b0, int k0, int b1, int k1,
                     long long N, GemmBlocks* blk, int* pi, double* flops, int npass, cudaStream_t s);
// ev[i][b] = ev_new[i][b] for the axes b in trans_mask (end of a step).
void launch_z2_advance(int* ev, const int* ev_new, int batch, unsigned trans_mask, cudaStream_t s);
template <class Tin, class Tout>
void launch_build_y_z2(const Tin* X, long long x_slot, const Planes<Tout>& out, long long out_slot, long long ld, Geom g,
                       int a, const Z2Tables& t, const Z2Layout* L, const int* pi, int ng, int nb, cudaStream_t s);
template <class Tin, class Tout>
void launch_build_bt_z2(const Tin* Tt, long long tt_inst, const Planes<Tout>& out, long long out_inst, long long ld, Geom g,
                        int c3, const double* U3, long long u_inst, int chi3, const Z2Tables& t, const Z2Layout* L, int ng,
                        cudaStream_t s);
// First epilogue contraction (over slot t0, Dt x Dt -> chi) from the parity-blocked GEMM output;
// rest / sk / out_base / st as for launch_pair_contract_all (instance j's layout L + j, slot z's parity pi + z).
template <class Tin, class Tout>
void launch_epi_z2(const Tin* O, long long ldO, Tout* out, const View& rest, long long sk, long long out_base, int t0,
                   int Dt, const double* U, int chi, const Z2Layout* L, const int* pi, const SlotStrides& st,
                   cudaStream_t s);

}  // namespace hotrg
