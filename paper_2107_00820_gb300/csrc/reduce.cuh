// Single-launch, bitwise-reproducible reductions and the one-thread GMRES
// bookkeeping that runs in the epilogue of the last block of a reduction.
//
// Every block writes the partial sums of its columns to a workspace row, takes
// a ticket from a counter, and the block holding the last ticket adds the
// partials of all blocks in a fixed order (so the result does not depend on
// which block finished last) and resets the counter.  Workspace layout: slot 0
// is the counter, the partials [block][column] start at slot 1.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

#include "df64.cuh"

namespace als {

constexpr int RED_THREADS = 256;
constexpr int RED_MAX_BLOCKS = 1216;   // 8 x 152 SMs: one full wave at 256 threads per block
constexpr int KMAXB = 8;               // columns reduced together in registers

// blocks for a reduction over n entries: about `per_thread` entries per thread
inline unsigned red_blocks(long long n, int per_thread = 4) {
  long long b = (n + (long long)RED_THREADS * per_thread - 1) / ((long long)RED_THREADS * per_thread);
  if (b > RED_MAX_BLOCKS) b = RED_MAX_BLOCKS;
  if (b < 1) b = 1;
  return (unsigned)b;
}

// a warp's sums of P columns: lane l returns that of column l mod P.  The columns are halved as
// the lanes are paired (a lane passes on the half that its partner keeps), P - 1 + log2(32 / P)
// additions instead of 5 P.
template <int P, typename T>
__device__ __forceinline__ T warp_totals(const T (&acc)[KMAXB]) {
  const int lane = threadIdx.x & 31;
  T v[P];
#pragma unroll
  for (int j = 0; j < P; ++j) v[j] = acc[j];
#pragma unroll
  for (int w = P / 2; w > 0; w >>= 1) {
    const bool up = (lane & w) != 0;
#pragma unroll
    for (int j = 0; j < w; ++j) {
      const T give = up ? v[j] : v[j + w];
      v[j] = (up ? v[j + w] : v[j]) + __shfl_xor_sync(0xffffffffu, give, w);
    }
  }
#pragma unroll
  for (int o = P; o < 32; o <<= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  return v[0];
}

// Sum of kk <= KMAXB columns over a block, returned to thread j < kk (the others' value is
// unspecified).  The caller puts a barrier between the return and the next use of sh.  Few
// instructions above all for FP64, where a warp's takes 64 cycles of its scheduler: with a shuffle
// tree per column and a serial sum over the warps the sums of four columns took 28 additions, 9 now.
template <typename T>
__device__ __forceinline__ T block_total(const T (&acc)[KMAXB], int kk, T (&sh)[RED_THREADS / 32][KMAXB]) {
  static_assert(RED_THREADS == 256 && KMAXB == 8, "a warp adds 8 rows of 8 columns");
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const T v = kk == 1 ? warp_totals<1>(acc) : kk == 2 ? warp_totals<2>(acc) : kk <= 4 ? warp_totals<4>(acc) : warp_totals<8>(acc);
  if (lane < kk) sh[w][lane] = v;
  __syncthreads();
  T t = T(0);
  if (w == 0) {
    const int c = lane & 7, r = lane >> 3;
    if (c < kk) t = sh[r][c] + sh[r + 4][c];
    t += __shfl_xor_sync(0xffffffffu, t, 8);
    t += __shfl_xor_sync(0xffffffffu, t, 16);
  }
  return t;
}

// block partials of kk <= KMAXB columns, written to row[0..kk) and fenced
__device__ __forceinline__ void block_partials(const double (&acc)[KMAXB], int kk, double* row) {
  __shared__ double sh[RED_THREADS / 32][KMAXB];
  const double v = block_total<double>(acc, kk, sh);
  if ((int)threadIdx.x < kk) {
    row[threadIdx.x] = v;
    __threadfence();   // the writers publish their partial before the block takes its ticket
  }
  __syncthreads();
}

// called right after block_partials (whose writers fenced their partials)
__device__ __forceinline__ bool last_block(double* ws) {
  __shared__ bool is_last;
  if (threadIdx.x == 0) is_last = atomicAdd(reinterpret_cast<unsigned int*>(ws), 1u) == gridDim.x - 1;
  __syncthreads();
  return is_last;
}

// Run by every thread of the last block: out[j] = sum over blocks of column j.  The partials (rows
// from ws + 1) are read through L2 (other blocks wrote them), each thread over a fixed
// strided subset, then one fixed block reduction per group of KMAXB columns.
__device__ __forceinline__ void finish_sums(double* ws, int k, double* out) {
  __shared__ double sh[RED_THREADS / 32][KMAXB];
  if (threadIdx.x == 0) __threadfence();
  __syncthreads();
  const double* partial = ws + 1;
  for (int j0 = 0; j0 < k; j0 += KMAXB) {
    const int kk = (k - j0) < KMAXB ? (k - j0) : KMAXB;
    double acc[KMAXB];
#pragma unroll
    for (int j = 0; j < KMAXB; ++j) acc[j] = 0.0;
#pragma unroll 4
    for (int b = threadIdx.x; b < (int)gridDim.x; b += RED_THREADS) {
#pragma unroll
      for (int j = 0; j < KMAXB; ++j)
        if (j < kk) acc[j] += __ldcg(partial + (long long)b * k + j0 + j);
    }
    const double v = block_total<double>(acc, kk, sh);
    if ((int)threadIdx.x < kk) out[j0 + threadIdx.x] = v;
    __syncthreads();
  }
  if (threadIdx.x == 0) *reinterpret_cast<unsigned int*>(ws) = 0u;
}

// acc[j] += the thread's share (blocks tid, tid + 256, ..) of column j of nb block partials
template <typename T>
__device__ __forceinline__ void sum_rows(const T* __restrict__ rows, int nb, int k, T (&acc)[KMAXB]) {
#pragma unroll
  for (int j = 0; j < KMAXB; ++j) acc[j] = T(0);
#pragma unroll 4
  for (int b = threadIdx.x; b < nb; b += RED_THREADS) {
#pragma unroll
    for (int j = 0; j < KMAXB; ++j)
      if (j < k) acc[j] += __ldcg(rows + j * nb + b);
  }
}

// ---------------------------------------------------------------------------
// GMRES(s) state on the device, in S = small_t<T> for a smoother of precision T (column-major
// Hessenberg H, leading dim ldh): FP64, or, for an FP32 smoother, double-float.  The least-squares
// problem of a smoothing amplifies a change of its small numbers into the iterate, as it does the roundings
// of the vectors.  Relative error of one FP32 96^2 five-level cycle (gamma 100, contrast 1e6, P2) against FP64
// over 240 problems, median and 90th percentile: 3.1e-7 and 5.8e-7 with the state, the coefficients and the
// combinations of columns in plain FP32, 2.2e-7 and 3.1e-7 so (with the cells' differences to their middle
// node and the node sums of the tiles, apply_cells.cuh and arnoldi2.cuh, which are part of that).  One
// cycle, us, plain / so: 2D 16^2 96 / 105, 128^2 333 / 354, order 3 1013 / 1028, 3D 32^3 1643 / 1657.
// The Krylov basis is stored unnormalised:
// column i holds hn_i v_i, where v_i is the orthonormal Arnoldi vector, and
// Z_i = D^-1 (column i) likewise; their consumers multiply by rhn[i] = 1 / hn_i, and rr[i] = 1 / R_ii
// (both 0 where the divisor is): the divisions are done once, by the bookkeeping block beside
// the vector work, and none but those of the last step is left for the update.
// Layout of the state array, in elements of S (eight bytes either way):
// H [ldh s] | cs [s] | sn [s] | g [s+1] | y [s] | res | beta | nrm2 | rhn [s+1] | rr [s].
// ---------------------------------------------------------------------------
template <typename T> struct SmallReal { using S = double; };
template <> struct SmallReal<float> { using S = DF64; };
template <typename T> using small_t = typename SmallReal<T>::S;

__device__ __forceinline__ double to_small(double v) { return v; }
__device__ __forceinline__ DF64 to_small(float v) { return DF64{v, 0.f}; }
__device__ __forceinline__ double load_small(const double* p) { return __ldcg(p); }
__device__ __forceinline__ DF64 load_small(const DF64* p) {
  const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
  return DF64{v.x, v.y};
}
__device__ __forceinline__ double shfl_small(double v, int l) { return __shfl_sync(0xffffffffu, v, l); }
__device__ __forceinline__ DF64 shfl_small(DF64 v, int l) {
  return DF64{__shfl_sync(0xffffffffu, v.hi, l), __shfl_sync(0xffffffffu, v.lo, l)};
}
// 1 / a, or 0 where a is 0 or so small that 1 / a overflows (no direction is left)
__device__ __forceinline__ double recip_or_zero(double a) {
  const double r = 1.0 / a;
  return isfinite(r) ? r : 0.0;
}
__device__ __forceinline__ DF64 recip_or_zero(DF64 a) {
  const float r = __frcp_rn(a.hi);
  if (!isfinite(r) || r == 0.f) return DF64{0.f, 0.f};
  const float e = __fmaf_rn(-r, a.lo, __fmaf_rn(-r, a.hi, 1.f));   // 1 - r a
  return df_quick_two_sum(r, __fmul_rn(r, e));
}
// r = sqrt(a) and 1 / r, 0 where a <= 0 (1 / r: or so small that it overflows).  Double-float: one Newton step from the
// FP32 reciprocal root, no division.  FP64: 1 / r is left to recip_of, on the path that needs it.
__device__ __forceinline__ void sqrt_recip(double a, double& r, double& inv) {
  r = sqrt(fmax(a, 0.0));
  inv = 0.0;
}
__device__ __forceinline__ double recip_of(double r, double) { return recip_or_zero(r); }
__device__ __forceinline__ DF64 recip_of(DF64, DF64 inv) { return inv; }
__device__ __forceinline__ void sqrt_recip(DF64 a, DF64& r, DF64& inv) {
  const float y = rsqrtf(fmaxf(a.hi, 0.f));
  r = inv = DF64{0.f, 0.f};
  if (!isfinite(y)) return;
  if (y == 0.f) { r = a; return; }   // a = inf
  const float t = __fmul_rn(a.hi, y);
  const float tl = __fmaf_rn(a.lo, y, __fmaf_rn(a.hi, y, -t));     // a y = t + tl
  const float e = __fmul_rn(0.5f, __fmaf_rn(-tl, y, __fmaf_rn(-t, y, 1.f)));   // (1 - a y^2) / 2
  r = df_quick_two_sum(t, __fmaf_rn(t, e, tl));
  inv = df_quick_two_sum(y, __fmul_rn(y, e));
}

// start + sum_i v_i c_i for entries v_i of precision T and coefficients c_i of small_t<T>.  T = float: the low parts
// of the coefficients and the roundings of the sum (all but a bit of them) are kept beside it and added at
// the end, five instructions a term (the exact error of every product and sum takes eleven).
template <typename T> struct LinComb;
template <> struct LinComb<double> {
  double s;
  __device__ __forceinline__ explicit LinComb(double v) : s(v) {}
  __device__ __forceinline__ void add(double v, double c) { s += v * c; }
  __device__ __forceinline__ void sub(double v, double c) { s -= v * c; }
  __device__ __forceinline__ void scale(double c) { s *= c; }
  __device__ __forceinline__ double value() const { return s; }
};
template <> struct LinComb<float> {
  float hi, lo;
  __device__ __forceinline__ explicit LinComb(float v) : hi(v), lo(0.f) {}
  __device__ __forceinline__ void add(float v, DF64 c) {
    const float t = __fmaf_rn(v, c.hi, hi);
    lo = __fmaf_rn(v, c.lo, __fadd_rn(lo, __fmaf_rn(v, c.hi, __fsub_rn(hi, t))));
    hi = t;
  }
  __device__ __forceinline__ void sub(float v, DF64 c) { add(v, -c); }
  __device__ __forceinline__ void scale(DF64 c) {   // before any term
    const float v = hi;
    hi = __fmul_rn(v, c.hi);
    lo = __fmaf_rn(v, c.lo, __fmaf_rn(v, c.hi, -hi));
  }
  __device__ __forceinline__ float value() const { return __fadd_rn(hi, lo); }
};

struct GmresLayout {
  int s, ldh;
  int H, cs, sn, g, y, res, beta, nrm2, rhn, rr, total;
  __host__ __device__ constexpr explicit GmresLayout(int steps)
      : s(steps), ldh(steps + 1), H(0), cs((steps + 1) * steps), sn(cs + steps), g(sn + steps), y(g + steps + 1),
        res(y + steps), beta(res + 1), nrm2(beta + 1), rhn(nrm2 + 1), rr(rhn + steps + 1), total(rr + steps) {}
};

// host-side handle: the state array (elements of small_t), s, and the block
// partials of the reductions.  A reduction kernel only writes its partials, [column][block];
// every block of the kernel that needs the sums adds them for itself, in one fixed order (on large levels
// after a kernel has folded them, see kFoldFrom).
// (A last-block finish, with its fence, ticket, second fence, reload and one-thread
// bookkeeping, cost 1 to 2 us at the end of each of the two reductions of a step: a third of a
// small level's time.)  The dots of step j: nbd blocks in one of two areas from rows, by the parity of
// j.  |column j|^2: at rows + noff + (j & 1) nstride.  (A kernel that reads one area may write the
// other.)  nb0 blocks for column 0 (gather or copy), nbn for columns 1 .. s - 1 and ceil(n / 1024) for s.
struct GmresDev {
  void* base;
  int s;
  void* rows;
  int nbd, nb0, nbn, noff, nstride;
  int foff;   // where the folded partials lie, beyond the others; 0: a level that does not fold
  int late;   // the kernel before the last Gram-Schmidt step writes more than its column (see arnoldi2.cuh)
  // The Gram-Schmidt and update kernels trigger their successor right after the wait, not at their end: all
  // but FP64 in 3D, whose successors take the registers that the predecessors' long blocks
  // are still to be given (16^3: 1844 us late, 1874 early).  Late / early, us: 2D 128^2 345 / 332, 20 x 28 x 12
  // 593 / 582, 32^3 1654 / 1639, FP64 40 x 72 707 / 701, order 3 128^2 1032 / 1009 and 12^3 1433 / 1407.
  int early;
};

template <typename T>
__host__ __device__ __forceinline__ T* dot_rows(const GmresDev& d, int j) {
  return static_cast<T*>(d.rows) + (j & 1) * (d.nbd * KMAXB);
}
template <typename T>
__host__ __device__ __forceinline__ T* norm_rows(const GmresDev& d, int j) {
  return static_cast<T*>(d.rows) + d.noff + (j & 1) * d.nstride;
}
constexpr int GM_PER = 4;   // entries per thread of the smoother's vector kernels
__host__ __device__ __forceinline__ int gm_blocks(long long n) {
  return (int)((n + RED_THREADS * GM_PER - 1) / (RED_THREADS * GM_PER));
}
__host__ __device__ __forceinline__ int norm_count(const GmresDev& d, int j, long long n) {
  return j == 0 ? d.nb0 : j < d.s ? d.nbn : gm_blocks(n);
}

// Every consumer block reads every partial, which grows with the square of the level.  Levels whose kernels have more than
// kFoldFrom blocks put a kernel between (k_gm_fold) that leaves kFold sums a column.  One cycle, us, without / with it
// on every level: 3D FP32 32^3 (804 blocks on the finest) 1651 / 1683, 36^3 (1,140) 2927 / 2935, 40^3 (1,615) 2855 / 2838;
// FP64 40^3 17198 / 17039; beyond: FP32 96^3 35400 / 29600, 2D 2048^2 31200 / 16700, FP64 256800 / 220100, 234700 / 143400.
constexpr int kFoldFrom = 1400, kFold = 32;
template <typename T>
__host__ __device__ __forceinline__ T* fold_dots(const GmresDev& d, int j) {
  return static_cast<T*>(d.rows) + d.foff + (j & 1) * (KMAXB * kFold);
}
template <typename T>
__host__ __device__ __forceinline__ T* fold_norm(const GmresDev& d, int j) {
  return static_cast<T*>(d.rows) + d.foff + (2 * KMAXB + (j & 1)) * kFold;
}
// what the consumers add: the dots of step j (columns dot_parts apart), |column j|^2
template <typename T>
__device__ __forceinline__ const T* dot_sums(const GmresDev& d, int j) { return d.foff ? fold_dots<T>(d, j) : dot_rows<T>(d, j); }
__device__ __forceinline__ int dot_parts(const GmresDev& d) { return d.foff ? kFold : d.nbd; }
template <typename T>
__device__ __forceinline__ const T* norm_sums(const GmresDev& d, int j) { return d.foff ? fold_norm<T>(d, j) : norm_rows<T>(d, j); }
__device__ __forceinline__ int norm_parts(const GmresDev& d, int j, long long n) { return d.foff ? kFold : norm_count(d, j, n); }

// the block partials of a gather: |y|^2 of column 0 (start) or the k dots (every thread calls)
template <typename T>
__device__ __forceinline__ void store_partials(const GmresDev& d, int start, int k, const T (&acc)[KMAXB], unsigned bx,
                                               unsigned nb) {
  __shared__ T sh[RED_THREADS / 32][KMAXB];
  const int kk = start ? 1 : k;
  const T v = block_total<T>(acc, kk, sh);
  if ((int)threadIdx.x < kk) (start ? norm_rows<T>(d, 0) : dot_rows<T>(d, k - 1))[threadIdx.x * nb + bx] = v;
}

template <typename S>
struct GmresView {
  S* H;
  int ldh;
  S* cs;
  S* sn;
  S* g;       // rotated right-hand side, length s + 1
  S* rhn;     // 1 / norms of the stored columns, length s + 1 (written by the Gram-Schmidt steps)
  S* rr;      // 1 / R_ii, length s
  S* beta;    // |r0|
  int m;      // s + 1
};

// T: the smoother's precision
template <typename T>
__host__ __device__ __forceinline__ GmresView<small_t<T>> gmres_view(const GmresDev& d) {
  const GmresLayout L(d.s);
  small_t<T>* b = static_cast<small_t<T>*>(d.base);
  return GmresView<small_t<T>>{b + L.H, L.ldh, b + L.cs, b + L.sn, b + L.g, b + L.rhn, b + L.rr, b + L.beta, d.s + 1};
}

// Givens rotation (c, s) of (a, b), b >= 0, r = |(a, b)| and 1 / r for recip_of; the plain
// sum of squares where it is far from over- and underflow (hypot takes several times the FP64 instructions)
__device__ __forceinline__ void givens(double a, double b, double& c, double& s, double& r, double& rr) {
  const double q = a * a + b * b;
  r = q > 1e-200 && q < 1e200 ? sqrt(q) : hypot(a, b);
  c = 1.0;
  s = 0.0;
  if (r > 0.0) { c = a / r; s = b / r; }
  rr = 0.0;
}
__device__ __forceinline__ void givens(DF64 a, DF64 b, DF64& c, DF64& s, DF64& r, DF64& rr) {
  const DF64 q = a * a + b * b;
  c = DF64{1.f, 0.f};
  s = DF64{0.f, 0.f};
  if (q.hi > 1e-20f && q.hi < 1e20f) {
    sqrt_recip(q, r, rr);
    c = a * rr;
    s = b * rr;
  } else {
    r = DF64{hypotf(a.hi, b.hi), 0.f};
    rr = recip_or_zero(r);
    if (r.hi > 0.f) { c = a / r; s = b / r; }
  }
}

// start: beta = |r0|, g = (beta, 0, ...)   (one thread)
template <typename S>
__device__ __forceinline__ void gmres_start(const GmresView<S>& st, S nrm2) {
  S b, inv;
  sqrt_recip(nrm2, b, inv);
  st.beta[0] = b;
  st.g[0] = b;
  for (int i = 1; i < st.m; ++i) st.g[i] = S{};
}

// step k (k < KMAXB): H[k+1][k] = |w|, then the rotations of
// column k; all operands are loaded first and every index is a compile-time one (loops
// unrolled to KMAXB, predicated), so the chain runs in registers (one thread).  With runtime
// loop bounds the arrays lived in local memory, and this chain, on the serial tail of every
// Gram-Schmidt step, took about three times as long.
template <typename S>
__device__ __forceinline__ void gmres_step(const GmresView<S>& st, int k, S nrm2) {
  S* hg = st.H + (long long)k * st.ldh;
  S h[KMAXB], cs[KMAXB], sn[KMAXB];
#pragma unroll
  for (int i = 0; i < KMAXB; ++i) {
    h[i] = i <= k ? hg[i] : S{};
    cs[i] = i < k ? st.cs[i] : S{1};
    sn[i] = i < k ? st.sn[i] : S{};
  }
  const S gk = st.g[k];
  S hk1, unused;
  sqrt_recip(nrm2, hk1, unused);
  S a = h[0];                       // the entry the next rotation starts from
#pragma unroll
  for (int i = 0; i < KMAXB - 1; ++i)
    if (i < k) {
      const S b = h[i + 1];
      h[i] = cs[i] * a + sn[i] * b;
      a = -sn[i] * a + cs[i] * b;
    }
  S c, sv, r, rr;
  givens(a, hk1, c, sv, r, rr);
#pragma unroll
  for (int i = 0; i < KMAXB; ++i)
    if (i <= k) hg[i] = i == k ? r : h[i];
  hg[k + 1] = S{};
  st.rr[k] = recip_of(r, rr);
  st.cs[k] = c; st.sn[k] = sv;
  st.g[k + 1] = -sv * gk;
  st.g[k] = c * gk;
}

// The last step's rotations (k = s - 1, not written back) and, by the warp that calls,
//   what = 0: lane i < s: y_i / hn_i, y = R^-1 g by back substitution on the rotated matrix;
//   what = 1: lane i <= s: u_i, u = Q^T (g[s] e_s) / hn (Q = product of the Givens rotations),
// so that x + sum_i Z_i y_i / hn_i is the GMRES iterate and its residual is
// sum_i u_i (stored column i) by the Arnoldi relation.  Lane i holds row i: what the rotations
// and the substitution do to all rows is one instruction each, and the chains are one
// multiply-add a step.
template <typename S>
__device__ __forceinline__ S gmres_finish(const GmresView<S>& st, S nrm2, int what) {
  const int s = st.m - 1, k = s - 1, lane = threadIdx.x & 31, i = lane < KMAXB ? lane : 0;
  const S* hg = st.H + (long long)k * st.ldh;
  const bool old = lane < k;
  const S cs = old ? st.cs[i] : S{1}, sn = old ? st.sn[i] : S{};
  const S b1 = old ? hg[i + 1] : S{};
  S hk1, inv;
  sqrt_recip(nrm2, hk1, inv);
  // a_0 = h_0;  a_(i+1) = cs_i h_(i+1) - sn_i a_i;  R_ik = cs_i a_i + sn_i h_(i+1)
  const S q = cs * b1;
  S a = hg[0], mine = a;
#pragma unroll
  for (int t = 0; t < KMAXB - 1; ++t)
    if (t < k) {
      a = RealOps<S>::sub_prod(shfl_small(q, t), shfl_small(sn, t), a);
      if (lane == t + 1) mine = a;
    }
  S c, sv, r, rk;
  givens(a, hk1, c, sv, r, rk);
  const S gk = st.g[k];
  if (what == 0) {
    S acc = lane < k ? st.g[i] : lane == k ? c * gk : S{};
    const S rik = cs * mine + sn * b1;
    const S rr = lane < k ? st.rr[i] : lane == k ? recip_of(r, rk) : S{};
    S y = S{};
#pragma unroll
    for (int t = KMAXB - 1; t >= 0; --t)
      if (t < s) {
        const S yt = shfl_small(acc * rr, t);
        if (lane == t) y = yt;
        const S h = t == k ? rik : lane < t ? st.H[(long long)t * st.ldh + i] : S{};
        acc = RealOps<S>::sub_prod(acc, h, yt);
      }
    return lane < s ? y * st.rhn[i] : S{};
  }
  // u_i = cs_(i-1) b_i / hn_i with b_s = g[s], b_(i-1) = -sn_(i-1) b_i; u_0 = b_0 / hn_0
  S b = -sv * gk, u = b;
#pragma unroll
  for (int t = KMAXB - 1; t >= 0; --t)
    if (t < s) {
      const S ct = t == k ? c : shfl_small(cs, t), st_ = t == k ? sv : shfl_small(sn, t);
      if (lane == t + 1) u = ct * b;
      b = -(st_ * b);
    }
  if (lane == 0) u = b;
  return lane < s ? u * st.rhn[lane] : lane == s ? u * recip_of(hk1, inv) : S{};
}

}  // namespace als
