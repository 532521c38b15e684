// K1: matrix-free application of the augmented Stokes operators on one level.
//
// The cells' contributions are evaluated with sum factorisation (apply_lines.cuh, apply_cells.cuh).  The nodal sum is formed without atomics, in a fixed order so
// every result is bitwise reproducible: normally all cells write their local
// outputs to a per-cell buffer and one gather kernel sums the <= 2^d values of
// each node (two launches per apply); batched applies (many vectors at once)
// instead run the cells in 2^d colours (parity of the cell index per axis) whose
// cells share no node and add into y directly.  Dirichlet rows carry
// the identity (y_D = x_D) and Dirichlet columns are masked (x_D treated as 0),
// which is the constrained operator of Eq. (augstokessys) in the form Firedrake
// and PETSc use.  B u (Eq. (stokessys)) is cell-local and written directly.
#include "batch.cuh"
#include "cell.cuh"
#include "cell_ops.cuh"
#include "level.h"
#include "reduce.cuh"
#include "pdl.cuh"

#include <stdexcept>
#include <type_traits>

namespace als {

// y_D = x_D (identity rows) when keep_bnd, else 0; interior rows zeroed.
template <typename T>
__global__ void k_init_out(Geom g, const T* __restrict__ x, T* __restrict__ y, int keep_bnd, long long vstride) {
  x += blockIdx.y * vstride;
  y += blockIdx.y * vstride;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long total = g.N * g.dim;
  if (t >= total) return;
  const long long nd = t % g.N;
  const int i = (int)(nd % g.nn[0]);
  const long long r = nd / g.nn[0];
  const int j = (int)(r % g.nn[1]);
  const int k = (int)(r / g.nn[1]);
  const bool bnd = on_boundary(g, i, j, k);
  y[t] = (bnd && keep_bnd) ? x[t] : T(0);
}

// (A x) along a row of global nodes: one thread sums GX = 4 consecutive nodes
// x = 4j .. 4j+3 of row (c, y, z) from the staged outputs (row layout, see
// stage_row).  Per (y, z) tap pair the four nodes read the six contiguous
// columns 6j-1 .. 6j+4; a column exists iff it lies in [0, 3 n0).  The taps are
// added in a fixed order (z tap, y tap, then the x pair), so results are
// reproducible.  Dirichlet rows: x_D (keep_bnd) or 0, unless raw.
template <typename T, int DIM>
__device__ __forceinline__ void gather_chunk(const Geom& g, const T* __restrict__ ebuf, const T* __restrict__ x,
                                             const RowChunk& rc, int keep_bnd, int raw, T (&out)[GX]) {
  const int nn0 = g.nn[0];
  const bool row_bnd = rc.y == 0 || rc.y == g.nn[1] - 1 || (DIM == 3 && (rc.z == 0 || rc.z == g.nn[2] - 1));
  if (!raw && row_bnd) {
#pragma unroll
    for (int q = 0; q < GX; ++q) {
      const int xi = GX * rc.j + q;
      out[q] = (keep_bnd && xi < nn0) ? x[rc.t0 + q] : T(0);
    }
    return;
  }
  // y and z taps: (cell, local index, exists)
  int cyv[2], lyv[2], czv[2], lzv[2];
  bool oky[2], okz[2];
  {
    const int yy = rc.y;
    if (yy & 1) { cyv[0] = yy >> 1; lyv[0] = 1; oky[0] = true; cyv[1] = 0; lyv[1] = 0; oky[1] = false; }
    else { cyv[0] = (yy >> 1) - 1; lyv[0] = 2; oky[0] = yy > 0; cyv[1] = yy >> 1; lyv[1] = 0; oky[1] = yy < 2 * g.n[1]; }
    const int zz = DIM == 3 ? rc.z : 1;
    const int n2 = DIM == 3 ? g.n[2] : 1;
    if (zz & 1) { czv[0] = zz >> 1; lzv[0] = 1; okz[0] = true; czv[1] = 0; lzv[1] = 0; okz[1] = false; }
    else { czv[0] = (zz >> 1) - 1; lzv[0] = 2; okz[0] = zz > 0; czv[1] = zz >> 1; lzv[1] = 0; okz[1] = zz < 2 * n2; }
    if (DIM == 2) { czv[0] = 0; lzv[0] = 0; }
  }
  const int ncol = 3 * g.n[0];
  const int p0 = 6 * rc.j - 1;
  // all loads first, predicated: a branch per tap pair would make each wait for the one before
  constexpr int TZ = DIM == 3 ? 2 : 1;
  T v[TZ][2][6];
#pragma unroll
  for (int tz = 0; tz < TZ; ++tz)
#pragma unroll
    for (int ty = 0; ty < 2; ++ty) {
      const bool ok = oky[ty] && (DIM == 2 || okz[tz]);
      const T* rowp = ebuf + (long long)(ok ? stage_row(g, rc.c, lyv[ty], lzv[tz], cyv[ty], czv[tz]) : 0) * ncol;
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const int p = p0 + k;
        v[tz][ty][k] = (ok && p >= 0 && p < ncol) ? rowp[p] : T(0);
      }
    }
  T acc[GX];
#pragma unroll
  for (int q = 0; q < GX; ++q) acc[q] = T(0);
#pragma unroll
  for (int tz = 0; tz < TZ; ++tz)
#pragma unroll
    for (int ty = 0; ty < 2; ++ty) {
      const T* w = v[tz][ty];
      acc[0] += w[0] + w[1];
      acc[1] += w[2];
      acc[2] += w[3] + w[4];
      acc[3] += w[5];
    }
#pragma unroll
  for (int q = 0; q < GX; ++q) {
    const int xi = GX * rc.j + q;
    if (!raw && (xi == 0 || xi == nn0 - 1)) acc[q] = (keep_bnd && xi < nn0) ? x[rc.t0 + q] : T(0);
    out[q] = acc[q];
  }
}

template <typename T, int DIM>
__device__ __forceinline__ void gather_cells_body(unsigned bx, const Geom& g, const T* __restrict__ ebuf,
                                                  const T* __restrict__ x, T* __restrict__ y, int keep_bnd, int raw,
                                                  const T* __restrict__ b) {
  RowChunk rc;
  const bool have = row_chunk(g, DIM, bx * blockDim.x + threadIdx.x, rc);
  pdl_wait();
  if (have) {
    T out[GX], bv[GX];
#pragma unroll
    for (int q = 0; q < GX; ++q) bv[q] = b && GX * rc.j + q < g.nn[0] ? b[rc.t0 + q] : T(0);
    gather_chunk<T, DIM>(g, ebuf, x, rc, keep_bnd, raw, out);
#pragma unroll
    for (int q = 0; q < GX; ++q)
      if (GX * rc.j + q < g.nn[0]) y[rc.t0 + q] = b ? bv[q] - out[q] : out[q];
  }
  pdl_trigger();
}
template <typename T, int DIM>
__global__ void k_gather_cells(Geom g, const T* __restrict__ ebuf, const T* __restrict__ x, T* __restrict__ y,
                               int keep_bnd, int raw, const T* __restrict__ b) {
  gather_cells_body<T, DIM>(blockIdx.x, g, ebuf, x, y, keep_bnd, raw, b);
}

static unsigned gather_threads(const Geom& g) {
  return (unsigned)(g.dim * g.nn[1] * g.nn[2] * ((g.nn[0] + GX - 1) / GX));
}

// Gather fused with the reduction that consumes the result:
//   y = b + sigma A x (b NULL: y = sigma A x);  block partials of V_j . y, j < k, or, start,
//   of |y|^2.  Fixed grid and order: reproducible.
// All sums run in T.
// KC = k, or 0 for start (with arrays of KMAXB columns, predicated, a block took 80 registers, three
// an SM, whatever it needed).
template <typename T, int DIM, int KC>
__device__ __forceinline__ void gather_epi_body(unsigned bx, unsigned nb, const Geom& g, const T* __restrict__ ebuf,
                                                const T* __restrict__ x, T* __restrict__ y, const T* __restrict__ b,
                                                double sigma, const T* __restrict__ V, long long ld,
                                                const GmresDev& sd) {
  constexpr bool start = KC == 0;
  T acc[KMAXB];
#pragma unroll
  for (int j = 0; j < KMAXB; ++j) acc[j] = T(0);
  RowChunk rc;
  const bool have = row_chunk(g, DIM, bx * blockDim.x + threadIdx.x, rc);
  // The basis columns come from earlier kernels of the chain, which completed before
  // this launch began (every kernel waits on its predecessor before it lets its
  // successor start): they are read through L2 while the preceding kernel finishes.
  T vp[GX][start ? 1 : KC];
#pragma unroll
  for (int q = 0; q < GX; ++q)
#pragma unroll
    for (int jj = 0; jj < KC; ++jj)
      vp[q][jj] = have && GX * rc.j + q < g.nn[0] ? __ldcg(V + (long long)jj * ld + rc.t0 + q) : T(0);
  pdl_wait();
  if (have) {
    T ax[GX];
    gather_chunk<T, DIM>(g, ebuf, x, rc, 1, 0, ax);
#pragma unroll
    for (int q = 0; q < GX; ++q) {
      if (GX * rc.j + q >= g.nn[0]) break;
      const long long t = rc.t0 + q;
      const T v = (b ? b[t] : T(0)) + (T)sigma * ax[q];
      y[t] = v;
      if constexpr (start) {
        acc[0] += v * v;
      } else {
#pragma unroll
        for (int jj = 0; jj < KC; ++jj) acc[jj] += vp[q][jj] * v;
      }
    }
  }
  pdl_trigger();
  store_partials<T>(sd, start, KC, acc, bx, nb);
}
template <typename T, int DIM, int KC>
__global__ void __launch_bounds__(RED_THREADS) k_gather_epi(Geom g, const T* __restrict__ ebuf,
                                                            const T* __restrict__ x, T* __restrict__ y,
                                                            const T* __restrict__ b, double sigma,
                                                            const T* __restrict__ V, long long ld, GmresDev sd) {
  gather_epi_body<T, DIM, KC>(blockIdx.x, gridDim.x, g, ebuf, x, y, b, sigma, V, ld, sd);
}
template <typename T, int DIM>
static auto gather_epi_kernel(int start, int k) {
  static constexpr decltype(&k_gather_epi<T, DIM, 0>) f[KMAXB + 1] = {
      k_gather_epi<T, DIM, 0>, k_gather_epi<T, DIM, 1>, k_gather_epi<T, DIM, 2>, k_gather_epi<T, DIM, 3>, k_gather_epi<T, DIM, 4>,
      k_gather_epi<T, DIM, 5>, k_gather_epi<T, DIM, 6>, k_gather_epi<T, DIM, 7>, k_gather_epi<T, DIM, 8>};
  return f[start ? 0 : k];
}

#include "apply_lines.cuh"
#include "apply_cells.cuh"

// Which form a 3D scalar apply takes.  Measured (apply_agamma call on n^3 cells, us, line form
// against register form): FP32 16^3 32.4 / 32.7, 20^3 35.0 / 33.8, 24^3 40.0 / 35.8, 32^3
// 54.8 / 42.3; FP64 12^3 59.3 / 71.3, 14^3 74.8 / 71.3, 16^3 90.3 / 72.0, 20^3 136 / 99 (a warp's
// FP64 instruction takes 64 cycles of its scheduler's pipe, so the register form's longer chain
// is a floor of about 40 us until its warps outnumber the schedulers).
static bool cells_in_registers(const Geom& g, bool fp64) { return g.ncells >= (fp64 ? 2500 : 5000); }

// the cell kernel of one apply: 2D two lanes per cell; 3D the line form, or, where a whole apply
// is staged (STAGED; all cells, one vector), the register form on large levels
// (ZP, staged only: the input comes from the star-patch outputs, see PatchIn)
template <typename T, int DIM, bool TENSOR, int MODE, bool STAGED, bool ZP = false>
static void launch_cells(int nvec, cudaStream_t s, const Geom& g, const Colour& col, const CellConst<T>& cc,
                         const T* x, T* y, const T* coef, const T* p_in, T* p_out, long long vstride, T* ebuf,
                         const T* winv, PatchIn<T> pin = PatchIn<T>{}) {
  if constexpr (DIM == 3) {
    if constexpr (STAGED && !TENSOR) {
      if (cells_in_registers(g, sizeof(T) == 8)) {
        using C = Cells3<T, MODE>;
        launch_pdl(k_apply_cells3<T, MODE, ZP>, (unsigned)((g.ncells + C::CELLS - 1) / C::CELLS), C::THREADS, 0, s, g,
                   cc, x, coef, p_in, p_out, ebuf, winv, pin);
        return;
      }
    }
    launch_pdl(k_apply_lines<T, TENSOR, MODE, STAGED, ZP>, dim3((unsigned)((col.count + 7) / 8), nvec), 256, 0, s, g,
               col, cc, x, y, coef, p_in, p_out, vstride, ebuf, winv, pin);
  } else {
    launch_pdl(k_apply_cells2<T, TENSOR, MODE, STAGED, ZP>,
               dim3((unsigned)((col.count + C2_CELLS - 1) / C2_CELLS), nvec), C2_THREADS, 0, s, g, col, cc, x, y,
               coef, p_in, p_out, vstride, ebuf, winv, pin);
  }
}

template <typename T, int DIM, bool TENSOR, int MODE>
static void launch_apply(const LevelDev& L, double gamma, const void* x, void* y, const void* p_in,
                         void* p_out, int nvec, long long vstride, cudaStream_t s, const void* b = nullptr) {
  const Geom& g = L.g;
  constexpr bool NEED_FLUX = (MODE & (OP_VISC | OP_AL | OP_BT)) != 0;
  const T* coef = nullptr;
  const T* winv = nullptr;
  if constexpr (std::is_same<T, double>::value) { coef = L.coef64; winv = L.winv64; }
  else { coef = L.coef32; winv = L.winv32; }
  const int keep_bnd = ((MODE & OP_VISC) && !(MODE & OP_RAW)) ? 1 : 0;
  if (nvec == 1 && L.ebuf) {
    // one launch over all cells into the per-cell buffer, one gather launch per node
    const Colour col = all_cells(g);
    launch_cells<T, DIM, TENSOR, MODE, true>(1, s, g, col,
                                             cell_const<T>(g, gamma), (const T*)x, (T*)y, coef, (const T*)p_in,
                                             (T*)p_out, 0, (T*)L.ebuf, winv);
    if (NEED_FLUX) {
      launch_pdl(k_gather_cells<T, DIM>, (gather_threads(g) + 255) / 256, 256, 0, s, g, (const T*)L.ebuf,
                 (const T*)x, (T*)y, keep_bnd, (MODE & OP_RAW) ? 1 : 0, (const T*)b);
    }
    count_launch(NEED_FLUX ? 2 : 1);
    return;
  }
  for (int v0 = 0; v0 < nvec; v0 += 65535) {
    const int nv = nvec - v0 < 65535 ? nvec - v0 : 65535;
    const T* xv = (const T*)x + v0 * vstride;
    T* yv = (T*)y + v0 * vstride;
    if (NEED_FLUX) {
      const long long tot = g.N * g.dim;
      dim3 grid((unsigned)((tot + 255) / 256), nv);
      k_init_out<T><<<grid, 256, 0, s>>>(g, xv, yv, keep_bnd, vstride);
    }
    const int ncol = NEED_FLUX ? (1 << DIM) : 1;   // B u alone is cell-local: one launch
    for (int colour = 0; colour < ncol; ++colour) {
      const Colour col = NEED_FLUX ? make_colour(g, colour) : all_cells(g);
      launch_cells<T, DIM, TENSOR, MODE, false>(nv, s, g, col, cell_const<T>(g, gamma), xv, yv, coef,
                                                (const T*)p_in, (T*)p_out, vstride, nullptr, winv);
    }
    count_launch((NEED_FLUX ? 1 : 0) + ncol);
  }
}

template <typename T, int DIM, bool TENSOR>
static void dispatch_mode(const LevelDev& L, int mode, double gamma, const void* x, void* y,
                          const void* p_in, void* p_out, int nvec, long long vstride, cudaStream_t s) {
  switch (mode) {
    case OP_VISC | OP_AL:
      launch_apply<T, DIM, TENSOR, OP_VISC | OP_AL>(L, gamma, x, y, p_in, p_out, nvec, vstride, s); break;
    case OP_AL: launch_apply<T, DIM, TENSOR, OP_AL>(L, gamma, x, y, p_in, p_out, nvec, vstride, s); break;
    case OP_B: launch_apply<T, DIM, TENSOR, OP_B>(L, gamma, x, y, p_in, p_out, nvec, vstride, s); break;
    case OP_BT: launch_apply<T, DIM, TENSOR, OP_BT>(L, gamma, x, y, p_in, p_out, nvec, vstride, s); break;
    default:
      if constexpr (std::is_same<T, double>::value) {
        switch (mode) {
          case OP_VISC | OP_AL | OP_BT | OP_B:
            launch_apply<T, DIM, TENSOR, OP_VISC | OP_AL | OP_BT | OP_B>(L, gamma, x, y, p_in, p_out, nvec, vstride, s);
            break;
          case OP_VISC | OP_AL | OP_RAW:
            launch_apply<T, DIM, TENSOR, OP_VISC | OP_AL | OP_RAW>(L, gamma, x, y, p_in, p_out, nvec, vstride, s);
            break;
          case OP_B | OP_RAW:
            launch_apply<T, DIM, TENSOR, OP_B | OP_RAW>(L, gamma, x, y, p_in, p_out, nvec, vstride, s); break;
          case OP_VISC | OP_BT | OP_B | OP_RAW:   // the nonlinear residual's operators (Newton)
            launch_apply<T, DIM, TENSOR, OP_VISC | OP_BT | OP_B | OP_RAW>(L, gamma, x, y, p_in, p_out, nvec, vstride,
                                                                          s);
            break;
          default: break;
        }
      }
      break;
  }
}

static void op_dispatch(const LevelDev& L, int prec, int mode, double gamma, const void* x, void* y,
                        const void* p_in, void* p_out, int nvec, long long vstride, cudaStream_t s) {
  if (prec == PREC_F64) {
    if (L.g.dim == 2) {
      if (L.tensor) dispatch_mode<double, 2, true>(L, mode, gamma, x, y, p_in, p_out, nvec, vstride, s);
      else dispatch_mode<double, 2, false>(L, mode, gamma, x, y, p_in, p_out, nvec, vstride, s);
    } else {
      if (L.tensor) dispatch_mode<double, 3, true>(L, mode, gamma, x, y, p_in, p_out, nvec, vstride, s);
      else dispatch_mode<double, 3, false>(L, mode, gamma, x, y, p_in, p_out, nvec, vstride, s);
    }
  } else {
    if (L.g.dim == 2) {
      if (L.tensor) dispatch_mode<float, 2, true>(L, mode, gamma, x, y, p_in, p_out, nvec, vstride, s);
      else dispatch_mode<float, 2, false>(L, mode, gamma, x, y, p_in, p_out, nvec, vstride, s);
    } else {
      if (L.tensor) dispatch_mode<float, 3, true>(L, mode, gamma, x, y, p_in, p_out, nvec, vstride, s);
      else dispatch_mode<float, 3, false>(L, mode, gamma, x, y, p_in, p_out, nvec, vstride, s);
    }
  }
}

void op_apply(const LevelDev& L, int prec, int mode, double gamma, const void* x, void* y,
              const void* p_in, void* p_out, cudaStream_t s) {
  if (L.k == 3) {
    qk_apply(L, prec, mode, gamma, x, y, p_in, p_out, s);
    return;
  }
  op_dispatch(L, prec, mode, gamma, x, y, p_in, p_out, 1, 0, s);
}

template <typename T, int DIM>
static void residual_dim(const LevelDev& L, int mode, double gamma, const void* x, const void* b, void* y,
                         cudaStream_t s) {
  if (mode == OP_AL) launch_apply<T, DIM, false, OP_AL>(L, gamma, x, y, nullptr, nullptr, 1, 0, s, b);
  else if (L.tensor) launch_apply<T, DIM, true, OP_VISC | OP_AL>(L, gamma, x, y, nullptr, nullptr, 1, 0, s, b);
  else launch_apply<T, DIM, false, OP_VISC | OP_AL>(L, gamma, x, y, nullptr, nullptr, 1, 0, s, b);
}
void op_residual(const LevelDev& L, int prec, int mode, double gamma, const void* x, const void* b, void* y,
                 cudaStream_t s) {
  if (!L.ebuf) throw std::logic_error("op_residual: a level without the staging buffer");   // the coloured form takes no b
  if (prec == PREC_F64) {
    if (L.g.dim == 2) residual_dim<double, 2>(L, mode, gamma, x, b, y, s);
    else residual_dim<double, 3>(L, mode, gamma, x, b, y, s);
  } else {
    if (L.g.dim == 2) residual_dim<float, 2>(L, mode, gamma, x, b, y, s);
    else residual_dim<float, 3>(L, mode, gamma, x, b, y, s);
  }
}

template <typename T, int DIM, bool TENSOR>
static void launch_apply_epi(const LevelDev& L, double gamma, const void* x, void* y, const ApplyEpi& e,
                             cudaStream_t s, cudaEvent_t e0, cudaEvent_t e1) {
  const Geom& g = L.g;
  const T* coef = nullptr;
  const T* winv = nullptr;
  if constexpr (std::is_same<T, double>::value) { coef = L.coef64; winv = L.winv64; }
  else { coef = L.coef32; winv = L.winv32; }
  const Colour col = all_cells(g);
  // External records become event-record nodes when the stream is being captured
  if (e0) cudaEventRecordWithFlags(e0, s, cudaEventRecordExternal);
  if (e.pout)   // x = z formed from the patch outputs; z stored on the way
    launch_cells<T, DIM, TENSOR, OP_VISC | OP_AL, true, true>(
        1, s, g, col, cell_const<T>(g, gamma), nullptr, (T*)y, coef, nullptr, nullptr, 0, (T*)L.ebuf, winv,
        PatchIn<T>{(const T*)e.pout, (T*)x});
  else
    launch_cells<T, DIM, TENSOR, OP_VISC | OP_AL, true>(1, s, g, col, cell_const<T>(g, gamma), (const T*)x, (T*)y,
                                                         coef, nullptr, nullptr, 0, (T*)L.ebuf, winv);
  if (e1) cudaEventRecordWithFlags(e1, s, cudaEventRecordExternal);
  launch_pdl(gather_epi_kernel<T, DIM>(e.start, e.k), apply_epi_blocks(L), RED_THREADS, 0, s, g, (const T*)L.ebuf,
             (const T*)x, (T*)y, (const T*)e.b, e.sigma, (const T*)e.V, e.ld, e.st);
  count_launch(2);
}

int apply_epi_blocks(const LevelDev& L) {
  return L.k == 3 ? qk_epi_blocks(L) : (int)((gather_threads(L.g) + RED_THREADS - 1) / RED_THREADS);
}

void op_apply_epi(const LevelDev& L, int prec, double gamma, const void* x, void* y, const ApplyEpi& e,
                  cudaStream_t s, cudaEvent_t e0, cudaEvent_t e1) {
  if (L.k == 3) {
    qk_apply_epi(L, prec, gamma, x, y, e, s, e0, e1);
    return;
  }
  if (prec == PREC_F64) {
    if (L.g.dim == 2) {
      if (L.tensor) launch_apply_epi<double, 2, true>(L, gamma, x, y, e, s, e0, e1);
      else launch_apply_epi<double, 2, false>(L, gamma, x, y, e, s, e0, e1);
    } else {
      if (L.tensor) launch_apply_epi<double, 3, true>(L, gamma, x, y, e, s, e0, e1);
      else launch_apply_epi<double, 3, false>(L, gamma, x, y, e, s, e0, e1);
    }
  } else {
    if (L.g.dim == 2) {
      if (L.tensor) launch_apply_epi<float, 2, true>(L, gamma, x, y, e, s, e0, e1);
      else launch_apply_epi<float, 2, false>(L, gamma, x, y, e, s, e0, e1);
    } else {
      if (L.tensor) launch_apply_epi<float, 3, true>(L, gamma, x, y, e, s, e0, e1);
      else launch_apply_epi<float, 3, false>(L, gamma, x, y, e, s, e0, e1);
    }
  }
}

// ---------------------------------------------------------------------------
// merged launches (batch.cuh): FP32, scalar viscosity, 2D and 3D instances in one launch
// (each item in the form its single-instance apply takes)
// ---------------------------------------------------------------------------
struct CellArgs {
  Geom g;
  Colour col;
  CellConst<float> cc;
  const float* x;
  float* y;
  const float* coef;
  float* ebuf;
  const float* winv;
  PatchIn<float> pin;
};
// ZP: x is formed from the star-patch outputs (PatchIn), as op_apply_epi does with ApplyEpi::pout.
// Three kernels, for 2D items, 3D items in the line form and 3D items in the register form
template <int MODE, bool ZP>
__global__ void __launch_bounds__(C2_THREADS) k_cells2_b(const __grid_constant__ BatchTab<CellArgs> tb) {
  const int i = batch_slot(tb, blockIdx.x);
  const CellArgs& a = tb.a[i];
  apply_cells2_body<float, false, MODE, true, ZP>((blockIdx.x - tb.start[i]) * (C2_THREADS / 32) + threadIdx.x / 32,
                                                  a.g, a.col, a.cc, a.x, a.y, a.coef, nullptr, nullptr, 0, a.ebuf, a.winv, a.pin);
}
template <int MODE, bool ZP>
__global__ void __launch_bounds__(256) k_lines_b(const __grid_constant__ BatchTab<CellArgs> tb) {
  const int i = batch_slot(tb, blockIdx.x);
  const CellArgs& a = tb.a[i];
  apply_lines_body<float, false, MODE, true, ZP>(blockIdx.x - tb.start[i], a.g, a.col, a.cc, a.x, a.y, a.coef, nullptr,
                                                 nullptr, 0, a.ebuf, a.winv, a.pin);
}
template <int MODE, bool ZP>
__global__ void __launch_bounds__(Cells3<float, MODE>::THREADS, Cells3<float, MODE>::BLOCKS)
    k_cells3_b(const __grid_constant__ BatchTab<CellArgs> tb) {
  __shared__ typename Cells3<float, MODE>::Smem sm;
  const int i = batch_slot(tb, blockIdx.x);
  const CellArgs& a = tb.a[i];
  apply_cells3_body<float, MODE, ZP>(blockIdx.x - tb.start[i], a.g, a.cc, a.x, a.coef, nullptr, nullptr, a.ebuf,
                                     a.winv, a.pin, sm);
}

struct GatherArgs {
  Geom g;
  const float* ebuf;
  const float* x;
  float* y;
  const float* b;
  double sigma;
  int keep_bnd;
  const float* V;
  long long ld;
  GmresDev st;
};
template <int KC>
__global__ void __launch_bounds__(RED_THREADS) k_gather_epi_b(const __grid_constant__ BatchTab<GatherArgs> tb) {
  const int i = batch_slot(tb, blockIdx.x);
  const GatherArgs& a = tb.a[i];
  const unsigned bx = blockIdx.x - tb.start[i], nb = tb.start[i + 1] - tb.start[i];
  if (a.g.dim == 3)
    gather_epi_body<float, 3, KC>(bx, nb, a.g, a.ebuf, a.x, a.y, a.b, a.sigma, a.V, a.ld, a.st);
  else
    gather_epi_body<float, 2, KC>(bx, nb, a.g, a.ebuf, a.x, a.y, a.b, a.sigma, a.V, a.ld, a.st);
}
__global__ void __launch_bounds__(256) k_gather_cells_b(const __grid_constant__ BatchTab<GatherArgs> tb) {
  const int i = batch_slot(tb, blockIdx.x);
  const GatherArgs& a = tb.a[i];
  const unsigned bx = blockIdx.x - tb.start[i];
  if (a.g.dim == 3) gather_cells_body<float, 3>(bx, a.g, a.ebuf, a.x, a.y, a.keep_bnd, 0, a.b);
  else gather_cells_body<float, 2>(bx, a.g, a.ebuf, a.x, a.y, a.keep_bnd, 0, a.b);
}

static CellArgs cell_args(const BApply& it, bool zp) {
  const LevelDev& L = *it.L;
  CellArgs a{};
  a.g = L.g;
  a.col = all_cells(L.g);
  a.cc = cell_const<float>(L.g, it.gamma);
  a.x = (const float*)it.x;
  a.y = (float*)it.y;
  a.coef = L.coef32;
  a.ebuf = (float*)L.ebuf;
  a.winv = L.winv32;
  if (zp) a.pin = PatchIn<float>{(const float*)it.e.pout, (float*)it.x};
  return a;
}
// the cell kernels of every item (all of them with star-patch input, or none), one launch per
// kernel that some item takes
template <int MODE, bool ZP>
static int batch_cells(const std::vector<BApply>& items, cudaStream_t s) {
  std::vector<CellArgs> a[3];
  std::vector<unsigned> nb[3];
  using C3 = Cells3<float, MODE>;
  const int per[3] = {C2_CELLS, 8, C3::CELLS};
  for (const BApply& it : items) {
    const Geom& g = it.L->g;
    const int k = g.dim == 2 ? 0 : (cells_in_registers(g, false) ? 2 : 1);
    a[k].push_back(cell_args(it, ZP));
    nb[k].push_back((unsigned)((g.ncells + per[k] - 1) / per[k]));
  }
  int n = 0;
  if (!a[0].empty()) n += launch_batch(k_cells2_b<MODE, ZP>, a[0], nb[0], C2_THREADS, 0, s);
  if (!a[1].empty()) n += launch_batch(k_lines_b<MODE, ZP>, a[1], nb[1], 256, 0, s);
  if (!a[2].empty())
    n += launch_batch(k_cells3_b<MODE, ZP>, a[2], nb[2], C3::THREADS, 0, s);
  return n;
}

int batch_apply_epi(const std::vector<BApply>& items, cudaStream_t s) {
  const bool zp = !items.empty() && items[0].e.pout;   // a smoothing's items agree
  int n = zp ? batch_cells<OP_VISC | OP_AL, true>(items, s) : batch_cells<OP_VISC | OP_AL, false>(items, s);
  std::vector<GatherArgs> a;
  std::vector<unsigned> nb;
  for (const BApply& it : items) {
    const LevelDev& L = *it.L;
    a.push_back(GatherArgs{L.g, (const float*)L.ebuf, (const float*)it.x, (float*)it.y, (const float*)it.e.b,
                           it.e.sigma, 1, (const float*)it.e.V, it.e.ld, it.e.st});
    nb.push_back(apply_epi_blocks(L));
  }
  static constexpr decltype(&k_gather_epi_b<0>) f[KMAXB + 1] = {
      k_gather_epi_b<0>, k_gather_epi_b<1>, k_gather_epi_b<2>, k_gather_epi_b<3>, k_gather_epi_b<4>,
      k_gather_epi_b<5>, k_gather_epi_b<6>, k_gather_epi_b<7>, k_gather_epi_b<8>};
  n += launch_batch(f[items[0].e.start ? 0 : items[0].e.k], a, nb, RED_THREADS, 0, s);   // the items agree in k and start
  count_launch(n);
  return n;
}

int batch_apply_al(const std::vector<BApply>& items, cudaStream_t s) {
  int n = batch_cells<OP_AL, false>(items, s);
  std::vector<GatherArgs> a;
  std::vector<unsigned> nb;
  for (const BApply& it : items) {
    const LevelDev& L = *it.L;
    GatherArgs g{};
    g.g = L.g;
    g.ebuf = (const float*)L.ebuf;
    g.x = (const float*)it.x;
    g.y = (float*)it.y;
    g.b = (const float*)it.e.b;
    g.keep_bnd = 0;   // OP_AL alone: zero Dirichlet rows, as op_apply
    a.push_back(g);
    nb.push_back((gather_threads(L.g) + 255) / 256);
  }
  n += launch_batch(k_gather_cells_b, a, nb, 256, 0, s);
  count_launch(n);
  return n;
}

// Several independent FP64 applies of A_gamma (used to form the coarse matrix
// column by column from unit vectors): vector v at X + v*stride.
void op_apply_multi(const LevelDev& L, double gamma, const double* X, double* Y, int nvec,
                    long long stride, cudaStream_t s) {
  op_dispatch(L, PREC_F64, OP_VISC | OP_AL, gamma, X, Y, nullptr, nullptr, nvec, stride, s);
}

// F_(c,a) = sum_q |J| w_q f_c(x_q) phi_a(x_q): the load vector of the body force.
template <int DIM>
__global__ void k_load(Geom g, Colour col, double wdet, const double* __restrict__ f, double* __restrict__ F) {
  constexpr int NB = Sz<DIM>::NB;
  int cx, cy, cz;
  if (!colour_cell(col, (long long)blockIdx.x * blockDim.x + threadIdx.x, cx, cy, cz)) return;
  const long long cell = (long long)cx + (long long)g.n[0] * ((long long)cy + (long long)g.n[1] * cz);
  double loc[DIM][NB];
#pragma unroll
  for (int c = 0; c < DIM; ++c)
#pragma unroll
    for (int a = 0; a < NB; ++a) loc[c][a] = 0.0;
  for (int q = 0; q < NB; ++q) {
    const int qx = q % 3, qy = (q / 3) % 3, qz = q / 9;
    double w = wdet * Ref<double>::W(qx) * Ref<double>::W(qy) * (DIM == 3 ? Ref<double>::W(qz) : 1.0);
    double fq[DIM];
#pragma unroll
    for (int c = 0; c < DIM; ++c) fq[c] = f[(cell * NB + q) * DIM + c] * w;
#pragma unroll
    for (int a = 0; a < NB; ++a) {
      const int ax = a % 3, ay = (a / 3) % 3, az = a / 9;
      const double phi = Ref<double>::B(qx, ax) * Ref<double>::B(qy, ay) * (DIM == 3 ? Ref<double>::B(qz, az) : 1.0);
#pragma unroll
      for (int c = 0; c < DIM; ++c) loc[c][a] += fq[c] * phi;
    }
  }
#pragma unroll
  for (int a = 0; a < NB; ++a) {
    const int i = 2 * cx + a % 3, j = 2 * cy + (a / 3) % 3, k = (DIM == 3) ? 2 * cz + a / 9 : 0;
    const long long nd = node_id(g, i, j, k);
#pragma unroll
    for (int c = 0; c < DIM; ++c) F[c * g.N + nd] += loc[c][a];
  }
}

void op_load_vector(const LevelDev& L, const double* f_qp, double* F, cudaStream_t s) {
  if (L.k == 3) {
    qk_load_vector(L, f_qp, F, s);
    return;
  }
  const Geom& g = L.g;
  double wdet = 1.0;
  for (int k = 0; k < g.dim; ++k) wdet *= 0.5 * g.h[k];
  cudaMemsetAsync(F, 0, sizeof(double) * g.N * g.dim, s);
  for (int colour = 0; colour < (1 << g.dim); ++colour) {
    const Colour col = make_colour(g, colour);
    const unsigned blocks = (unsigned)((col.count + 127) / 128);
    if (g.dim == 2) k_load<2><<<blocks, 128, 0, s>>>(g, col, wdet, f_qp, F);
    else k_load<3><<<blocks, 128, 0, s>>>(g, col, wdet, f_qp, F);
  }
  count_launch(1 << g.dim);
}

}  // namespace als
