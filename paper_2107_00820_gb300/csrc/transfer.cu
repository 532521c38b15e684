// K5: standard Q2 prolongation P_H and its transpose (Sec. 4.2).
//
// V_H is a subspace of V_h, so P_H is nested interpolation: a fine node at a
// coarse node takes its value; a fine node at a quarter point of a coarse cell
// takes the coarse quadratic there, 1D weights (3/8, 3/4, -1/8) at 1/4 and
// (-1/8, 3/4, 3/8) at 3/4, tensorised over the axes.  Dirichlet rows (fine
// boundary) and columns (coarse boundary) are zero.  Both directions are
// gathers, so they need no atomics.
#include "batch.cuh"
#include "level.h"
#include "pdl.cuh"

namespace als {

// The 1D weights are dyadic (1, 3/4, 3/8, -1/8), so they and their products are
// exact in either precision; the sums run in the vector's precision T.
//
// Prolongation: a thread takes four consecutive fine nodes x = 4j .. 4j+3 of a row, which are
// combinations of the three coarse nodes 2j .. 2j+2 of the 1 or 3 x 1 or 3 coarse rows around it: all of
// those are loaded at once, predicated.  A tap counts
// only if it lies off the Dirichlet ends of its axis: the boundary of the box is exactly the set of
// nodes with some coordinate at an end.  A thread per node, 27 taps each, took 18 us on 32^3 cells; with
// both directions as they are now, and the coarse correction's residual formed by the gather before the
// restriction, a 40 x 24 x 32 level's apply, smoothing, restriction and prolongation take 263 us, 279 before,
// and an FP64 cycle on 16^3 cells 1924, 1969 before.
template <typename T>
__device__ __forceinline__ void prolong_rows(int f, int nc, int (&m)[3], T (&w)[3], bool (&ok)[3]) {
  const int c = f >> 2;
  const bool odd = f & 1, first = (f & 3) == 1;
  m[0] = odd ? 2 * c : f >> 1;
  m[1] = m[0] + 1;
  m[2] = m[0] + 2;
  w[0] = odd ? (first ? T(0.375) : T(-0.125)) : T(1);
  w[1] = T(0.75);
  w[2] = first ? T(-0.125) : T(0.375);
#pragma unroll
  for (int q = 0; q < 3; ++q) ok[q] = (odd || q == 0) && m[q] >= 1 && m[q] <= nc - 2;
}

template <typename T, int DIM>
__device__ __forceinline__ void prolong_body(unsigned bx, const Geom& gc, const Geom& gf, const T* __restrict__ xc,
                                             T* __restrict__ xf, T* __restrict__ xadd) {
  RowChunk rc;
  const bool have = row_chunk(gf, DIM, bx * blockDim.x + threadIdx.x, rc);
  pdl_wait();
  if (have) {
    constexpr int NZ = DIM == 3 ? 3 : 1;
    int my[3], mz[3] = {0, 0, 0};
    T wy[3], wz[3] = {T(1), T(0), T(0)};
    bool oy[3], oz[3] = {true, false, false};
    prolong_rows<T>(rc.y, gc.nn[1], my, wy, oy);
    if (DIM == 3) prolong_rows<T>(rc.z, gc.nn[2], mz, wz, oz);
    const bool inner = rc.y > 0 && rc.y < gf.nn[1] - 1 && (DIM == 2 || (rc.z > 0 && rc.z < gf.nn[2] - 1));
    const T* xcc = xc + (long long)rc.c * gc.N;
    T v[NZ][3][3], old[GX];
#pragma unroll
    for (int cz = 0; cz < NZ; ++cz)
#pragma unroll
      for (int cy = 0; cy < 3; ++cy) {
        const bool ok = inner && oy[cy] && oz[cz];
        const int row = ok ? gc.nn[0] * (my[cy] + gc.nn[1] * mz[cz]) : 0;
#pragma unroll
        for (int cx = 0; cx < 3; ++cx) {
          const int mx = 2 * rc.j + cx;
          v[cz][cy][cx] = ok && mx >= 1 && mx <= gc.nn[0] - 2 ? xcc[row + mx] : T(0);
        }
      }
#pragma unroll
    for (int q = 0; q < GX; ++q) old[q] = xadd && GX * rc.j + q < gf.nn[0] ? xadd[rc.t0 + q] : T(0);
    // the taps in one order (z, y, x) for every node: the robust correction that follows amplifies
    // a change of rounding here by gamma / mu
    T out[GX] = {T(0), T(0), T(0), T(0)};
#pragma unroll
    for (int cz = 0; cz < NZ; ++cz)
#pragma unroll
      for (int cy = 0; cy < 3; ++cy) {
        const T w = wy[cy] * wz[cz], *u = v[cz][cy];   // dyadic: every product of weights is exact
        out[0] += w * u[0];
        out[1] += (T(0.375) * w) * u[0];
        out[1] += (T(0.75) * w) * u[1];
        out[1] += (T(-0.125) * w) * u[2];
        out[2] += w * u[1];
        out[3] += (T(-0.125) * w) * u[0];
        out[3] += (T(0.75) * w) * u[1];
        out[3] += (T(0.375) * w) * u[2];
      }
#pragma unroll
    for (int q = 0; q < GX; ++q) {
      const int x = GX * rc.j + q;
      if (x >= gf.nn[0]) break;
      const bool in = inner && x > 0 && x < gf.nn[0] - 1;
      xf[rc.t0 + q] = in ? out[q] : T(0);
      if (xadd && in) xadd[rc.t0 + q] = old[q] + out[q];
    }
  }
  pdl_trigger();
}
template <typename T, int DIM>
__global__ void __launch_bounds__(256) k_prolong(Geom gc, Geom gf, const T* __restrict__ xc, T* __restrict__ xf,
                                                 T* __restrict__ xadd) {
  prolong_body<T, DIM>(blockIdx.x, gc, gf, xc, xf, xadd);
}
static unsigned prolong_blocks(const Geom& gf) {
  return (unsigned)(((long long)gf.dim * gf.nn[1] * gf.nn[2] * ((gf.nn[0] + GX - 1) / GX) + 255) / 256);
}

// Restriction (the transpose): a block takes 8 x 4 x 4 coarse nodes (8 x 16 in 2D) of a component,
// loads the fine nodes that they draw on once, zero at and beyond the Dirichlet ends, and sums
// along x, y and z in turn through shared memory: coarse node m takes fine nodes 2m with weight 1,
// 2m +- 1 with 3/4 (m odd, the middle of a cell) or 3/8, and for m even 2m +- 3 with -1/8.
// A thread per coarse node, its 125 taps straight from global memory with the zero weights of the odd
// axes included, took 13 us on 32^3 cells (see above for both).
template <int DIM>
struct RestrictTile {
  static constexpr int X = 8, Y = DIM == 3 ? 4 : 16, Z = DIM == 3 ? 4 : 1, OUT = X * Y * Z;
  static constexpr int FX = 2 * X + 3, FY = 2 * Y + 3, FZ = DIM == 3 ? 2 * Z + 3 : 1;   // first 2m - 3 of the first node
  static constexpr int FINE = FX * FY * FZ, XS = X * FY * FZ, YS = X * Y * FZ;
  static_assert(OUT == 128, "half a block's threads");
};
template <typename T>
__device__ __forceinline__ T restrict_line(const T* p, int stride, bool odd) {
  if (odd) return p[0] + T(0.75) * (p[-stride] + p[stride]);
  return p[0] + T(0.375) * (p[-stride] + p[stride]) - T(0.125) * (p[-3 * stride] + p[3 * stride]);
}

__host__ __device__ __forceinline__ unsigned restrict_blocks(const Geom& gc) {
  const int x = (gc.nn[0] + 7) >> 3;
  return gc.dim == 3 ? (unsigned)(3 * x * ((gc.nn[1] + 3) >> 2) * ((gc.nn[2] + 3) >> 2))
                     : (unsigned)(2 * x * ((gc.nn[1] + 15) >> 4));
}

template <typename T, int DIM>
__device__ __forceinline__ void restrict_body(unsigned bx, const Geom& gc, const Geom& gf, const T* __restrict__ rf,
                                              T* __restrict__ rc, T* fine, T* xs) {
  using R = RestrictTile<DIM>;
  const int tid = threadIdx.x;
  const int nx = (gc.nn[0] + R::X - 1) / R::X, ny = (gc.nn[1] + R::Y - 1) / R::Y, nz = DIM == 3 ? (gc.nn[2] + R::Z - 1) / R::Z : 1;
  int t = (int)bx;
  const int bi = t % nx;
  t /= nx;
  const int bj = t % ny;
  t /= ny;
  const int bk = t % nz, c = t / nz;
  const int m0 = bi * R::X, m1 = bj * R::Y, m2 = DIM == 3 ? bk * R::Z : 0;
  constexpr int NQ = (R::FINE + 255) / 256;
  int at[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int e = tid + 256 * q, r = e / R::FX, px = e - r * R::FX, pz = r / R::FY, py = r - pz * R::FY;
    const int x = 2 * m0 - 3 + px, y = 2 * m1 - 3 + py, z = DIM == 3 ? 2 * m2 - 3 + pz : 0;
    const bool ok = e < R::FINE && x >= 1 && x <= gf.nn[0] - 2 && y >= 1 && y <= gf.nn[1] - 2 &&
                    (DIM == 2 || (z >= 1 && z <= gf.nn[2] - 2));
    at[q] = ok ? c * (int)gf.N + x + gf.nn[0] * (y + gf.nn[1] * z) : -1;
  }
  pdl_wait();
  T v[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) v[q] = at[q] >= 0 ? rf[at[q]] : T(0);
#pragma unroll
  for (int q = 0; q < NQ; ++q)
    if (tid + 256 * q < R::FINE) fine[tid + 256 * q] = v[q];
  pdl_trigger();
  __syncthreads();
  for (int e = tid; e < R::XS; e += 256) {   // along x: [z][y][i]
    const int i = e % R::X, r = e / R::X;
    xs[e] = restrict_line<T>(fine + r * R::FX + 2 * i + 3, 1, i & 1);
  }
  __syncthreads();
  for (int e = tid; e < R::YS; e += 256) {   // along y: [z][j][i]
    const int i = e % R::X, r = e / R::X, j = r % R::Y, z = r / R::Y;
    fine[e] = restrict_line<T>(xs + (z * R::FY + 2 * j + 3) * R::X + i, R::X, j & 1);
  }
  __syncthreads();
  if (tid < R::OUT) {
    const int i = tid % R::X, r = tid / R::X, j = r % R::Y, k = r / R::Y;
    const int x = m0 + i, y = m1 + j, z = m2 + k;
    if (x < gc.nn[0] && y < gc.nn[1] && z < gc.nn[2]) {
      T s;
      if (DIM == 3) s = restrict_line<T>(fine + (2 * k + 3) * R::Y * R::X + j * R::X + i, R::Y * R::X, k & 1);
      else s = fine[tid];
      rc[c * (int)gc.N + x + gc.nn[0] * (y + gc.nn[1] * z)] = on_boundary(gc, x, y, z) ? T(0) : s;
    }
  }
}
template <typename T, int DIM>
__global__ void __launch_bounds__(256) k_restrict(Geom gc, Geom gf, const T* __restrict__ rf, T* __restrict__ rc) {
  __shared__ T fine[RestrictTile<DIM>::FINE], xs[RestrictTile<DIM>::XS];
  restrict_body<T, DIM>(blockIdx.x, gc, gf, rf, rc, fine, xs);
}

// merged launches (batch.cuh), FP32, 2D and 3D instances together
struct TransferArgs {
  Geom gc, gf;
  const float* in;
  float* out;
  float* aux;   // prolongation: xadd (may be NULL)
};
__global__ void __launch_bounds__(256) k_prolong_b(const __grid_constant__ BatchTab<TransferArgs> tb) {
  const int i = batch_slot(tb, blockIdx.x);
  const TransferArgs& a = tb.a[i];
  const unsigned bx = blockIdx.x - tb.start[i];
  if (a.gf.dim == 3) prolong_body<float, 3>(bx, a.gc, a.gf, a.in, a.out, a.aux);
  else prolong_body<float, 2>(bx, a.gc, a.gf, a.in, a.out, a.aux);
}
__global__ void __launch_bounds__(256) k_restrict_b(const __grid_constant__ BatchTab<TransferArgs> tb) {
  const int i = batch_slot(tb, blockIdx.x);
  const TransferArgs& a = tb.a[i];
  const unsigned bx = blockIdx.x - tb.start[i];
  __shared__ float fine[RestrictTile<3>::FINE], xs[RestrictTile<3>::XS];
  static_assert(RestrictTile<2>::FINE <= RestrictTile<3>::FINE && RestrictTile<2>::XS <= RestrictTile<3>::XS, "shared memory");
  if (a.gf.dim == 3) restrict_body<float, 3>(bx, a.gc, a.gf, a.in, a.out, fine, xs);
  else restrict_body<float, 2>(bx, a.gc, a.gf, a.in, a.out, fine, xs);
}

void prolong_std(const LevelDev& coarse, const LevelDev& fine, int prec, const void* xc, void* xf, cudaStream_t s,
                 void* xadd) {
  if (fine.k == 3) {
    qk_prolong(coarse, fine, prec, xc, xf, s, xadd);
    return;
  }
  const unsigned b = prolong_blocks(fine.g);
  if (prec == PREC_F64) {
    if (fine.g.dim == 2)
      launch_pdl(k_prolong<double, 2>, b, 256, 0, s, coarse.g, fine.g, (const double*)xc, (double*)xf, (double*)xadd);
    else launch_pdl(k_prolong<double, 3>, b, 256, 0, s, coarse.g, fine.g, (const double*)xc, (double*)xf, (double*)xadd);
  } else {
    if (fine.g.dim == 2)
      launch_pdl(k_prolong<float, 2>, b, 256, 0, s, coarse.g, fine.g, (const float*)xc, (float*)xf, (float*)xadd);
    else launch_pdl(k_prolong<float, 3>, b, 256, 0, s, coarse.g, fine.g, (const float*)xc, (float*)xf, (float*)xadd);
  }
  count_launch(1);
}

void restrict_std(const LevelDev& coarse, const LevelDev& fine, int prec, const void* rf, void* rc, cudaStream_t s) {
  if (fine.k == 3) {
    qk_restrict(coarse, fine, prec, rf, rc, s, nullptr);
    return;
  }
  const unsigned b = restrict_blocks(coarse.g);
  if (prec == PREC_F64) {
    if (fine.g.dim == 2) launch_pdl(k_restrict<double, 2>, b, 256, 0, s, coarse.g, fine.g, (const double*)rf, (double*)rc);
    else launch_pdl(k_restrict<double, 3>, b, 256, 0, s, coarse.g, fine.g, (const double*)rf, (double*)rc);
  } else {
    if (fine.g.dim == 2) launch_pdl(k_restrict<float, 2>, b, 256, 0, s, coarse.g, fine.g, (const float*)rf, (float*)rc);
    else launch_pdl(k_restrict<float, 3>, b, 256, 0, s, coarse.g, fine.g, (const float*)rf, (float*)rc);
  }
  count_launch(1);
}

int batch_prolong(const std::vector<BTransfer>& items, cudaStream_t s) {
  std::vector<TransferArgs> a;
  std::vector<unsigned> nb;
  for (const BTransfer& it : items) {
    a.push_back(TransferArgs{it.coarse->g, it.fine->g, (const float*)it.in, (float*)it.out, (float*)it.aux});
    nb.push_back(prolong_blocks(it.fine->g));
  }
  const int n = launch_batch(k_prolong_b, a, nb, 256, 0, s);
  count_launch(n);
  return n;
}

int batch_restrict(const std::vector<BTransfer>& items, cudaStream_t s) {
  std::vector<TransferArgs> a;
  std::vector<unsigned> nb;
  for (const BTransfer& it : items) {
    a.push_back(TransferArgs{it.coarse->g, it.fine->g, (const float*)it.in, (float*)it.out, nullptr});
    nb.push_back(restrict_blocks(it.coarse->g));
  }
  const int n = launch_batch(k_restrict_b, a, nb, 256, 0, s);
  count_launch(n);
  return n;
}

}  // namespace als
