// The order-3 discretisation in three dimensions: [Q3]^3 x P2^disc on uniform hexahedral
// meshes (the discretisation of the 3D sinker runs, Table linear, and the k = 3 column of
// Table k, Sec. 5.2.2), FP64 and FP32: operator applies, vertex-star setup and smoother,
// robust transfers, coarse images, mass and Schur blocks, so that the context's cycle and
// FGMRES run on it unchanged (qk.cu's entry points dispatch here for 3D levels).
//
// Velocity: continuous Q3, nodal basis on the 4 equispaced nodes -1, -1/3, 1/3, 1 per axis
// and cell, node lattice 3n + 1 per direction, x fastest; local node a = ax + 4 ay + 16 az.
// Pressure: discontinuous P2, the monomials in reference coordinates ordered by total
// degree, then x before y before z: {1, xi, eta, zeta, xi^2, xi eta, xi zeta, eta^2,
// eta zeta, zeta^2}; 10 per cell.  Quadrature: 4 x 4 x 4 Gauss-Legendre points, point
// q = qx + 4 qy + 16 qz.  Vertex stars: the free nodes at lattice offsets -2..2 from 3v in
// each direction (125 nodes, 375 dofs at an interior vertex); the interior of a coarse cell
// is the star of the fine vertex at its centre (Eq. (Ptilde)).
//
// The cell kernel factorises the tensor-product basis (sum factorisation: three 4-point
// contractions per direction instead of the 64 x 64 point-node products), one 64-thread
// group per cell.  The 375 x 375 star matrices do not fit in shared memory: each CTA of the
// persistent setup kernel assembles its star in a global workspace row block and inverts it
// by block Gauss-Jordan elimination (16 pivots per pass, the pivot block and the panels in
// shared memory).  Deterministic: per-cell and per-star outputs are staged and summed per
// node in a fixed order.
#include <cuda_bf16.h>
#include <math.h>

#include <type_traits>
#include <vector>

#include "cell.cuh"
#include "df64.cuh"
#include "krylov.h"
#include "level.h"
#include "pdl.cuh"
#include "qk_tables.h"
#include "tma.cuh"

namespace als {
namespace qk3 {

constexpr int K = 3;
constexpr int N1 = K + 1;          // nodes (and Gauss points) per axis and cell
constexpr int NB = N1 * N1 * N1;   // nodes per cell (64)
constexpr int NQ = NB;             // Gauss points per cell
constexpr int NPR = 10;            // pressure monomials per cell
constexpr int S1 = 2 * K - 1;      // star nodes per axis (5)
constexpr int SN = S1 * S1 * S1;   // star nodes (125)
constexpr int NS = 3 * SN;         // star dofs (375)
constexpr int NF = 2 * K + 1;      // fine lattice nodes per coarse cell and axis (7)
constexpr int CPB = 4;             // cells per block of the cell kernel (64 threads each)

__constant__ double cL[N1][N1], cD[N1][N1], cW[N1], cPSI[NQ][NPR], cPW[NF][N1];
// the FP32 cycle's copies (an FP64 operation costs ~70 FP32 ones here, conversions included)
// and the 3D point weights w_qx w_qy w_qz in both precisions
__constant__ float cLf[N1][N1], cDf[N1][N1], cPSIf[NQ][NPR], cPWf[NF][N1], cW3f[NQ];
__constant__ double cW3[NQ];
template <typename T> struct Tab;
template <> struct Tab<double> {
  static __device__ __forceinline__ double L(int q, int a) { return cL[q][a]; }
  static __device__ __forceinline__ double D(int q, int a) { return cD[q][a]; }
  static __device__ __forceinline__ double psi(int q, int p) { return cPSI[q][p]; }
  static __device__ __forceinline__ double pw(int f, int a) { return cPW[f][a]; }
  static __device__ __forceinline__ double w3(int q) { return cW3[q]; }
};
template <> struct Tab<float> {
  static __device__ __forceinline__ float L(int q, int a) { return cLf[q][a]; }
  static __device__ __forceinline__ float D(int q, int a) { return cDf[q][a]; }
  static __device__ __forceinline__ float psi(int q, int p) { return cPSIf[q][p]; }
  static __device__ __forceinline__ float pw(int f, int a) { return cPWf[f][a]; }
  static __device__ __forceinline__ float w3(int q) { return cW3f[q]; }
};
// per-level scalars of the cell kernel in its precision, formed on the host: the reference
// to physical derivative scales 2 / h_j, |J| = h0 h1 h2 / 8, and gamma
template <typename T>
struct CellScal {
  T s[3], wdet, gamma;
};
template <typename T>
static CellScal<T> cell_scal(const Geom& g, double gamma) {
  CellScal<T> c;
  for (int j = 0; j < 3; ++j) c.s[j] = (T)(2.0 / g.h[j]);
  c.wdet = (T)(0.125 * g.h[0] * g.h[1] * g.h[2]);
  c.gamma = (T)gamma;
  return c;
}

void ensure_tables() {
  static bool done = false;
  if (done) return;
  double G[N1], L[N1][N1], D[N1][N1], W[N1], PW[NF][N1], PSI[NQ][NPR];
  qk_tab::tables_1d(G, L, D, W, PW);
  const int ex[NPR][3] = {{0, 0, 0}, {1, 0, 0}, {0, 1, 0}, {0, 0, 1}, {2, 0, 0},
                          {1, 1, 0}, {1, 0, 1}, {0, 2, 0}, {0, 1, 1}, {0, 0, 2}};
  for (int q = 0; q < NQ; ++q) {
    const double x[3] = {G[q % N1], G[(q / N1) % N1], G[q / (N1 * N1)]};
    for (int p = 0; p < NPR; ++p) PSI[q][p] = pow(x[0], ex[p][0]) * pow(x[1], ex[p][1]) * pow(x[2], ex[p][2]);
  }
  cudaMemcpyToSymbol(cL, L, sizeof(L));
  cudaMemcpyToSymbol(cD, D, sizeof(D));
  cudaMemcpyToSymbol(cW, W, sizeof(W));
  cudaMemcpyToSymbol(cPSI, PSI, sizeof(PSI));
  cudaMemcpyToSymbol(cPW, PW, sizeof(PW));
  float Lf[N1][N1], Df[N1][N1], PSIf[NQ][NPR], PWf[NF][N1], W3f[NQ];
  double W3[NQ];
  for (int q = 0; q < N1; ++q)
    for (int a = 0; a < N1; ++a) { Lf[q][a] = (float)L[q][a]; Df[q][a] = (float)D[q][a]; }
  for (int q = 0; q < NQ; ++q) {
    for (int p = 0; p < NPR; ++p) PSIf[q][p] = (float)PSI[q][p];
    W3[q] = W[q % N1] * W[(q / N1) % N1] * W[q / (N1 * N1)];
    W3f[q] = (float)W3[q];
  }
  for (int f = 0; f < NF; ++f)
    for (int a = 0; a < N1; ++a) PWf[f][a] = (float)PW[f][a];
  cudaMemcpyToSymbol(cLf, Lf, sizeof(Lf));
  cudaMemcpyToSymbol(cDf, Df, sizeof(Df));
  cudaMemcpyToSymbol(cPSIf, PSIf, sizeof(PSIf));
  cudaMemcpyToSymbol(cPWf, PWf, sizeof(PWf));
  cudaMemcpyToSymbol(cW3f, W3f, sizeof(W3f));
  cudaMemcpyToSymbol(cW3, W3, sizeof(W3));
  done = true;
}

__device__ __forceinline__ bool bnd_node(const Geom& g, int i, int j, int k) {
  return i == 0 || i == g.nn[0] - 1 || j == 0 || j == g.nn[1] - 1 || k == 0 || k == g.nn[2] - 1;
}
__device__ __forceinline__ double wq_of(int q, double wdet) {
  return cW[q % N1] * cW[(q / N1) % N1] * cW[q / (N1 * N1)] * wdet;
}

// ---------------------------------------------------------------------------
// operator apply: 64 threads per cell.  Forward: u at the 64 nodes -> the 3 x 3 velocity
// gradient at the 64 points by contractions along x, y, z; then the pressure moments
// (B u)_p = -sum_q w |J| psi_p div u (a 64-thread reduction), the AL field
// gamma psi . W^-1 B u and the flux s_cj = w |J| (2 mu eps_cj - P delta_cj) (2 / h_j);
// backward: y_c(a) = sum_q sum_j s_cj d_j phi_a by the transposed contractions z, y, x.
// ---------------------------------------------------------------------------
template <typename T>
struct CellShared {
  T L[N1][N1], D[N1][N1];
  T psi[NQ][NPR];
  T wq[NQ];
  T b0[CPB][9][NB];
  T b1[CPB][9][NB];
  T red[CPB][2][NPR];
  T sp[CPB][NPR];
};

// the vertices whose stars contain lattice index i (|i - 3v| <= 2), two taps: v0 = i / 3, then
// v0 + 1 unless i = 3 v0; o: offset index in the star, 0 .. S1 - 1
struct StarTaps {
  int v[2], o[2];
  bool two;
  __device__ __forceinline__ explicit StarTaps(int i) {
    const int v0 = i / K, r = i - K * v0;
    v[0] = v0; o[0] = r + K - 1;
    v[1] = v0 + 1; o[1] = r - 1;
    two = r != 0;
  }
};

// z at node (i, j, k) = sum over the (up to 8) stars containing it, of their outputs sc, fixed order
template <typename T>
__device__ __forceinline__ T star_sum(const Geom& g, const T* __restrict__ sc, int comp, int i, int j, int k) {
  const StarTaps tx(i), ty(j), tz(k);
  T v[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int a = q & 1, b = (q >> 1) & 1, c = q >> 2;
    const bool ok = (a == 0 || tx.two) && (b == 0 || ty.two) && (c == 0 || tz.two);
    const int vid = tx.v[a] + g.nv[0] * (ty.v[b] + g.nv[1] * tz.v[c]);
    v[q] = ok ? sc[vid * NS + comp * SN + tx.o[a] + S1 * ty.o[b] + S1 * S1 * tz.o[c]] : T(0);
  }
  T acc = v[0];
#pragma unroll
  for (int q = 1; q < 8; ++q) acc += v[q];
  return acc;
}

// a warp's sums of NPR <= 16 values a lane; lane l < NPR returns that of value l (the columns are
// halved as the lanes are paired: 16 shuffles, where a tree per value takes 5 NPR)
template <typename T>
__device__ __forceinline__ T warp_moments(const T (&in)[NPR]) {
  static_assert(NPR <= 16, "sixteen columns");
  const int lane = threadIdx.x & 31;
  T v[16];
#pragma unroll
  for (int p = 0; p < 16; ++p) v[p] = p < NPR ? in[p] : T(0);
#pragma unroll
  for (int w = 8; w > 0; w >>= 1) {
    const bool up = (lane & w) != 0;
#pragma unroll
    for (int p = 0; p < w; ++p) {
      const T give = up ? v[p] : v[p + w];
      v[p] = (up ? v[p + w] : v[p]) + __shfl_xor_sync(0xffffffffu, give, w);
    }
  }
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 16);
}

// ZP: u is formed from the star outputs sc and stored to z, each node by the cell that owns it (the
// last cell also the upper ends).  One 12^3 three-level FP32 cycle: 1478 us, 1550 with a launch of its
// own for the node sums, plain launches of the cells, gathers and transfers, and a shuffle tree per
// pressure moment.
template <typename T, int MODE, bool ZP>
__global__ void __launch_bounds__(64 * CPB) k_qk3_cells(Geom g, CellScal<T> cs, const T* __restrict__ x,
                                                        const T* __restrict__ mu, const T* __restrict__ winv,
                                                        const T* __restrict__ p_in, T* __restrict__ p_out,
                                                        T* __restrict__ ebuf, const T* __restrict__ sc,
                                                        T* __restrict__ z) {
  constexpr bool RAW = (MODE & OP_RAW) != 0, VISC = (MODE & OP_VISC) != 0, AL = (MODE & OP_AL) != 0;
  constexpr bool BT = (MODE & OP_BT) != 0, BO = (MODE & OP_B) != 0;
  constexpr bool NEED_U = VISC || AL || BO, NEED_FLUX = VISC || AL || BT;
  __shared__ CellShared<T> sh;
  const int tid = threadIdx.x;
  if (tid < N1 * N1) {
    sh.L[tid / N1][tid % N1] = Tab<T>::L(tid / N1, tid % N1);
    sh.D[tid / N1][tid % N1] = Tab<T>::D(tid / N1, tid % N1);
  }
  for (int e = tid; e < NQ * NPR; e += blockDim.x) sh.psi[e / NPR][e % NPR] = Tab<T>::psi(e / NPR, e % NPR);
  if (tid < NQ) sh.wq[tid] = Tab<T>::w3(tid) * cs.wdet;
  const int w = tid >> 6, t = tid & 63, t0 = t & 3, t1 = (t >> 2) & 3, t2 = t >> 4;
  const long long cell = (long long)blockIdx.x * CPB + w;
  const bool valid = cell < g.ncells;
  const int cx = valid ? (int)(cell % g.n[0]) : 0;
  const int cy = valid ? (int)((cell / g.n[0]) % g.n[1]) : 0;
  const int cz = valid ? (int)(cell / ((long long)g.n[0] * g.n[1])) : 0;
  const T sx = cs.s[0], sy = cs.s[1], sz = cs.s[2];
  T(*b0)[NB] = sh.b0[w];
  T(*b1)[NB] = sh.b1[w];
  const T m2 = (VISC && valid) ? T(2) * mu[cell * NQ + t] : T(0);
  pdl_wait();
  pdl_trigger();
  if constexpr (ZP) {
    const int i = K * cx + t0, j = K * cy + t1, k = K * cz + t2;
    const bool in = valid && !bnd_node(g, i, j, k);
    const bool own = valid && (t0 < K || cx == g.n[0] - 1) && (t1 < K || cy == g.n[1] - 1) && (t2 < K || cz == g.n[2] - 1);
    T v[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) v[c] = in ? star_sum<T>(g, sc, c, i, j, k) : T(0);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      b0[c][t] = v[c];
      if (own) z[c * (int)g.N + i + g.nn[0] * (j + g.nn[1] * k)] = v[c];
    }
  } else {
    const int i = K * cx + t0, j = K * cy + t1, k = K * cz + t2;
    const bool bnd = bnd_node(g, i, j, k);
    const long long nd = node_id(g, i, j, k);
    for (int c = 0; c < 3; ++c) b0[c][t] = (valid && NEED_U && (RAW || !bnd)) ? x[c * g.N + nd] : T(0);
  }
  __syncthreads();
  // x: (ax, ay, az) -> (qx, ay, az): A = L u, B = D u
  {
    const int qx = t0, base = N1 * t1 + N1 * N1 * t2;
    for (int c = 0; c < 3; ++c) {
      T a = T(0), b = T(0);
#pragma unroll
      for (int ax = 0; ax < N1; ++ax) {
        const T u = b0[c][base + ax];
        a += sh.L[qx][ax] * u;
        b += sh.D[qx][ax] * u;
      }
      b1[c][t] = a;
      b1[3 + c][t] = b;
    }
  }
  __syncthreads();
  // y: (qx, ay, az) -> (qx, qy, az): AL = L A, AD = D A, BL = L B
  {
    const int qy = t1, base = t0 + N1 * N1 * t2;
    for (int c = 0; c < 3; ++c) {
      T al = T(0), ad = T(0), bl = T(0);
#pragma unroll
      for (int ay = 0; ay < N1; ++ay) {
        const T a = b1[c][base + N1 * ay], b = b1[3 + c][base + N1 * ay];
        al += sh.L[qy][ay] * a;
        ad += sh.D[qy][ay] * a;
        bl += sh.L[qy][ay] * b;
      }
      b0[c][t] = al;
      b0[3 + c][t] = ad;
      b0[6 + c][t] = bl;
    }
  }
  __syncthreads();
  // z: (qx, qy, az) -> (qx, qy, qz): the gradient G[c][j] at point q = t
  T G[3][3];
  {
    const int qz = t2, base = t0 + N1 * t1;
    for (int c = 0; c < 3; ++c) {
      T gx = T(0), gy = T(0), gz = T(0);
#pragma unroll
      for (int az = 0; az < N1; ++az) {
        const int o = base + N1 * N1 * az;
        gx += sh.L[qz][az] * b0[6 + c][o];
        gy += sh.L[qz][az] * b0[3 + c][o];
        gz += sh.D[qz][az] * b0[c][o];
      }
      G[c][0] = gx * sx;
      G[c][1] = gy * sy;
      G[c][2] = gz * sz;
    }
  }
  const int q = t;
  const T div = G[0][0] + G[1][1] + G[2][2];
  T P = T(0);   // gamma pi + p_in at the point
  if (AL || BO) {
    // (B u)_p over the cell's 64 points: warp sums, then the two warps in a fixed order
    T bu[NPR];
#pragma unroll
    for (int p = 0; p < NPR; ++p) bu[p] = -sh.wq[q] * sh.psi[q][p] * div;
    const T tot = warp_moments<T>(bu);
    if ((t & 31) < NPR) sh.red[w][t >> 5][t & 31] = tot;
    __syncthreads();
    for (int p = 0; p < NPR; ++p) bu[p] = sh.red[w][0][p] + sh.red[w][1][p];
    if (BO && valid && t == 0)
      for (int p = 0; p < NPR; ++p) p_out[cell * NPR + p] = bu[p];
    if (AL) {
      if (valid && t < NPR) {
        const T* Wc = winv + cell * NPR * NPR;
        T s = T(0);
        for (int r = 0; r < NPR; ++r) s += Wc[t * NPR + r] * bu[r];
        sh.sp[w][t] = s;
      }
      __syncthreads();
      T pi = T(0);
      if (valid)
        for (int p = 0; p < NPR; ++p) pi += sh.psi[q][p] * sh.sp[w][p];
      P += cs.gamma * pi;
    }
  }
  if (BT && valid)
    for (int p = 0; p < NPR; ++p) P += sh.psi[q][p] * p_in[cell * NPR + p];
  if (!NEED_FLUX) return;   // uniform over the block
  {
    const T wq = sh.wq[q];
    const T sj[3] = {sx, sy, sz};
    for (int c = 0; c < 3; ++c)
      for (int j = 0; j < 3; ++j) {
        const T eps = T(0.5) * (G[c][j] + G[j][c]);
        b1[3 * c + j][t] = wq * (m2 * eps - (c == j ? P : T(0))) * sj[j];
      }
  }
  __syncthreads();
  // z^T: (qx, qy, qz) -> (qx, qy, az): T0 = L s_c0, T1 = L s_c1, T2 = D s_c2
  {
    const int az = t2, base = t0 + N1 * t1;
    for (int c = 0; c < 3; ++c) {
      T s0 = T(0), s1 = T(0), s2 = T(0);
#pragma unroll
      for (int qz = 0; qz < N1; ++qz) {
        const int o = base + N1 * N1 * qz;
        s0 += sh.L[qz][az] * b1[3 * c][o];
        s1 += sh.L[qz][az] * b1[3 * c + 1][o];
        s2 += sh.D[qz][az] * b1[3 * c + 2][o];
      }
      b0[3 * c][t] = s0;
      b0[3 * c + 1][t] = s1;
      b0[3 * c + 2][t] = s2;
    }
  }
  __syncthreads();
  // y^T: (qx, qy, az) -> (qx, ay, az): V = L T0 (x derivative still to come), W = D T1 + L T2
  {
    const int ay = t1, base = t0 + N1 * N1 * t2;
    for (int c = 0; c < 3; ++c) {
      T v = T(0), wv = T(0);
#pragma unroll
      for (int qy = 0; qy < N1; ++qy) {
        const int o = base + N1 * qy;
        v += sh.L[qy][ay] * b0[3 * c][o];
        wv += sh.D[qy][ay] * b0[3 * c + 1][o] + sh.L[qy][ay] * b0[3 * c + 2][o];
      }
      b1[c][t] = v;
      b1[3 + c][t] = wv;
    }
  }
  __syncthreads();
  // x^T: (qx, ay, az) -> (ax, ay, az): y_c = D V + L W
  if (valid) {
    const int ax = t0, base = N1 * t1 + N1 * N1 * t2;
    for (int c = 0; c < 3; ++c) {
      T y = T(0);
#pragma unroll
      for (int qx = 0; qx < N1; ++qx) y += sh.D[qx][ax] * b1[c][base + qx] + sh.L[qx][ax] * b1[3 + c][base + qx];
      ebuf[(cell * 3 + c) * NB + t] = y;
    }
  }
}

// the cells containing lattice index i along an axis of n cells, two taps in a fixed order:
// (c - 1, local K) where i is the cell corner between c - 1 and c, then (c, i - K c)
struct CellTaps {
  int c[2], a[2];
  bool ok[2];
  __device__ __forceinline__ CellTaps(int i, int n) {
    const int c0 = i / K, r = i - K * c0;
    c[0] = c0 - 1; a[0] = K; ok[0] = r == 0 && c0 > 0;
    c[1] = c0; a[1] = r; ok[1] = c0 < n;
  }
};

// component and lattice coordinates of vector entry t (32-bit: entries stay below 2^31)
__device__ __forceinline__ void entry_coords(const Geom& g, unsigned t, int& comp, int& i, int& j, int& k) {
  const unsigned N = (unsigned)g.N, nx = (unsigned)g.nn[0], ny = (unsigned)g.nn[1];
  comp = (int)(t / N);
  const unsigned nd = t - comp * N, r = nd / nx;
  i = (int)(nd - r * nx);
  k = (int)(r / ny);
  j = (int)(r - k * ny);
}

// y(node) = sum of the staged cell outputs of the (up to 8) cells containing it, fixed
// order; keep_bnd: y = x at Dirichlet nodes; raw: no Dirichlet treatment.  Predicated taps, so
// that all loads issue at once.
template <typename T>
__device__ __forceinline__ T gather_value(const Geom& g, const T* __restrict__ ebuf, const T* __restrict__ x,
                                          unsigned t, int keep_bnd, int raw) {
  int comp, i, j, k;
  entry_coords(g, t, comp, i, j, k);
  if (bnd_node(g, i, j, k) && !raw) return keep_bnd ? x[t] : T(0);
  const CellTaps tx(i, g.n[0]), ty(j, g.n[1]), tz(k, g.n[2]);
  T v[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int a = q & 1, b = (q >> 1) & 1, c = q >> 2;
    const int cell = tx.c[a] + g.n[0] * (ty.c[b] + g.n[1] * tz.c[c]);
    v[q] = tx.ok[a] && ty.ok[b] && tz.ok[c]
               ? ebuf[(cell * 3 + comp) * NB + tx.a[a] + N1 * ty.a[b] + N1 * N1 * tz.a[c]]
               : T(0);
  }
  T acc = v[0];
#pragma unroll
  for (int q = 1; q < 8; ++q) acc += v[q];
  return acc;
}

template <typename T>
__global__ void k_qk3_gather(Geom g, const T* __restrict__ ebuf, const T* __restrict__ x, T* __restrict__ y,
                             int keep_bnd, int raw) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  pdl_wait();
  pdl_trigger();
  if (t >= 3u * (unsigned)g.N) return;
  y[t] = gather_value<T>(g, ebuf, x, t, keep_bnd, raw);
}

// The gather fused with the reduction that consumes its result, as for order 2 (the
// GMRES smoother's Arnoldi step): y = b + sigma A x (b NULL: sigma A x; Dirichlet rows of
// A x are x, the identity);  block partials of V_j . y, j < k, or, start = 1, of |y|^2.
// PER entries a thread, 256 apart: large levels take kEpiPer, which keeps the partials that
// every block of the Gram-Schmidt kernel adds at about a thousand.
template <typename T, int PER>
__global__ void __launch_bounds__(RED_THREADS) k_qk3_gather_epi(Geom g, const T* __restrict__ ebuf,
                                                               const T* __restrict__ x, T* __restrict__ y,
                                                               const T* __restrict__ b, double sigma, int k,
                                                               const T* __restrict__ V, long long ld, int start,
                                                               GmresDev sd) {
  T acc[KMAXB];
#pragma unroll
  for (int jj = 0; jj < KMAXB; ++jj) acc[jj] = T(0);
  const unsigned n = 3 * (unsigned)g.N, t0 = blockIdx.x * (RED_THREADS * PER) + threadIdx.x;
  // the basis columns come from kernels before the predecessor: ahead of the wait
  T vp[PER][KMAXB];
#pragma unroll
  for (int q = 0; q < PER; ++q)
#pragma unroll
    for (int jj = 0; jj < KMAXB; ++jj)
      vp[q][jj] = !start && jj < k && t0 + q * RED_THREADS < n ? __ldcg(V + (long long)jj * ld + t0 + q * RED_THREADS) : T(0);
  pdl_wait();
  pdl_trigger();
  T v[PER];
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const unsigned t = t0 + q * RED_THREADS;
    v[q] = t < n ? (b ? b[t] : T(0)) + (T)sigma * gather_value<T>(g, ebuf, x, t, 1, 0) : T(0);
  }
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const unsigned t = t0 + q * RED_THREADS;
    if (t < n) y[t] = v[q];
    if (start) {
      acc[0] += v[q] * v[q];
    } else {
#pragma unroll
      for (int jj = 0; jj < KMAXB; ++jj)
        if (jj < k) acc[jj] += vp[q][jj] * v[q];
    }
  }
  store_partials<T>(sd, start, k, acc, blockIdx.x, gridDim.x);
}

template <typename T, int MODE, bool ZP = false>
static void launch_cells(const LevelDev& L, double gamma, const void* x, const void* p_in, void* p_out, cudaStream_t s,
                         const void* sc = nullptr, void* z = nullptr) {
  const T* mu = std::is_same<T, double>::value ? (const T*)L.coef64 : (const T*)L.coef32;
  const T* winv = std::is_same<T, double>::value ? (const T*)L.winv64 : (const T*)L.winv32;
  launch_pdl(k_qk3_cells<T, MODE, ZP>, (unsigned)((L.g.ncells + CPB - 1) / CPB), 64 * CPB, 0, s, L.g,
             cell_scal<T>(L.g, gamma), (const T*)x, mu, winv, (const T*)p_in, (T*)p_out, (T*)L.ebuf, (const T*)sc, (T*)z);
}

template <typename T, int MODE>
static void apply_mode(const LevelDev& L, double gamma, const void* x, void* y, const void* p_in, void* p_out,
                       cudaStream_t s) {
  constexpr bool NEED_FLUX = (MODE & (OP_VISC | OP_AL | OP_BT)) != 0;
  launch_cells<T, MODE>(L, gamma, x, p_in, p_out, s);
  if (NEED_FLUX) {
    const int keep = ((MODE & OP_VISC) && !(MODE & OP_RAW)) ? 1 : 0;
    launch_pdl(k_qk3_gather<T>, (unsigned)((3 * L.g.N + 255) / 256), 256, 0, s, L.g, (const T*)L.ebuf, (const T*)x, (T*)y,
               keep, (MODE & OP_RAW) ? 1 : 0);
  }
  count_launch(NEED_FLUX ? 2 : 1);
}

template <typename T>
static void apply_t(const LevelDev& L, int mode, double gamma, const void* x, void* y, const void* p_in, void* p_out,
                    cudaStream_t s) {
  switch (mode) {
    case OP_VISC | OP_AL: apply_mode<T, OP_VISC | OP_AL>(L, gamma, x, y, p_in, p_out, s); break;
    case OP_AL: apply_mode<T, OP_AL>(L, gamma, x, y, p_in, p_out, s); break;
    case OP_B: apply_mode<T, OP_B>(L, gamma, x, y, p_in, p_out, s); break;
    case OP_BT: apply_mode<T, OP_BT>(L, gamma, x, y, p_in, p_out, s); break;
    case OP_VISC | OP_AL | OP_BT | OP_B: apply_mode<T, OP_VISC | OP_AL | OP_BT | OP_B>(L, gamma, x, y, p_in, p_out, s); break;
    case OP_VISC | OP_AL | OP_RAW: apply_mode<T, OP_VISC | OP_AL | OP_RAW>(L, gamma, x, y, p_in, p_out, s); break;
    case OP_B | OP_RAW: apply_mode<T, OP_B | OP_RAW>(L, gamma, x, y, p_in, p_out, s); break;
    default: break;
  }
}

template <typename T>
static void apply_epi_t(const LevelDev& L, double gamma, const void* x, void* y, const ApplyEpi& e, cudaStream_t s,
                        cudaEvent_t e0, cudaEvent_t e1) {
  // External records become event-record nodes when the stream is being captured
  if (e0) cudaEventRecordWithFlags(e0, s, cudaEventRecordExternal);
  if (std::is_same<T, float>::value && e.pout)   // x = z formed from the star outputs; z stored on the way
    launch_cells<float, OP_VISC | OP_AL, true>(L, gamma, nullptr, nullptr, nullptr, s, e.pout, const_cast<void*>(x));
  else
    launch_cells<T, OP_VISC | OP_AL>(L, gamma, x, nullptr, nullptr, s);
  if (e1) cudaEventRecordWithFlags(e1, s, cudaEventRecordExternal);
  const auto kernel = qk_epi_per(L) == 1 ? k_qk3_gather_epi<T, 1> : k_qk3_gather_epi<T, kEpiPer>;
  launch_pdl(kernel, qk_epi_blocks(L), RED_THREADS, 0, s, L.g, (const T*)L.ebuf, (const T*)x, (T*)y, (const T*)e.b,
             e.sigma, e.k, (const T*)e.V, e.ld, e.start, e.st);
  count_launch(2);
}

// F_(c,a) = sum_q |J| w_q f_c(x_q) phi_a(x_q), staged per cell, summed per node; f is
// [cell][q][3]
__global__ void k_qk3_load(Geom g, const double* __restrict__ f, double* __restrict__ ebuf) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= g.ncells * 3 * NB) return;
  const long long cell = t / (3 * NB);
  const int e = (int)(t % (3 * NB)), comp = e / NB, a = e % NB;
  const int ax = a % N1, ay = (a / N1) % N1, az = a / (N1 * N1);
  const double wdet = 0.125 * g.h[0] * g.h[1] * g.h[2];
  double acc = 0.0;
  for (int q = 0; q < NQ; ++q) {
    const double phi = cL[q % N1][ax] * cL[(q / N1) % N1][ay] * cL[q / (N1 * N1)][az];
    acc += wq_of(q, wdet) * f[(cell * NQ + q) * 3 + comp] * phi;
  }
  ebuf[(cell * 3 + comp) * NB + a] = acc;
}

// ---------------------------------------------------------------------------
// per-cell mass blocks: M_K(1/mu)^-1 and M_K^-1 (10 x 10, Gauss-Jordan), the augmentation
// weight's inverse W^-1 (W = M_p or M_p(1/mu)) and the Schur blocks S of Eq. (P1P2):
// P1: M_K(1/mu)^-1 + gamma M_K^-1, P2: (1 + gamma) M_K(1/mu)^-1.  One thread per cell.
// ---------------------------------------------------------------------------
__device__ void inv10(double (&A)[NPR][NPR], DevStatus* st, long long where) {
  double Iv[NPR][NPR];
  for (int i = 0; i < NPR; ++i)
    for (int j = 0; j < NPR; ++j) Iv[i][j] = i == j ? 1.0 : 0.0;
  for (int k = 0; k < NPR; ++k) {
    const double pv = A[k][k];
    if (!(pv > 0.0)) { report(st, 4 /* ALS_ENOTSPD */, where); return; }
    const double ip = 1.0 / pv;
    for (int j = 0; j < NPR; ++j) { A[k][j] *= ip; Iv[k][j] *= ip; }
    for (int i = 0; i < NPR; ++i) {
      if (i == k) continue;
      const double f = A[i][k];
      for (int j = 0; j < NPR; ++j) { A[i][j] -= f * A[k][j]; Iv[i][j] -= f * Iv[k][j]; }
    }
  }
  for (int i = 0; i < NPR; ++i)
    for (int j = 0; j < NPR; ++j) A[i][j] = Iv[i][j];
}

__global__ void k_qk3_mass(Geom g, double gamma, const double* __restrict__ mu, int w_mu, int variant,
                           double* __restrict__ winv64, float* __restrict__ winv32, double* __restrict__ S,
                           DevStatus* st) {
  const long long cell = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (cell >= g.ncells) return;
  const double wdet = 0.125 * g.h[0] * g.h[1] * g.h[2];
  double Mm[NPR][NPR], M[NPR][NPR];
  for (int p = 0; p < NPR; ++p)
    for (int r = 0; r < NPR; ++r) { Mm[p][r] = 0.0; M[p][r] = 0.0; }
  for (int q = 0; q < NQ; ++q) {
    const double wq = wq_of(q, wdet);
    const double im = 1.0 / mu[cell * NQ + q];
    for (int p = 0; p < NPR; ++p)
      for (int r = 0; r < NPR; ++r) {
        M[p][r] += wq * cPSI[q][p] * cPSI[q][r];
        Mm[p][r] += wq * im * cPSI[q][p] * cPSI[q][r];
      }
  }
  inv10(Mm, st, cell);
  inv10(M, st, cell);
  for (int p = 0; p < NPR; ++p)
    for (int r = 0; r < NPR; ++r) {
      const double wv = w_mu ? Mm[p][r] : M[p][r];
      if (winv64) winv64[cell * NPR * NPR + p * NPR + r] = wv;
      if (winv32) winv32[cell * NPR * NPR + p * NPR + r] = (float)wv;
      if (S) S[cell * NPR * NPR + p * NPR + r] = variant == 0 ? Mm[p][r] + gamma * M[p][r] : (1.0 + gamma) * Mm[p][r];
    }
}

// ---------------------------------------------------------------------------
// vertex stars: setup (assembly from the star's 8 cells into a workspace row block in
// global memory, block Gauss-Jordan inversion, FP64 packed-by-diagonals and its FP32
// rounding), products, node gather
// ---------------------------------------------------------------------------
// star entry e = comp * 125 + (ox + 2) + 5 (oy + 2) + 25 (oz + 2) of vertex v: node 3v + o
__device__ __forceinline__ bool star_node(const Geom& g, int vx, int vy, int vz, int e, long long& nd) {
  const int o = e % SN;
  const int i = K * vx + o % S1 - (K - 1), j = K * vy + (o / S1) % S1 - (K - 1), k = K * vz + o / (S1 * S1) - (K - 1);
  if (i <= 0 || i >= g.nn[0] - 1 || j <= 0 || j >= g.nn[1] - 1 || k <= 0 || k >= g.nn[2] - 1) return false;
  nd = node_id(g, i, j, k);
  return true;
}

constexpr int LDM = NS + 1;   // row stride of a star matrix in the workspace (doubles)
// FP32 star storage (k_qk3_stars): the free dofs' inverse in 15 x 15 blocks (I, J), I <= J,
// off-diagonal blocks first (row-major over I < J), then the diagonal ones (upper triangle,
// 120 entries).  Interleaved by block in quads of four entries, so that the threads of a star,
// one block each, read consecutive quads: quads 0..29 of all blocks, then quads 30..56 of the
// off-diagonal ones (225 entries and three zeros).  An interior vertex's star has 375 free dofs
// (25 x 25 blocks); a face, edge or corner vertex's only 150, 60 or 24, which is all that is
// stored of it.
constexpr int SB = 15, SQ1 = 30, SQ2 = 27;
struct StarBlocks {
  int nbr, nblk, noff;   // block rows, blocks, off-diagonal blocks
  __host__ __device__ constexpr explicit StarBlocks(int m)
      : nbr((m + SB - 1) / SB), nblk(((m + SB - 1) / SB) * ((m + SB - 1) / SB + 1) / 2),
        noff(((m + SB - 1) / SB) * ((m + SB - 1) / SB - 1) / 2) {}
  __host__ __device__ constexpr int q2() const { return 4 * SQ1 * nblk; }
  __host__ __device__ constexpr int entries() const { return 4 * (SQ1 * nblk + SQ2 * noff); }
  __device__ __forceinline__ void block_of(int b, int& I, int& J) const {
    if (b >= noff) {
      I = J = b - noff;
    } else {
      int rem = b;
      I = 0;
      while (rem >= nbr - 1 - I) { rem -= nbr - 1 - I; ++I; }
      J = I + 1 + rem;
    }
  }
};
constexpr int kFullRows = StarBlocks(NS).nbr, kFullBlocks = StarBlocks(NS).nblk, kFullOff = StarBlocks(NS).noff;
constexpr int kFullEntries = StarBlocks(NS).entries();

// the free dofs of a vertex's star: a box of node offsets, all five where the vertex is interior
// along the axis, the two inward ones where it lies on the boundary
struct StarBox {
  int lo[3], cnt[3], m;
  __host__ __device__ StarBox(const Geom& g, int vx, int vy, int vz) {
    const int v[3] = {vx, vy, vz};
    m = 3;
    for (int a = 0; a < 3; ++a) {
      lo[a] = v[a] == 0 ? K : 0;
      cnt[a] = v[a] == 0 || v[a] == g.nv[a] - 1 ? K - 1 : S1;
      m *= cnt[a];
    }
  }
  // star entry (component-major, offsets x-fastest) of free dof a; increases with a
  __device__ __forceinline__ int entry(int a) const {
    const int ix = a % cnt[0], q = a / cnt[0], iy = q % cnt[1], q2 = q / cnt[1], iz = q2 % cnt[2], c = q2 / cnt[2];
    return c * SN + (lo[0] + ix) + S1 * (lo[1] + iy) + S1 * S1 * (lo[2] + iz);
  }
};
constexpr int BB = 16;        // pivots per Gauss-Jordan pass
constexpr int SETUP_THREADS = 256;
// shared memory of the setup kernel (doubles): the assembly's tables or the elimination's
// pivot block and panels, whichever is larger
constexpr int ASM_DOUBLES = NQ * 27 * 3 + NQ + 2 * NPR * 81 + 8 * 3 * 3;
constexpr int GJ_DOUBLES = BB * BB + 2 * BB * NS + 2 * BB;
constexpr int SETUP_DOUBLES = ASM_DOUBLES > GJ_DOUBLES ? ASM_DOUBLES : GJ_DOUBLES;
constexpr size_t SETUP_SMEM = sizeof(double) * SETUP_DOUBLES + 16;

// entry e (0 <= e < N (N + 1) / 2) of the upper triangle of an N x N matrix, N odd, as
// (i, j), i <= j: the rows are taken in pairs (p, N - 1 - p), p < (N - 1) / 2, of N + 1
// entries together, then the middle row (consecutive e: consecutive j)
template <int N>
__device__ __forceinline__ void tri_entry(int e, int& i, int& j) {
  static_assert(N % 2 == 1, "odd order");
  constexpr int HALF = (N - 1) / 2;
  const int p = e / (N + 1), off = e - p * (N + 1);
  if (p < HALF) {
    if (off < N - p) { i = p; j = p + off; }
    else { i = N - 1 - p; j = i + off - (N - p); }
  } else {
    i = HALF;
    j = HALF + off;
  }
}

// One CTA per star at a time (persistent over the stars v = blockIdx.x, += gridDim.x), its
// star matrix in ws + blockIdx.x * NS * LDM.
// RM: the arithmetic of the elimination, double or DF64 (double-float, about 48 bits, on
// the FP32 pipes; the assembly is FP64 either way)
template <typename RM>
__global__ void __launch_bounds__(SETUP_THREADS) k_qk3_star_setup(Geom g, double gamma, const double* __restrict__ mu,
                                                                  const double* __restrict__ winv,
                                                                  double* __restrict__ ws, double* __restrict__ inv64,
                                                                  int pstride,
                                                                  DevStatus* st) {
  static_assert(sizeof(RM) == sizeof(double), "the workspace holds 8-byte entries");
  using Ops = RealOps<RM>;
  extern __shared__ double smem[];
  __shared__ int s_bad;
  const int tid = threadIdx.x, nt = blockDim.x;
  double* M = ws + (long long)blockIdx.x * NS * LDM;
  const double sx = 2.0 / g.h[0], sy = 2.0 / g.h[1], sz = 2.0 / g.h[2];
  const double wdet = 0.125 * g.h[0] * g.h[1] * g.h[2];
  for (long long v = blockIdx.x; v < g.nverts; v += gridDim.x) {
    const int vx = (int)(v % g.nv[0]), vy = (int)((v / g.nv[0]) % g.nv[1]), vz = (int)(v / ((long long)g.nv[0] * g.nv[1]));
    if (tid == 0) s_bad = 0;
    for (int e = tid; e < NS * LDM; e += nt) M[e] = 0.0;
    __syncthreads();
    // ---- assembly: the cells (cx, cy, cz) in {v-1, v}^3 inside the mesh
    double* gq = smem;                      // [q][n][3]: d_j phi_n at q, the cell's 27 star nodes n
    double* wm = gq + NQ * 27 * 3;          // [q]: w |J| mu
    double* Bm = wm + NQ;                   // [p][c * 27 + n]: -sum_q w |J| psi_p d_c phi_n
    double* WB = Bm + NPR * 81;             // W^-1 Bm
    for (int cc = 0; cc < 8; ++cc) {
      const int cx = vx - 1 + (cc & 1), cy = vy - 1 + ((cc >> 1) & 1), cz = vz - 1 + (cc >> 2);
      if (cx < 0 || cy < 0 || cz < 0 || cx >= g.n[0] || cy >= g.n[1] || cz >= g.n[2]) continue;   // uniform
      const long long cell = (long long)cx + (long long)g.n[0] * ((long long)cy + (long long)g.n[1] * cz);
      // the star's nodes in this cell: local index a = m + off per axis, m = 0..2
      const int offx = cx == vx - 1 ? 1 : 0, offy = cy == vy - 1 ? 1 : 0, offz = cz == vz - 1 ? 1 : 0;
      for (int e = tid; e < NQ * 27; e += nt) {
        const int q = e / 27, n = e % 27;
        const int ax = n % 3 + offx, ay = (n / 3) % 3 + offy, az = n / 9 + offz;
        const int qx = q % N1, qy = (q / N1) % N1, qz = q / (N1 * N1);
        gq[e * 3 + 0] = cD[qx][ax] * cL[qy][ay] * cL[qz][az] * sx;
        gq[e * 3 + 1] = cL[qx][ax] * cD[qy][ay] * cL[qz][az] * sy;
        gq[e * 3 + 2] = cL[qx][ax] * cL[qy][ay] * cD[qz][az] * sz;
      }
      for (int q = tid; q < NQ; q += nt) wm[q] = wq_of(q, wdet) * mu[cell * NQ + q];
      __syncthreads();
      for (int e = tid; e < NPR * 81; e += nt) {
        const int p = e / 81, j = e % 81, c = j / 27, n = j % 27;
        double acc = 0.0;
        for (int q = 0; q < NQ; ++q) acc -= wq_of(q, wdet) * cPSI[q][p] * gq[(q * 27 + n) * 3 + c];
        Bm[e] = acc;
      }
      __syncthreads();
      const double* Wc = winv + cell * NPR * NPR;
      for (int e = tid; e < NPR * 81; e += nt) {
        const int p = e / 81, j = e % 81;
        double acc = 0.0;
        for (int r = 0; r < NPR; ++r) acc += Wc[p * NPR + r] * Bm[r * 81 + j];
        WB[e] = acc;
      }
      __syncthreads();
      // node pairs: H[a][b] = sum_q w |J| mu d_a phi_ni d_b phi_nj; the element entry of
      // (ci, ni), (cj, nj) is 2 mu eps(phi_ni e_ci) : eps(phi_nj e_cj) integrated,
      // = delta_(ci cj) trace H + H[cj][ci], plus gamma (B^T W^-1 B)
      for (int e = tid; e < 27 * 28 / 2; e += nt) {   // unordered node pairs ni <= nj
        int ni, nj;
        tri_entry<27>(e, ni, nj);
        double H[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
        for (int q = 0; q < NQ; ++q) {
          const double* gi = gq + (q * 27 + ni) * 3;
          const double* gj = gq + (q * 27 + nj) * 3;
          const double wv = wm[q];
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            const double wa = wv * gi[a];
#pragma unroll
            for (int b = 0; b < 3; ++b) H[a][b] += wa * gj[b];
          }
        }
        const double tr = H[0][0] + H[1][1] + H[2][2];
        const int sni = (ni % 3 + offx + K * cx - K * vx + 2) + S1 * ((ni / 3) % 3 + offy + K * cy - K * vy + 2) +
                        S1 * S1 * (ni / 9 + offz + K * cz - K * vz + 2);
        const int snj = (nj % 3 + offx + K * cx - K * vx + 2) + S1 * ((nj / 3) % 3 + offy + K * cy - K * vy + 2) +
                        S1 * S1 * (nj / 9 + offz + K * cz - K * vz + 2);
        // the 9 entries of the node block (ni, nj), each into the upper triangle (the
        // block (nj, ni) holds their transposes; for ni == nj only ci <= cj)
        for (int ci = 0; ci < 3; ++ci)
          for (int cj = 0; cj < 3; ++cj) {
            if (ni == nj && ci > cj) continue;
            double al = 0.0;
            for (int p = 0; p < NPR; ++p) al += Bm[p * 81 + ci * 27 + ni] * WB[p * 81 + cj * 27 + nj];
            const int si = ci * SN + sni, sj = cj * SN + snj;
            const int lo = si < sj ? si : sj, hi = si < sj ? sj : si;
            M[(long long)lo * LDM + hi] += (ci == cj ? tr : 0.0) + H[cj][ci] + gamma * al;
          }
      }
      __syncthreads();
    }
    // identity rows and columns at absent and Dirichlet nodes; the entries in the
    // elimination's arithmetic RM from here on (each thread converts its own entries).
    // From here only the upper triangle i <= j is kept (see the elimination below).
    RM* Mr = reinterpret_cast<RM*>(M);
    for (int e = tid; e < NS * (NS + 1) / 2; e += nt) {
      int i, j;
      tri_entry<NS>(e, i, j);
      long long nd;
      const bool fi = star_node(g, vx, vy, vz, i, nd), fj = star_node(g, vx, vy, vz, j, nd);
      const double val = (!fi || !fj) ? (i == j ? 1.0 : 0.0) : M[(long long)i * LDM + j];
      Mr[(long long)i * LDM + j] = Ops::from(val);
    }
    __syncthreads();
    // ---- block Gauss-Jordan inversion in place on the upper triangle (SPD: the pivot
    // blocks are Schur complements, no pivoting).  Per pass over pivots K = [k0, k0 + b):
    // Dk = M_KK^-1, C = M_.K (column panel), R = Dk M_K. (row panel); then M_KK = Dk,
    // M_Kj = R_j, M_iK = -C_i Dk, M_ij -= C_i R_j.  With s_x = -1 for the indices swept
    // so far and +1 for the others, every pass keeps M_ji = s_i s_j M_ij, so the upper
    // triangle determines the rest: X_x = M(min(x, K), max(x, K)) is C_x, and the raw row
    // panel is sigma_x X_x (sigma_x = -1 for x < k0, +1 beyond K).  With Y_x = Dk X_x the
    // pass sets M_ij -= sigma_j X_i . Y_j (i <= j outside K), M_iK = -Y_i (i < k0),
    // M_Kj = Y_j (j beyond K), M_KK = Dk; at the end all signs agree and M is A^-1.
    RM* Dk = reinterpret_cast<RM*>(smem);   // [BB][BB]
    RM* Yp = Dk + BB * BB;                  // [BB][NS]
    RM* C = Yp + BB * NS;                   // [NS][BB]: X
    RM* rowk = C + NS * BB;                 // [BB]
    RM* colk = rowk + BB;                   // [BB]
    const RM zero = Ops::from(0.0), one = Ops::from(1.0);
    for (int k0 = 0; k0 < NS; k0 += BB) {
      const int b = NS - k0 < BB ? NS - k0 : BB;
      for (int e = tid; e < BB * BB; e += nt) {
        const int m = e / BB, l = e % BB, lo = m < l ? m : l, hi = m < l ? l : m;
        Dk[e] = (m < b && l < b) ? Mr[(long long)(k0 + lo) * LDM + k0 + hi] : (m == l ? one : zero);
      }
      for (int e = tid; e < NS * BB; e += nt) {
        const int x = e / BB, l = e % BB, k = k0 + l;
        const bool inK = x >= k0 && x < k0 + b;
        C[e] = (l < b && !inK) ? (x < k ? Mr[(long long)x * LDM + k] : Mr[(long long)k * LDM + x]) : zero;
      }
      __syncthreads();
      for (int kk = 0; kk < b; ++kk) {   // scalar Gauss-Jordan on the pivot block
        const RM pv = Dk[kk * BB + kk];
        const bool ok = pv > 0.0f;
        if (!ok && tid == 0 && !s_bad) { report(st, 4 /* ALS_ENOTSPD */, v); s_bad = 1; }
        const RM ip = ok ? one / pv : one;
        if (tid < BB) {
          rowk[tid] = Dk[kk * BB + tid] * ip;
          colk[tid] = Dk[tid * BB + kk];
        }
        __syncthreads();
        if (tid < BB * BB) {
          const int m = tid / BB, l = tid % BB;
          RM val;
          if (m == kk && l == kk) val = ip;
          else if (m == kk) val = rowk[l];
          else if (l == kk) val = -(colk[m] * ip);
          else val = Ops::sub_prod(Dk[tid], colk[m], rowk[l]);
          Dk[tid] = val;
        }
        __syncthreads();
      }
      for (int e = tid; e < BB * NS; e += nt) {
        const int m = e / NS, x = e % NS;
        RM acc = zero;
        if (m < b)
          for (int l = 0; l < b; ++l) acc = Ops::add_prod(acc, Dk[m * BB + l], C[x * BB + l]);
        Yp[e] = acc;
      }
      __syncthreads();
      // EPT entries per thread at a time, EPT independent chains: the chain of one entry
      // is a sequence of dependent operations (16 double-float updates of ~15 FP32
      // instructions each), so the entries of a thread interleave to hide its latency
      constexpr int EPT = 4;
      constexpr int NT = NS * (NS + 1) / 2;
      for (int e0 = tid; e0 < NT; e0 += EPT * nt) {
        RM acc[EPT];
        const RM* xi[EPT];
        int jj[EPT];
        bool neg[EPT];
#pragma unroll
        for (int q = 0; q < EPT; ++q) {
          const int e = e0 + q * nt;
          int i, j;
          tri_entry<NS>(e < NT ? e : 0, i, j);
          xi[q] = C + i * BB;
          jj[q] = j;
          neg[q] = j < k0;   // sigma_j = -1: the chain runs on -M_ij and is negated back
          const RM m = Mr[(long long)i * LDM + j];
          acc[q] = neg[q] ? -m : m;
        }
#pragma unroll
        for (int l = 0; l < BB; ++l)
#pragma unroll
          for (int q = 0; q < EPT; ++q) acc[q] = Ops::sub_prod(acc[q], xi[q][l], Yp[l * NS + jj[q]]);
#pragma unroll
        for (int q = 0; q < EPT; ++q) {
          const int e = e0 + q * nt;
          if (e >= NT) continue;
          int i, j;
          tri_entry<NS>(e, i, j);
          const int mi = i - k0, mj = j - k0;
          const bool ik = mi >= 0 && mi < b, jk = mj >= 0 && mj < b;
          RM val = neg[q] ? -acc[q] : acc[q];
          if (ik && jk) val = Dk[mi * BB + mj];
          else if (jk) val = -Yp[mj * NS + i];
          else if (ik) val = Yp[mi * NS + j];
          Mr[(long long)i * LDM + j] = val;
        }
      }
      __syncthreads();
    }
    // upper triangle by diagonals (entry (i, i + t))
    for (int t = 0; t < NS; ++t) {
      const long long base = v * pstride + diag_start(NS, t);
      for (int i = tid; i + t < NS; i += nt) inv64[base + i] = Ops::to_double(Mr[(long long)i * LDM + i + t]);
    }
    __syncthreads();
  }
}


// y_v = A_v^-1 r|_v: one CTA of STAR_THREADS per star (vertex), rows by threads, over the
// wrapped diagonals (row i takes entry (i, (i + t) mod NS) at step t: entry i of diagonal t
// while i + t < NS, else entry i + t - NS of diagonal NS - t, its symmetric partner), so
// every thread multiplies at every step and each diagonal is read by consecutive threads.
// interior: the stars of the fine vertices 2c + 1 at the coarse-cell centres, written
// (mode 1) or subtracted (mode 2) straight into the nodes; else into the rows [vertex][375].
constexpr int STAR_THREADS = 128;
constexpr int STAR_ROWS = (NS + STAR_THREADS - 1) / STAR_THREADS;

template <typename T>
__global__ void __launch_bounds__(STAR_THREADS) k_qk3_star_apply(Geom g, const T* __restrict__ inv, int pstride,
                                                                 int interior, int mode, const T* __restrict__ r,
                                                                 T* __restrict__ out) {
  __shared__ T rs[NS];
  const int tid = threadIdx.x;
  const int ic[3] = {g.n[0] / 2, g.n[1] / 2, g.n[2] / 2};
  const long long count = interior ? (long long)ic[0] * ic[1] * ic[2] : g.nverts;
  const long long item = blockIdx.x;
  if (item >= count) return;   // uniform over the block
  int vx, vy, vz;
  if (interior) {
    vx = 2 * (int)(item % ic[0]) + 1;
    vy = 2 * (int)((item / ic[0]) % ic[1]) + 1;
    vz = 2 * (int)(item / ((long long)ic[0] * ic[1])) + 1;
  } else {
    vx = (int)(item % g.nv[0]);
    vy = (int)((item / g.nv[0]) % g.nv[1]);
    vz = (int)(item / ((long long)g.nv[0] * g.nv[1]));
  }
  const long long v = (long long)vx + (long long)g.nv[0] * ((long long)vy + (long long)g.nv[1] * vz);
  for (int e = tid; e < NS; e += STAR_THREADS) {
    long long nd;
    rs[e] = star_node(g, vx, vy, vz, e, nd) ? r[(e / SN) * g.N + nd] : T(0);
  }
  __syncthreads();
  const T* S = inv + v * pstride;
  T acc[STAR_ROWS];
#pragma unroll
  for (int k = 0; k < STAR_ROWS; ++k) acc[k] = T(0);
  // steps t and NS - t in the same iteration (NS is odd): both read the same two diagonals
  // (t and NS - t), each entry once for its row and once for its symmetric partner's, so
  // the second read of an entry follows the first within the iteration and hits in L1
  // instead of coming back from HBM
#pragma unroll
  for (int k = 0; k < STAR_ROWS; ++k) {
    const int i = tid + STAR_THREADS * k;
    if (i < NS) acc[k] += __ldg(S + i) * rs[i];   // t = 0: the main diagonal
  }
#pragma unroll 2
  for (int t = 1; t <= NS / 2; ++t) {
    const int u = NS - t;
    const T* dt = S + diag_start(NS, t);   // diagonal t (NS - t entries)
    const T* du = S + diag_start(NS, u);   // diagonal NS - t (t entries)
#pragma unroll
    for (int k = 0; k < STAR_ROWS; ++k) {
      const int i = tid + STAR_THREADS * k;
      if (i < NS) {
        // step t: entry (i, i + t) on diagonal t, else (i + t - NS, i) on diagonal NS - t;
        // step NS - t: entry (i, i + NS - t) on diagonal NS - t, else (i - t, i) on diagonal t
        const bool a = i < u, b = i < t;
        const T* p1 = a ? dt + i : du + (i - u);   // one load each, from the selected diagonal
        const T* p2 = b ? du + i : dt + (i - t);
        acc[k] += __ldg(p1) * rs[a ? i + t : i - u];
        acc[k] += __ldg(p2) * rs[b ? i + u : i - t];
      }
    }
  }
#pragma unroll
  for (int k = 0; k < STAR_ROWS; ++k) {
    const int i = tid + STAR_THREADS * k;
    if (i >= NS) continue;
    if (!interior) {
      out[v * NS + i] = acc[k];
    } else {
      long long nd;
      if (star_node(g, vx, vy, vz, i, nd)) {
        T* o = out + (i / SN) * g.N + nd;
        *o = mode == 2 ? *o - acc[k] : acc[k];
      }
    }
  }
}

// y_v = A_v^-1 r|_v in FP32 from the blocked storage; every entry of a block is used for both
// y_I += S r_J and y_J += S^T r_I from registers, the partial sums of a row (one per block
// column) meet in shared memory and are added in a fixed order.  TS: float, or bfloat16
// (ALS_STORE_BF16), widened on load; products and sums in FP32.
//
// Interior stars (285 KB each in FP32) are bound by their stream from memory: one persistent CTA
// an SM, whose producer warp keeps a ring of bulk copies (three quads of every block a stage in
// FP32) ahead of eleven consumer warps, one block a thread, across the stars' boundaries.
// The launch takes 70 us on 12^3 cells (381 MB, 5.4 TB/s) and 18 on 6^3 (one star an SM); with
// the same blocks loaded straight into registers, a CTA per star, it took 97 and 19, and before
// that, with every star padded to 375 dofs and wrapped rows staged two at a time (four shared
// loads for two FMAs), 140 and 60; six ring stages instead of nine give 74.
// Boundary stars, at most 55 blocks: 64 threads each, in a launch of their own beside it.
//
// Waits on the ring are bounded (wait_polls); on expiry the kernel records ALS_ETIMEOUT, stops
// storing, waits (at the default limit) for the copies in flight and returns.
constexpr int STARS_WARPS = 11, STARS_THREADS = 32 * (STARS_WARPS + 1);

// named barrier 1 of the consumer warps, and whether any of their threads brought a flag
__device__ __forceinline__ bool consumers_vote(int flag) {
  int any;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.s32 p, %1, 0;\n bar.red.or.pred q, 1, %2, p;\n selp.s32 %0, 1, 0, q;\n}\n"
      : "=r"(any)
      : "r"(flag), "n"(32 * STARS_WARPS)
      : "memory");
  return any != 0;
}

__device__ __forceinline__ float4 star_quad(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 star_quad(const __nv_bfloat16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
  const float2 c = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
  return make_float4(a.x, a.y, c.x, c.y);
}

// the products of quad q (compile-time after unrolling) of an off-diagonal block
__device__ __forceinline__ void quad_off(int q, float4 v4, const float (&rI)[SB], const float (&rJ)[SB],
                                         float (&yI)[SB], float (&yJ)[SB]) {
  const float v[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int e = 4 * q + k, rr = e / SB, cc = e % SB;
    if (e < SB * SB) {
      yI[rr] += v[k] * rJ[cc];
      yJ[cc] += v[k] * rI[rr];
    }
  }
}
// of a diagonal block: entries of the upper triangle
__device__ __forceinline__ void quad_diag(int q, float4 v4, const float (&rI)[SB], float (&yI)[SB]) {
  const float v[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int e = 4 * q + k;
    int rr = 0, at = 0;
#pragma unroll
    for (int x = 0; x < SB; ++x)
      if (e >= x * SB - x * (x - 1) / 2) { rr = x; at = x * SB - x * (x - 1) / 2; }
    const int cc = rr + e - at;
    yI[rr] += v[k] * rI[cc];
    if (cc != rr) yI[cc] += v[k] * rI[rr];
  }
}

template <typename TS>
struct StarRing {
  static constexpr int CQ = sizeof(TS) == 4 ? 3 : 6;              // quads per stage
  static constexpr int NA = SQ1 / CQ, NBS = (SQ2 + CQ - 1) / CQ;  // stages of the two parts of a star
  static constexpr int STAGES = 9;
  static constexpr int STAGE_ENTRIES = 4 * CQ * kFullBlocks;
  static constexpr size_t STAGE_BYTES = (size_t)STAGE_ENTRIES * sizeof(TS);
  static constexpr size_t BAR_BYTES = 256;
  static constexpr size_t SMEM = BAR_BYTES + STAGES * STAGE_BYTES + (NS + 1 + NS * kFullRows) * sizeof(float);
  static_assert(NA + NBS > STAGES && SQ1 % CQ == 0 && 2 * STAGES * 8 <= (int)BAR_BYTES, "ring layout");
  static_assert(STAGE_BYTES % 16 == 0 && (4 * 3 * kFullOff * sizeof(TS)) % 16 == 0 &&
                    (kFullEntries * sizeof(TS)) % 16 == 0 && (4 * SQ1 * kFullBlocks * sizeof(TS)) % 16 == 0,
                "bulk copies need 16-byte alignment");
};

// vertex of interior item `item` (interior: the fine vertex at a coarse cell's centre) and its
// index among the interior vertices
__device__ __forceinline__ long long star_item(const Geom& g, int interior, int item, int& vx, int& vy, int& vz) {
  const int nix = g.nv[0] - 2, niy = g.nv[1] - 2;
  if (interior) {
    const int cx = g.n[0] / 2, cy = g.n[1] / 2, q = item / cx;
    vx = 2 * (item - q * cx) + 1;
    vz = q / cy;
    vy = 2 * (q - vz * cy) + 1;
    vz = 2 * vz + 1;
  } else {
    const int q = item / nix;
    vx = item - q * nix + 1;
    vz = q / niy;
    vy = q - vz * niy + 1;
    vz += 1;
  }
  return (vx - 1) + nix * ((vy - 1) + (long long)niy * (vz - 1));
}

template <typename TS>
__global__ void __launch_bounds__(STARS_THREADS, 1) k_qk3_stars(Geom g, const TS* __restrict__ inv, int interior,
                                                                int mode, int count, const float* __restrict__ r,
                                                                float* __restrict__ out, DevStatus* st,
                                                                int wait_polls, int early_trigger) {
  using C = StarRing<TS>;
  extern __shared__ __align__(128) unsigned char smraw[];
  uint64_t* full = reinterpret_cast<uint64_t*>(smraw);
  uint64_t* empty = full + C::STAGES;
  TS* ring = reinterpret_cast<TS*>(smraw + C::BAR_BYTES);
  float* rs = reinterpret_cast<float*>(smraw + C::BAR_BYTES + C::STAGES * C::STAGE_BYTES);
  float* part = rs + NS + 1;
  __shared__ int s_fail;
  const int tid = threadIdx.x, warp = tid >> 5;
  if (tid == 0) {
    s_fail = 0;
    for (int i = 0; i < C::STAGES; ++i) {
      tma::mbar_init(&full[i], 1);
      tma::mbar_init(&empty[i], STARS_WARPS);
    }
    tma::fence_init();
  }
  __syncthreads();
  if (warp == STARS_WARPS) {
    // producer: the inverses are written by the setup only, so it fills the ring before the
    // dependency wait (a star has more stages than the ring); a stage is refilled once all consumer warps have released it
    if ((tid & 31) == 0) {
      int k = 0;   // stages issued
      for (int item = blockIdx.x; item < count; item += gridDim.x) {
        int vx, vy, vz;
        const TS* S = inv + star_item(g, interior, item, vx, vy, vz) * kFullEntries;
        for (int c = 0; c < C::NA + C::NBS; ++c, ++k) {
          const int s = k % C::STAGES;
          if (k == C::STAGES) {   // the ring is full of copies on their way
            pdl_wait();
            if (early_trigger) pdl_trigger();
          }
          if (k >= C::STAGES && !tma::mbar_wait(&empty[s], (uint32_t)((k / C::STAGES - 1) & 1))) {
            report(st, 7 /* ALS_ETIMEOUT */, item);
            *(volatile int*)&s_fail = 1;
          }
          if (*(volatile int*)&s_fail) break;
          const bool a = c < C::NA;
          const int q = a ? c * C::CQ : (c - C::NA) * C::CQ;
          const int nq = a ? C::CQ : (SQ2 - q < C::CQ ? SQ2 - q : C::CQ);
          const uint32_t bytes = (uint32_t)(4 * nq * (a ? kFullBlocks : kFullOff) * sizeof(TS));
          const TS* src = S + (a ? 4 * q * kFullBlocks : 4 * SQ1 * kFullBlocks + 4 * q * kFullOff);
          tma::mbar_expect_tx(&full[s], bytes);
          tma::bulk_load(ring + s * C::STAGE_ENTRIES, src, bytes, &full[s]);
        }
        if (*(volatile int*)&s_fail) break;
      }
      // after a failure: no copy may be in flight when the CTA exits
      for (int m = k > C::STAGES ? k - C::STAGES : 0; m < k; ++m)
        tma::mbar_wait(&full[m % C::STAGES], (uint32_t)((m / C::STAGES) & 1));
    }
  } else {
    int I = 0, J = 0;
    const int b = tid;
    const bool mine = b < kFullBlocks, off = b < kFullOff;
    if (mine) StarBlocks(NS).block_of(b, I, J);
    const int nn01 = g.nn[0] * g.nn[1];
    int eo[2];   // offsets of star entries tid and tid + 352 from node 3v - 2
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int e = tid + 32 * STARS_WARPS * k, c = e / SN, o = e - c * SN, oz = o / (S1 * S1), oxy = o - oz * (S1 * S1);
      eo[k] = c * (int)g.N + oxy % S1 + (oxy / S1) * g.nn[0] + oz * nn01;
    }
    const auto base_of = [&](int item, int& vx, int& vy, int& vz) {
      star_item(g, interior, item, vx, vy, vz);
      return (3 * vx - 2) + (3 * vy - 2) * g.nn[0] + (3 * vz - 2) * nn01;
    };
    pdl_wait();
    // early_trigger: the boundary-star kernel, which needs nothing this one writes, may start
    if (early_trigger) pdl_trigger();
    int vx, vy, vz, base = 0;
    float rn[2] = {0.f, 0.f};
    if ((int)blockIdx.x < count) {
      base = base_of(blockIdx.x, vx, vy, vz);
#pragma unroll
      for (int k = 0; k < 2; ++k)
        if (tid + 32 * STARS_WARPS * k < NS) rn[k] = r[base + eo[k]];
    }
    int k = 0;   // stages consumed
    for (int item = blockIdx.x; item < count; item += gridDim.x) {
#pragma unroll
      for (int q = 0; q < 2; ++q)
        if (tid + 32 * STARS_WARPS * q < NS) rs[tid + 32 * STARS_WARPS * q] = rn[q];
      asm volatile("bar.sync 1, %0;" ::"n"(32 * STARS_WARPS) : "memory");
      const long long v = (long long)vx + (long long)g.nv[0] * ((long long)vy + (long long)g.nv[1] * vz);
      const int here = base;
      if (item + (int)gridDim.x < count) {   // the next star's r, in flight over this one
        base = base_of(item + gridDim.x, vx, vy, vz);
#pragma unroll
        for (int q = 0; q < 2; ++q)
          if (tid + 32 * STARS_WARPS * q < NS) rn[q] = r[base + eo[q]];
      }
      float rI[SB], rJ[SB], yI[SB], yJ[SB];
#pragma unroll
      for (int q = 0; q < SB; ++q) {
        rI[q] = mine ? rs[SB * I + q] : 0.f;
        rJ[q] = mine ? rs[SB * J + q] : 0.f;
        yI[q] = yJ[q] = 0.f;
      }
#pragma unroll
      for (int c = 0; c < C::NA + C::NBS; ++c, ++k) {
        const int s = k % C::STAGES;
        if (!*(volatile int*)&s_fail && !tma::mbar_wait(&full[s], (uint32_t)((k / C::STAGES) & 1), wait_polls)) {
          report(st, 7 /* ALS_ETIMEOUT */, item);
          *(volatile int*)&s_fail = 1;
        }
        const TS* W = ring + s * C::STAGE_ENTRIES;
#pragma unroll
        for (int q = 0; q < C::CQ; ++q) {
          if (c < C::NA) {
            const int qq = c * C::CQ + q;
            if (off) quad_off(qq, star_quad(W + 4 * (q * kFullBlocks + b)), rI, rJ, yI, yJ);
            else if (mine) quad_diag(qq, star_quad(W + 4 * (q * kFullBlocks + b)), rI, yI);
          } else if (SQ1 + (c - C::NA) * C::CQ + q < SQ1 + SQ2) {
            if (off) quad_off(SQ1 + (c - C::NA) * C::CQ + q, star_quad(W + 4 * (q * kFullOff + b)), rI, rJ, yI, yJ);
          }
        }
        __syncwarp();
        if ((tid & 31) == 0) tma::mbar_arrive(&empty[s]);
      }
      if (mine) {
#pragma unroll
        for (int q = 0; q < SB; ++q) part[(SB * I + q) * kFullRows + J] = yI[q];
        if (off) {
#pragma unroll
          for (int q = 0; q < SB; ++q) part[(SB * J + q) * kFullRows + I] = yJ[q];
        }
      }
      // The producer may set s_fail at any time: the consumers vote, so that all of them leave or none (one that left
      // alone would be missing at the others' next barrier).
      if (consumers_vote(*(volatile int*)&s_fail)) break;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int i = tid + 32 * STARS_WARPS * q;
        if (i >= NS) continue;
        float acc = 0.f;
#pragma unroll
        for (int jb = 0; jb < kFullRows; ++jb) acc += part[i * kFullRows + jb];
        if (!interior) {
          out[v * NS + i] = acc;
        } else {
          float* o = out + here + eo[q];
          *o = mode == 2 ? *o - acc : acc;
        }
      }
    }
    if (!early_trigger) pdl_trigger();
  }
}

// the boundary stars: one star per 64-thread CTA; runs beside the interior-star kernel, which
// lets it start once its own dependency wait has returned, and waits for it only at its end
template <typename TS>
__global__ void __launch_bounds__(64) k_qk3_stars_bnd(Geom g, const TS* __restrict__ inv, const int* __restrict__ bvid,
                                                      const long long* __restrict__ boff,
                                                      const float* __restrict__ r, float* __restrict__ out) {
  constexpr int MMAX = 150, RMAX = MMAX / SB;
  __shared__ float rs[MMAX];
  __shared__ float part[MMAX * RMAX];
  const int t = threadIdx.x, v = __ldg(bvid + blockIdx.x);
  const TS* S = inv + __ldg(boff + blockIdx.x);
  const int vx = v % g.nv[0], q0 = v / g.nv[0], vy = q0 % g.nv[1], vz = q0 / g.nv[1];
  const StarBox box(g, vx, vy, vz);
  const StarBlocks sb(box.m);
  for (int a = t; a < sb.nbr * SB; a += 64) {
    float val = 0.f;
    if (a < box.m) {
      const int e = box.entry(a), c = e / SN, o = e - c * SN;
      val = __ldcg(r + (c * (int)g.N + (3 * vx - 2 + o % S1) +
                        g.nn[0] * ((3 * vy - 2 + (o / S1) % S1) + g.nn[1] * (3 * vz - 2 + o / (S1 * S1)))));
    }
    rs[a] = val;
  }
  __syncthreads();
  if (t < sb.nblk) {
    int I, J;
    sb.block_of(t, I, J);
    float rI[SB], yI[SB];
#pragma unroll
    for (int k = 0; k < SB; ++k) {
      rI[k] = rs[SB * I + k];
      yI[k] = 0.f;
    }
    if (I != J) {
      float rJ[SB], yJ[SB];
#pragma unroll
      for (int k = 0; k < SB; ++k) {
        rJ[k] = rs[SB * J + k];
        yJ[k] = 0.f;
      }
#pragma unroll
      for (int q = 0; q < SQ1; ++q) quad_off(q, star_quad(S + 4 * (q * sb.nblk + t)), rI, rJ, yI, yJ);
#pragma unroll
      for (int q = 0; q < SQ2; ++q) quad_off(SQ1 + q, star_quad(S + sb.q2() + 4 * (q * sb.noff + t)), rI, rJ, yI, yJ);
#pragma unroll
      for (int k = 0; k < SB; ++k) part[(SB * J + k) * sb.nbr + I] = yJ[k];
    } else {
#pragma unroll
      for (int q = 0; q < SQ1; ++q) quad_diag(q, star_quad(S + 4 * (q * sb.nblk + t)), rI, yI);
    }
#pragma unroll
    for (int k = 0; k < SB; ++k) part[(SB * I + k) * sb.nbr + J] = yI[k];
  }
  __syncthreads();
  for (int a = t; a < box.m; a += 64) {
    float acc = 0.f;
    for (int jb = 0; jb < sb.nbr; ++jb) acc += part[a * sb.nbr + jb];
    out[(long long)v * NS + box.entry(a)] = acc;   // absent and Dirichlet entries are never read
  }
  pdl_wait();
  pdl_trigger();
}

// the blocked storage from the FP64 packed diagonals, rounded to nearest: one CTA per star,
// interior vertices first
__device__ __forceinline__ void store_star(float* p, double v) { *p = (float)v; }
__device__ __forceinline__ void store_star(__nv_bfloat16* p, double v) { *p = __double2bfloat16(v); }
template <typename TS>
__global__ void __launch_bounds__(256) k_qk3_pack(Geom g, int pstride, int nint, const int* __restrict__ bvid,
                                                  const long long* __restrict__ boff,
                                                  const double* __restrict__ inv64, TS* __restrict__ dst0) {
  const int item = blockIdx.x, nix = g.nv[0] - 2, niy = g.nv[1] - 2;
  int vx, vy, vz;
  if (item < nint) {
    vx = item % nix + 1;
    vy = (item / nix) % niy + 1;
    vz = item / (nix * niy) + 1;
  } else {
    const int v = bvid[item - nint];
    vx = v % g.nv[0];
    vy = (v / g.nv[0]) % g.nv[1];
    vz = v / (g.nv[0] * g.nv[1]);
  }
  const StarBox box(g, vx, vy, vz);
  const StarBlocks sb(box.m);
  const double* src = inv64 + ((long long)vx + (long long)g.nv[0] * ((long long)vy + (long long)g.nv[1] * vz)) * pstride;
  TS* dst = dst0 + (item < nint ? (long long)item * kFullEntries : boff[item - nint]);
  for (int p = threadIdx.x; p < sb.entries(); p += blockDim.x) {
    const bool second = p >= sb.q2();
    const int w = (second ? p - sb.q2() : p) >> 2, n = second ? sb.noff : sb.nblk, q = w / n, b = w - q * n;
    const int e = 4 * (second ? q + SQ1 : q) + (p & 3);
    int I, J, rr, cc;
    sb.block_of(b, I, J);
    if (I != J) {
      rr = e / SB;
      cc = e % SB;
    } else {
      rr = 0;
      while (rr + 1 < SB && e >= (rr + 1) * SB - (rr + 1) * rr / 2) ++rr;
      cc = rr + e - (rr * SB - rr * (rr - 1) / 2);
    }
    const int i = SB * I + rr, j = SB * J + cc;
    double val = 0.0;
    if (rr < SB && i < box.m && j < box.m) {
      const int ei = box.entry(i), ej = box.entry(j);
      val = src[diag_start(NS, ej - ei) + ei];
    }
    store_star(dst + p, val);
  }
}

// z(node) = sum over the (up to 8) stars containing the node, fixed order; 0 at Dirichlet nodes
template <typename T>
__global__ void k_qk3_star_gather(Geom g, const T* __restrict__ sc, T* __restrict__ z) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  pdl_wait();
  if (t < 3u * (unsigned)g.N) {
    int comp, i, j, k;
    entry_coords(g, t, comp, i, j, k);
    T acc = T(0);
    if (!bnd_node(g, i, j, k)) acc = star_sum<T>(g, sc, comp, i, j, k);
    z[t] = acc;
  }
  pdl_trigger();
}

// ---------------------------------------------------------------------------
// transfers: P_H (the coarse Q3 basis at the fine nodes, tensor product of 1D weights;
// each fine node belongs to the coarse cell min(f div 6, nc - 1) per axis) and its
// transpose, by per-coarse-cell contractions; fine Dirichlet rows and coarse Dirichlet
// columns are zero
// ---------------------------------------------------------------------------

// xf = P_H xc (and xadd += xf): per coarse cell (one CTA) its 64 coarse values (zero at
// Dirichlet coarse nodes) contracted with the 1D weights along x, y, z into the 7^3 fine
// values, each written by the cell that owns the fine node (the owner rule of the
// restriction below; Dirichlet fine nodes get zero)
template <typename T>
__global__ void __launch_bounds__(128) k_qk3_prolong_cells(Geom gc, Geom gf, const T* __restrict__ xc,
                                                           T* __restrict__ xf, T* __restrict__ xadd) {
  __shared__ T u[3][NB];
  __shared__ T t1[3][NF * N1 * N1];
  __shared__ T t2[3][NF * NF * N1];
  __shared__ T pw[NF][N1];
  const int tid = threadIdx.x, nt = blockDim.x;
  const long long cell = blockIdx.x;
  const int cx = (int)(cell % gc.n[0]), cy = (int)((cell / gc.n[0]) % gc.n[1]),
            cz = (int)(cell / ((long long)gc.n[0] * gc.n[1]));
  if (tid < NF * N1) pw[tid / N1][tid % N1] = Tab<T>::pw(tid / N1, tid % N1);
  pdl_wait();
  pdl_trigger();
  for (int e = tid; e < 3 * NB; e += nt) {
    const int c = e / NB, a = e % NB;
    const int I = K * cx + a % N1, J = K * cy + (a / N1) % N1, Kz = K * cz + a / (N1 * N1);
    u[c][a] = bnd_node(gc, I, J, Kz) ? T(0) : xc[c * gc.N + node_id(gc, I, J, Kz)];
  }
  __syncthreads();
  for (int e = tid; e < 3 * NF * N1 * N1; e += nt) {   // x: (ax, ay, az) -> (fx, ay, az)
    const int c = e / (NF * N1 * N1), r = e % (NF * N1 * N1), fx = r % NF, yz = r / NF;
    T acc = T(0);
#pragma unroll
    for (int ax = 0; ax < N1; ++ax) acc += pw[fx][ax] * u[c][ax + N1 * yz];
    t1[c][r] = acc;
  }
  __syncthreads();
  for (int e = tid; e < 3 * NF * NF * N1; e += nt) {   // y: (fx, ay, az) -> (fx, fy, az)
    const int c = e / (NF * NF * N1), r = e % (NF * NF * N1), fx = r % NF, fy = (r / NF) % NF, az = r / (NF * NF);
    T acc = T(0);
#pragma unroll
    for (int ay = 0; ay < N1; ++ay) acc += pw[fy][ay] * t1[c][fx + NF * (ay + N1 * az)];
    t2[c][r] = acc;
  }
  __syncthreads();
  for (int e = tid; e < 3 * NF * NF * NF; e += nt) {   // z: (fx, fy, az) -> (fx, fy, fz), owned nodes
    const int c = e / (NF * NF * NF), r = e % (NF * NF * NF), fxy = r % (NF * NF), fx = r % NF, fy = fxy / NF,
              fz = r / (NF * NF);
    if ((fx == NF - 1 && cx != gc.n[0] - 1) || (fy == NF - 1 && cy != gc.n[1] - 1) ||
        (fz == NF - 1 && cz != gc.n[2] - 1))
      continue;
    T acc = T(0);
#pragma unroll
    for (int az = 0; az < N1; ++az) acc += pw[fz][az] * t2[c][fxy + NF * NF * az];
    const int i = 2 * K * cx + fx, j = 2 * K * cy + fy, k = 2 * K * cz + fz;
    const T v = bnd_node(gf, i, j, k) ? T(0) : acc;
    const long long fn = c * gf.N + node_id(gf, i, j, k);
    xf[fn] = v;
    if (xadd) xadd[fn] += v;
  }
}

// rc = P_H^T (rf - sub) in two steps.  Per coarse cell (one CTA): the 7^3 fine values it
// owns (a fine node on the face shared with the next coarse cell belongs to that cell;
// Dirichlet fine nodes are zero) contracted with the 1D weights along x, y, z into the
// cell's 64 node values, staged per cell; then k_qk3_gather sums the staged values of the
// cells containing each coarse node (zero at Dirichlet nodes).  A fine node outside the
// cells of a coarse node lies where that node's basis function vanishes, so the owner
// rule gives exactly P_H^T.
constexpr int RS_THREADS = 128;
template <typename T>
__global__ void __launch_bounds__(RS_THREADS) k_qk3_restrict_cells(Geom gc, Geom gf, const T* __restrict__ rf,
                                                                   const T* __restrict__ sub, T* __restrict__ stage) {
  __shared__ T v[3][NF * NF * NF];
  __shared__ T t1[3][N1 * NF * NF];
  __shared__ T t2[3][N1 * N1 * NF];
  __shared__ T pw[NF][N1];
  const int tid = threadIdx.x;
  const long long cell = blockIdx.x;
  const int cx = (int)(cell % gc.n[0]), cy = (int)((cell / gc.n[0]) % gc.n[1]),
            cz = (int)(cell / ((long long)gc.n[0] * gc.n[1]));
  if (tid < NF * N1) pw[tid / N1][tid % N1] = Tab<T>::pw(tid / N1, tid % N1);
  pdl_wait();
  pdl_trigger();
  for (int e = tid; e < NF * NF * NF; e += RS_THREADS) {
    const int fx = e % NF, fy = (e / NF) % NF, fz = e / (NF * NF);
    const bool own = (fx < NF - 1 || cx == gc.n[0] - 1) && (fy < NF - 1 || cy == gc.n[1] - 1) &&
                     (fz < NF - 1 || cz == gc.n[2] - 1);
    const int i = 2 * K * cx + fx, j = 2 * K * cy + fy, k = 2 * K * cz + fz;
    const bool use = own && !bnd_node(gf, i, j, k);
    const long long nd = node_id(gf, i, j, k);
    for (int c = 0; c < 3; ++c) {
      const long long fn = c * gf.N + nd;
      v[c][e] = use ? (sub ? rf[fn] - sub[fn] : rf[fn]) : T(0);
    }
  }
  __syncthreads();
  for (int e = tid; e < 3 * N1 * NF * NF; e += RS_THREADS) {   // x: (fx, fy, fz) -> (ax, fy, fz)
    const int c = e / (N1 * NF * NF), r = e % (N1 * NF * NF), ax = r % N1, yz = r / N1;
    T acc = T(0);
#pragma unroll
    for (int fx = 0; fx < NF; ++fx) acc += pw[fx][ax] * v[c][fx + NF * yz];
    t1[c][r] = acc;
  }
  __syncthreads();
  for (int e = tid; e < 3 * N1 * N1 * NF; e += RS_THREADS) {   // y: (ax, fy, fz) -> (ax, ay, fz)
    const int c = e / (N1 * N1 * NF), r = e % (N1 * N1 * NF), ax = r % N1, ay = (r / N1) % N1, fz = r / (N1 * N1);
    T acc = T(0);
#pragma unroll
    for (int fy = 0; fy < NF; ++fy) acc += pw[fy][ay] * t1[c][ax + N1 * (fy + NF * fz)];
    t2[c][r] = acc;
  }
  __syncthreads();
  for (int e = tid; e < 3 * NB; e += RS_THREADS) {              // z: (ax, ay, fz) -> (ax, ay, az)
    const int c = e / NB, a = e % NB, axy = a % (N1 * N1), az = a / (N1 * N1);
    T acc = T(0);
#pragma unroll
    for (int fz = 0; fz < NF; ++fz) acc += pw[fz][az] * t2[c][axy + N1 * N1 * fz];
    stage[(cell * 3 + c) * NB + a] = acc;
  }
}

}  // namespace qk3

// ---------------------------------------------------------------------------
// entry points, called by qk.cu's dispatchers for 3D levels
// ---------------------------------------------------------------------------
void qk3_tables() { qk3::ensure_tables(); }

void qk3_apply(const LevelDev& L, int prec, int mode, double gamma, const void* x, void* y, const void* p_in,
               void* p_out, cudaStream_t s) {
  if (prec == PREC_F64) qk3::apply_t<double>(L, mode, gamma, x, y, p_in, p_out, s);
  else qk3::apply_t<float>(L, mode, gamma, x, y, p_in, p_out, s);
}

void qk3_apply_epi(const LevelDev& L, int prec, double gamma, const void* x, void* y, const ApplyEpi& e,
                   cudaStream_t s, cudaEvent_t e0, cudaEvent_t e1) {
  if (prec == PREC_F64) qk3::apply_epi_t<double>(L, gamma, x, y, e, s, e0, e1);
  else qk3::apply_epi_t<float>(L, gamma, x, y, e, s, e0, e1);
}

void qk3_load_vector(const LevelDev& L, const double* f_qp, double* F, cudaStream_t s) {
  const long long tot = L.g.ncells * 3 * qk3::NB;
  qk3::k_qk3_load<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(L.g, f_qp, (double*)L.ebuf);
  qk3::k_qk3_gather<double><<<(unsigned)((3 * L.g.N + 255) / 256), 256, 0, s>>>(L.g, (const double*)L.ebuf, nullptr,
                                                                               F, 0, 1);
  count_launch(2);
}

void qk3_mass_setup(const LevelDev& L, double gamma, int w_mu, int variant, double* winv64, float* winv32, double* S,
                    DevStatus* st, cudaStream_t s) {
  qk3::k_qk3_mass<<<(unsigned)((L.g.ncells + 127) / 128), 128, 0, s>>>(L.g, gamma, L.mu64, w_mu, variant, winv64,
                                                                       winv32, S, st);
  count_launch(1);
}

// CTAs of the star setup (each holds one 375 x 376 FP64 star matrix in the workspace)
int qk3_setup_ctas(long long nverts) {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const long long want = 2LL * sms;
  return (int)(nverts < want ? nverts : want);
}
size_t qk3_setup_ws_doubles(int ctas) { return (size_t)ctas * qk3::NS * qk3::LDM; }
long long qk3_star_layout(const Geom& g, std::vector<int>& bvid, std::vector<long long>& boff) {
  const long long nint = (long long)(g.nv[0] - 2) * (g.nv[1] - 2) * (g.nv[2] - 2);
  long long at = nint * qk3::kFullEntries;
  for (int vz = 0; vz < g.nv[2]; ++vz)
    for (int vy = 0; vy < g.nv[1]; ++vy)
      for (int vx = 0; vx < g.nv[0]; ++vx) {
        const qk3::StarBox box(g, vx, vy, vz);
        if (box.m == qk3::NS) continue;
        bvid.push_back(vx + g.nv[0] * (vy + g.nv[1] * vz));
        boff.push_back(at);
        at += qk3::StarBlocks(box.m).entries();
      }
  return at;
}

void qk3_derive32(const LevelDev& L, cudaStream_t s) {
  const unsigned n = (unsigned)L.g.nverts;
  qk3::k_qk3_pack<float><<<n, 256, 0, s>>>(L.g, L.pstride, (int)L.nint, L.bvid, L.boff, L.inv64, L.inv32);
  count_launch(1);
  if (L.inv16) {   // ALS_STORE_BF16
    qk3::k_qk3_pack<__nv_bfloat16><<<n, 256, 0, s>>>(L.g, L.pstride, (int)L.nint, L.bvid, L.boff, L.inv64,
                                                     (__nv_bfloat16*)L.inv16);
    count_launch(1);
  }
}

template <typename TS>
static void launch_stars_t(const LevelDev& L, const TS* inv, int interior, int mode, const float* r, float* out,
                           cudaStream_t s) {
  const int count = interior ? (L.g.n[0] / 2) * (L.g.n[1] / 2) * (L.g.n[2] / 2) : (int)L.nint;
  const int bnd = interior ? 0 : (int)L.nbnd;
  launch_pdl(qk3::k_qk3_stars<TS>, (unsigned)(count < 152 ? count : 152), qk3::STARS_THREADS, qk3::StarRing<TS>::SMEM,
             s, L.g, inv, interior, mode, count, r, out, L.status, L.wait_polls, bnd > 0 ? 1 : 0);
  if (bnd > 0)
    launch_pdl(qk3::k_qk3_stars_bnd<TS>, (unsigned)bnd, 64, 0, s, L.g, inv, (const int*)L.bvid,
               (const long long*)L.boff, r, out);
  count_launch(bnd > 0 ? 2 : 1);
}
// the FP32 star products: every star into the scratch rows, or (interior) the local solves on
// the coarse-cell interiors
static void launch_stars32(const LevelDev& L, int interior, int mode, const float* r, float* out, cudaStream_t s) {
  if (L.inv16) launch_stars_t(L, (const __nv_bfloat16*)L.inv16, interior, mode, r, out, s);
  else launch_stars_t(L, (const float*)L.inv32, interior, mode, r, out, s);
}

void qk3_patch_setup(const LevelDev& L, double gamma, DevStatus* st, cudaStream_t s, int df64) {
  cudaFuncSetAttribute(qk3::k_qk3_stars<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)qk3::StarRing<float>::SMEM);
  cudaFuncSetAttribute(qk3::k_qk3_stars<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)qk3::StarRing<__nv_bfloat16>::SMEM);
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(qk3::k_qk3_star_setup<double>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)qk3::SETUP_SMEM);
    cudaFuncSetAttribute(qk3::k_qk3_star_setup<DF64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)qk3::SETUP_SMEM);
    attr = true;
  }
  const int ctas = L.qk_ws_ctas < L.g.nverts ? L.qk_ws_ctas : (int)L.g.nverts;
  if (df64)
    qk3::k_qk3_star_setup<DF64><<<(unsigned)ctas, qk3::SETUP_THREADS, qk3::SETUP_SMEM, s>>>(
        L.g, gamma, L.mu64, L.winv64, L.qk_ws, L.inv64, L.pstride, st);
  else
    qk3::k_qk3_star_setup<double><<<(unsigned)ctas, qk3::SETUP_THREADS, qk3::SETUP_SMEM, s>>>(
        L.g, gamma, L.mu64, L.winv64, L.qk_ws, L.inv64, L.pstride, st);
  count_launch(1);
  qk3_derive32(L, s);
}

void qk3_patch_products(const LevelDev& L, const void* r, void* scratch, cudaStream_t s) {
  launch_stars32(L, 0, 0, (const float*)r, (float*)scratch, s);
}

void qk3_patch_smooth(const LevelDev& L, int prec, const void* r, void* z, void* scratch, cudaStream_t s) {
  const unsigned b3 = (unsigned)((3 * L.g.N + 255) / 256);
  if (prec == PREC_F64) {
    qk3::k_qk3_star_apply<double><<<(unsigned)L.g.nverts, qk3::STAR_THREADS, 0, s>>>(
        L.g, L.inv64, L.pstride, 0, 0, (const double*)r, (double*)scratch);
    count_launch(1);
    launch_pdl(qk3::k_qk3_star_gather<double>, b3, 256, 0, s, L.g, (const double*)scratch, (double*)z);
  } else {
    launch_stars32(L, 0, 0, (const float*)r, (float*)scratch, s);
    launch_pdl(qk3::k_qk3_star_gather<float>, b3, 256, 0, s, L.g, (const float*)scratch, (float*)z);
  }
  count_launch(1);
}

void qk3_interior_solve(const LevelDev& fine, int prec, const void* in, void* out, int subtract, cudaStream_t s) {
  const long long nc = (long long)(fine.g.n[0] / 2) * (fine.g.n[1] / 2) * (fine.g.n[2] / 2);
  if (prec == PREC_F64) {
    qk3::k_qk3_star_apply<double><<<(unsigned)nc, qk3::STAR_THREADS, 0, s>>>(
        fine.g, fine.inv64, fine.pstride, 1, subtract ? 2 : 1, (const double*)in, (double*)out);
    count_launch(1);
  } else {
    launch_stars32(fine, 1, subtract ? 2 : 1, (const float*)in, (float*)out, s);
  }
}

void qk3_prolong(const LevelDev& coarse, const LevelDev& fine, int prec, const void* xc, void* xf, cudaStream_t s,
                 void* xadd) {
  const unsigned nc = (unsigned)coarse.g.ncells;
  if (prec == PREC_F64)
    launch_pdl(qk3::k_qk3_prolong_cells<double>, nc, 128, 0, s, coarse.g, fine.g, (const double*)xc, (double*)xf,
               (double*)xadd);
  else
    launch_pdl(qk3::k_qk3_prolong_cells<float>, nc, 128, 0, s, coarse.g, fine.g, (const float*)xc, (float*)xf,
               (float*)xadd);
  count_launch(1);
}

// the coarse level's per-cell output buffer stages the cell contributions (the coarse
// level's own applies, which use it too, come after the restriction on the stream)
void qk3_restrict(const LevelDev& coarse, const LevelDev& fine, int prec, const void* rf, void* rc, cudaStream_t s,
                  const void* sub) {
  const unsigned nc = (unsigned)coarse.g.ncells, b = (unsigned)((3 * coarse.g.N + 255) / 256);
  if (prec == PREC_F64) {
    launch_pdl(qk3::k_qk3_restrict_cells<double>, nc, qk3::RS_THREADS, 0, s, coarse.g, fine.g, (const double*)rf,
               (const double*)sub, (double*)coarse.ebuf);
    launch_pdl(qk3::k_qk3_gather<double>, b, 256, 0, s, coarse.g, (const double*)coarse.ebuf, (const double*)nullptr,
               (double*)rc, 0, 0);
  } else {
    launch_pdl(qk3::k_qk3_restrict_cells<float>, nc, qk3::RS_THREADS, 0, s, coarse.g, fine.g, (const float*)rf,
               (const float*)sub, (float*)coarse.ebuf);
    launch_pdl(qk3::k_qk3_gather<float>, b, 256, 0, s, coarse.g, (const float*)coarse.ebuf, (const float*)nullptr,
               (float*)rc, 0, 0);
  }
  count_launch(2);
}

}  // namespace als
