// K1: the cell apply with the 1D contractions in registers.
//
// Included by operator.cu and tiles2.cu inside namespace als, after apply_lines.cuh.  Same arguments
// and results as k_apply_lines up to the order of the sums.
//
// 3D, scalar viscosity, all cells into the staged rows: one thread per (cell, velocity
// component), 32 cells a block, a warp per component.  A thread holds its component's 27 nodal
// values and contracts them along x, y and z in registers; the nine gradient entries at the 27
// Gauss points then change hands once through shared memory ([entry][point][cell], a lane per
// cell: no bank conflicts), thread c forms the stresses of the nine points of layer c, and the
// fluxes go back the same way for the transposed contractions.  About 1700 instructions a
// thread, 160 warp instructions a cell; the line-per-lane form exchanges every contraction
// through shared memory and issues 843.  Both are bound by issue (FP32) or the FP64 pipe, so
// large levels take this one; on small levels, where one thread's chain is the time, the line
// form's shorter chain wins (cells_in_registers).
//
// 2D, scalar or tensor viscosity: two lanes per cell, one component each, 16 cells a warp; the
// lanes exchange the diagonal gradient entries and the shear by shuffles.
#pragma once

// 1D tables applied to a line of three values by even and odd parts (s = u0 + u2, d = u2 - u0,
// e = s - 2 u1):  values B u = (t - h d, u1, t + h d), t = 0.3 s + 0.4 u1, h = g / 2;
// derivatives f D u = (f/2 d - f g e, f/2 d, f/2 d + f g e), the factor f = 2 / h_axis in the table.
template <typename T>
struct DerivTab {
  T half, g;   // f / 2, f g
};
template <typename T>
__device__ __forceinline__ DerivTab<T> deriv_tab(T f) { return DerivTab<T>{T(0.5) * f, Ref<T>::g * f}; }
template <typename T>
__device__ __forceinline__ void line_values(T u0, T u1, T u2, T (&o)[3]) {
  const T s = u0 + u2, d = u2 - u0, t = T(0.3) * s + T(0.4) * u1;
  o[0] = t - T(0.5) * Ref<T>::g * d;
  o[1] = u1;
  o[2] = t + T(0.5) * Ref<T>::g * d;
}
template <typename T>
__device__ __forceinline__ void line_derivs(const DerivTab<T>& D, T u0, T u1, T u2, T (&o)[3]) {
  const T s = u0 + u2, d = u2 - u0, e = s - T(2) * u1, h = D.half * d;
  o[0] = h - D.g * e;
  o[1] = h;
  o[2] = h + D.g * e;
}
// the transposes, added into o (ADD) or stored
template <typename T, bool ADD>
__device__ __forceinline__ void line_values_t(T f0, T f1, T f2, T (&o)[3]) {
  const T s = f0 + f2, d = f2 - f0, t = T(0.3) * s, h = T(0.5) * Ref<T>::g * d;
  const T a = t - h, c = t + h, b = T(0.4) * s + f1;
  if (ADD) { o[0] += a; o[1] += b; o[2] += c; }
  else { o[0] = a; o[1] = b; o[2] = c; }
}
template <typename T, bool ADD>
__device__ __forceinline__ void line_derivs_t(const DerivTab<T>& D, T f0, T f1, T f2, T (&o)[3]) {
  const T e = D.g * (f2 - f0), h = D.half * ((f0 + f2) + f1);
  const T a = e - h, c = e + h;
  if (ADD) { o[0] += a; o[1] -= T(2) * e; o[2] += c; }
  else { o[0] = a; o[1] = -T(2) * e; o[2] = c; }
}

// u at the nodes of a cell's line set from the star outputs: node sums in the fixed order of the
// patch gather (z tap, y tap, then the x pair), 0 at Dirichlet nodes; z is stored by the cell
// that owns the node.  c: component.
template <typename T>
__device__ __forceinline__ void cell_from_stars(const Geom& g, const PatchIn<T>& pin, int c, int cx, int cy, int cz,
                                                T (&u)[27]) {
#pragma unroll
  for (int az = 0; az < 3; ++az)
#pragma unroll
    for (int ay = 0; ay < 3; ++ay) {
      T l[3];
      const int nj = 2 * cy + ay, nk = 2 * cz + az;
      // taps per axis: middle node 2v+1 -> vertices v (offset 2), v+1 (offset 0); corner 2v -> v (offset 1)
      const bool off = nj == 0 || nj == g.nn[1] - 1 || nk == 0 || nk == g.nn[2] - 1;
      const int ncol = 3 * g.nv[0];
      T acc[3] = {T(0), T(0), T(0)};
#pragma unroll
      for (int tz = 0; tz < (az == 1 ? 2 : 1); ++tz)
#pragma unroll
        for (int ty = 0; ty < (ay == 1 ? 2 : 1); ++ty) {
          const int vy = ay == 1 ? cy + ty : cy + (ay >> 1), oy = ay == 1 ? 2 - 2 * ty : 1;
          const int vz = az == 1 ? cz + tz : cz + (az >> 1), oz = az == 1 ? 2 - 2 * tz : 1;
          const int row = ((c * 3 + oz) * 3 + oy) * (g.nv[1] * g.nv[2]) + vz * g.nv[1] + vy;
          const T* rp = pin.out + (long long)row * ncol + 3 * cx;
          const T v1 = off ? T(0) : rp[1], v2 = off ? T(0) : rp[2], v3 = off ? T(0) : rp[3], v4 = off ? T(0) : rp[4];
          acc[0] += v1;
          acc[1] += v2 + v3;
          acc[2] += v4;
        }
      l[0] = cx == 0 ? T(0) : acc[0];
      l[1] = acc[1];
      l[2] = cx == g.n[0] - 1 ? T(0) : acc[2];
      const long long at = (long long)c * g.N + (long long)(unsigned)(g.nn[0] * (nj + g.nn[1] * nk)) + 2 * cx;
      if ((ay < 2 || cy == g.n[1] - 1) && (az < 2 || cz == g.n[2] - 1)) {
        pin.z[at] = l[0];
        pin.z[at + 1] = l[1];
        if (cx == g.n[0] - 1) pin.z[at + 2] = l[2];
      }
#pragma unroll
      for (int ax = 0; ax < 3; ++ax) u[(az * 3 + ay) * 3 + ax] = l[ax];
    }
}

// d u / d x_AXIS at the 27 points (the other axes interpolated), for the divergence alone
template <typename T, int AXIS>
__device__ __forceinline__ void derivative_fwd(const DerivTab<T>& D, T (&u)[27]) {
#pragma unroll
  for (int axis = 0; axis < 3; ++axis) {
    const int st = axis == 0 ? 1 : (axis == 1 ? 3 : 9);
#pragma unroll
    for (int l = 0; l < 9; ++l) {
      const int b = axis == 0 ? 3 * l : (axis == 1 ? 9 * (l / 3) + l % 3 : l);
      T o[3];
      if (axis == AXIS) line_derivs<T>(D, u[b], u[b + st], u[b + 2 * st], o);
      else line_values<T>(u[b], u[b + st], u[b + 2 * st], o);
#pragma unroll
      for (int q = 0; q < 3; ++q) u[b + q * st] = o[q];
    }
  }
}
// its transpose
template <typename T, int AXIS>
__device__ __forceinline__ void derivative_bwd(const DerivTab<T>& D, T (&u)[27]) {
#pragma unroll
  for (int axis = 2; axis >= 0; --axis) {
    const int st = axis == 0 ? 1 : (axis == 1 ? 3 : 9);
#pragma unroll
    for (int l = 0; l < 9; ++l) {
      const int b = axis == 0 ? 3 * l : (axis == 1 ? 9 * (l / 3) + l % 3 : l);
      T o[3];
      if (axis == AXIS) line_derivs_t<T, false>(D, u[b], u[b + st], u[b + 2 * st], o);
      else line_values_t<T, false>(u[b], u[b + st], u[b + 2 * st], o);
#pragma unroll
      for (int q = 0; q < 3; ++q) u[b + q * st] = o[q];
    }
  }
}

// Cells of a block and how its threads are laid out.  FP32, and FP64 without the viscous term:
// 32 cells, a warp per component.  FP64 with it: one warp of 10 cells x 3 components a block; the
// FP64 pipe takes 16 cycles for a warp's instruction whatever the SM holds, so a level's warps
// are spread over the SMs one by one, and no block barrier holds them together.
template <typename T, int MODE>
struct Cells3 {
  static constexpr bool VISC = (MODE & OP_VISC) != 0;
  static constexpr bool WARP = sizeof(T) == 8 && VISC;
  static constexpr int CELLS = WARP ? 10 : 32;
  static constexpr int THREADS = WARP ? 32 : 96;
  static constexpr int NE = VISC ? 9 : 3;  // entries exchanged per point: the gradient, or d u_c / d x_c alone
  struct Smem {
    T ex[NE * 27][CELLS];
    T mom[3][3][CELLS];
  };
  // resident blocks an SM asked of the compiler: FP32, seven (96 registers, 32 KB each), so
  // that 32^3 cells are one wave
  static constexpr int BLOCKS = sizeof(T) == 4 ? 7 : (WARP ? 8 : 2);
  __device__ __forceinline__ static void sync() {
    if (WARP) __syncwarp(0x3fffffffu);
    else __syncthreads();
  }
};

template <typename T, int MODE, bool ZP>
__device__ __forceinline__ void apply_cells3_body(unsigned bx, const Geom& g, const CellConst<T>& cc,
                                                  const T* __restrict__ x, const T* __restrict__ coef,
                                                  const T* __restrict__ p_in, T* __restrict__ p_out,
                                                  T* __restrict__ ebuf, const T* __restrict__ winv,
                                                  const PatchIn<T>& pin,
                                                  typename Cells3<T, MODE>::Smem& sm) {
  constexpr bool RAW = (MODE & OP_RAW) != 0;
  constexpr bool VISC = (MODE & OP_VISC) != 0;
  constexpr bool NEED_U = (MODE & (OP_VISC | OP_AL | OP_B)) != 0;
  constexpr bool NEED_FLUX = (MODE & (OP_VISC | OP_AL | OP_BT)) != 0;
  using C = Cells3<T, MODE>;
  const int c = threadIdx.x / C::CELLS, lane = threadIdx.x - c * C::CELLS;   // component (and point layer), cell slot
  if (C::WARP && c == 3) return;                                             // the two spare lanes
  const int ncells = (int)g.ncells, cell0 = (int)bx * C::CELLS, cell = cell0 + lane;
  const bool act = cell < ncells;
  const int cz = cell / (g.n[0] * g.n[1]), cyx = cell - cz * (g.n[0] * g.n[1]);
  const int cy = cyx / g.n[0], cx = cyx - cy * g.n[0];
  const DerivTab<T> dx = deriv_tab<T>(cc.s[0]), dy = deriv_tab<T>(cc.s[1]), dz = deriv_tab<T>(cc.s[2]);
  pdl_wait();
  if constexpr (NEED_U) {
    T u[27];
    if constexpr (ZP) {
      if (act) cell_from_stars<T>(g, pin, c, cx, cy, cz, u);
    } else if (act) {
      const bool inner = RAW || (cx > 0 && cx < g.n[0] - 1 && cy > 0 && cy < g.n[1] - 1 && cz > 0 && cz < g.n[2] - 1);
#pragma unroll
      for (int az = 0; az < 3; ++az)
#pragma unroll
        for (int ay = 0; ay < 3; ++ay) {
          const int nj = 2 * cy + ay, nk = 2 * cz + az;
          const T* row = x + (long long)c * g.N + (long long)(unsigned)(g.nn[0] * (nj + g.nn[1] * nk)) + 2 * cx;
#pragma unroll
          for (int ax = 0; ax < 3; ++ax)
            u[(az * 3 + ay) * 3 + ax] = (inner || !on_boundary(g, 2 * cx + ax, nj, nk)) ? row[ax] : T(0);
        }
    }
    if (!act) {
#pragma unroll
      for (int a = 0; a < 27; ++a) u[a] = T(0);
    }
    if constexpr (VISC) {
      // x lines, then per qx: y lines, z lines and the gradient entries of component c
      T bu[27], du[27];   // [az][ay][qx]
#pragma unroll
      for (int l = 0; l < 9; ++l) {
        T o0[3], o1[3];
        line_values<T>(u[3 * l], u[3 * l + 1], u[3 * l + 2], o0);
        line_derivs<T>(dx, u[3 * l], u[3 * l + 1], u[3 * l + 2], o1);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          bu[3 * l + q] = o0[q];
          du[3 * l + q] = o1[q];
        }
      }
#pragma unroll
      for (int qx = 0; qx < 3; ++qx) {
        T bb[3][3], db[3][3], bd[3][3];   // [qy][az]
#pragma unroll
        for (int az = 0; az < 3; ++az) {
          const int b = 9 * az + qx;
          T o0[3], o1[3], o2[3];
          line_values<T>(bu[b], bu[b + 3], bu[b + 6], o0);
          line_derivs<T>(dy, bu[b], bu[b + 3], bu[b + 6], o1);
          line_values<T>(du[b], du[b + 3], du[b + 6], o2);
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            bb[q][az] = o0[q];
            db[q][az] = o1[q];
            bd[q][az] = o2[q];
          }
        }
#pragma unroll
        for (int qy = 0; qy < 3; ++qy) {
          T gx[3], gy[3], gz[3];
          line_values<T>(bd[qy][0], bd[qy][1], bd[qy][2], gx);
          line_values<T>(db[qy][0], db[qy][1], db[qy][2], gy);
          line_derivs<T>(dz, bb[qy][0], bb[qy][1], bb[qy][2], gz);
#pragma unroll
          for (int qz = 0; qz < 3; ++qz) {
            const int p = qx + 3 * qy + 9 * qz;
            sm.ex[(3 * c + 0) * 27 + p][lane] = gx[qz];
            sm.ex[(3 * c + 1) * 27 + p][lane] = gy[qz];
            sm.ex[(3 * c + 2) * 27 + p][lane] = gz[qz];
          }
        }
      }
    } else {
      if (c == 0) derivative_fwd<T, 0>(dx, u);
      else if (c == 1) derivative_fwd<T, 1>(dy, u);
      else derivative_fwd<T, 2>(dz, u);
#pragma unroll
      for (int p = 0; p < 27; ++p) sm.ex[c * 27 + p][lane] = u[p];
    }
  }
  C::sync();
  // points of layer c: divergence moments, then the fluxes, in two passes over the exchange
  // buffer (holding the 81 gradient entries would take the registers of two more blocks an SM);
  // the viscosities are on their way meanwhile
  constexpr int D0 = 0, D1 = VISC ? 4 * 27 : 27, D2 = VISC ? 8 * 27 : 54;   // diagonal entries
  const T wz = cc.wdet * (c == 1 ? Ref<T>::W(1) : Ref<T>::W(0));
  const T gz = c == 0 ? Ref<T>::G(0) : (c == 1 ? T(0) : Ref<T>::G(2));
  T mu[VISC ? 9 : 1];
  if constexpr (VISC) {
    const T* src = coef + (long long)(act ? cell : cell0) * 27 + 9 * c;
#pragma unroll
    for (int q = 0; q < 9; ++q) mu[q] = src[q];
  }
  T pi[4] = {T(0), T(0), T(0), T(0)};
  if constexpr ((MODE & (OP_AL | OP_B)) != 0) {
    T m[4] = {T(0), T(0), T(0), T(0)};
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      const int p = 9 * c + q;
      const T dv = (Ref<T>::W(q % 3) * Ref<T>::W(q / 3)) * (sm.ex[D0 + p][lane] + sm.ex[D1 + p][lane] + sm.ex[D2 + p][lane]);
      m[0] += dv;
      if (q % 3 == 0) m[1] -= dv; else if (q % 3 == 2) m[1] += dv;
      if (q / 3 == 0) m[2] -= dv; else if (q / 3 == 2) m[2] += dv;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) sm.mom[k][c][lane] = (k == 0 ? wz : wz * Ref<T>::g) * m[k];
    C::sync();
    m[3] = Ref<T>::g * (sm.mom[0][2][lane] - sm.mom[0][0][lane]);
#pragma unroll
    for (int k = 0; k < 3; ++k) m[k] = (sm.mom[k][0][lane] + sm.mom[k][1][lane]) + sm.mom[k][2][lane];
    if constexpr ((MODE & OP_B) != 0) {
      if (act && c == 0) {
#pragma unroll
        for (int k = 0; k < 4; ++k) p_out[(long long)cell * 4 + k] = -m[k];
      }
    }
    if constexpr ((MODE & OP_AL) != 0) {
      if (winv) {   // W = M_p(1/mu): per-cell (d+1)^2 block of W^-1
        if (act) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            T s = T(0);
#pragma unroll
            for (int k = 0; k < 4; ++k) s += winv[((long long)cell * 4 + q) * 4 + k] * m[k];
            pi[q] = cc.gamma * s;
          }
        }
      } else {      // W = M_p = |K| diag(1, 1/3, ..)
#pragma unroll
        for (int q = 0; q < 4; ++q) pi[q] = cc.gamma * m[q] * (q == 0 ? cc.inv_m0 : cc.inv_m1);
      }
    }
  }
  if constexpr (!NEED_FLUX) {
    pdl_trigger();
    return;
  }
  if constexpr ((MODE & OP_BT) != 0) {
    if (act) {
#pragma unroll
      for (int q = 0; q < 4; ++q) pi[q] -= p_in[(long long)cell * 4 + q];
    }
  }
  // isotropic part of the stress (gamma Pi div u - p) and fluxes |J| w_q sigma_ak (the factor
  // 2 / h_k is in the transposed derivative)
  const T iso0 = pi[0] + pi[3] * gz, iso1 = pi[1] * Ref<T>::g, iso2 = pi[2] * Ref<T>::g;
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    const int p = 9 * c + q;
    T iso = iso0;
    if (q % 3 == 0) iso -= iso1; else if (q % 3 == 2) iso += iso1;
    if (q / 3 == 0) iso -= iso2; else if (q / 3 == 2) iso += iso2;
    const T w = wz * (Ref<T>::W(q % 3) * Ref<T>::W(q / 3)), wi = w * iso;
    if constexpr (VISC) {
      const T wm = w * mu[q];
      T gr[9];
#pragma unroll
      for (int e = 0; e < 9; ++e) gr[e] = sm.ex[e * 27 + p][lane];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        sm.ex[4 * a * 27 + p][lane] = wm * (gr[4 * a] + gr[4 * a]) + wi;
#pragma unroll
        for (int k = a + 1; k < 3; ++k) {
          const T f = wm * (gr[3 * a + k] + gr[3 * k + a]);
          sm.ex[(3 * a + k) * 27 + p][lane] = f;
          sm.ex[(3 * k + a) * 27 + p][lane] = f;
        }
      }
    } else {
#pragma unroll
      for (int a = 0; a < 3; ++a) sm.ex[a * 27 + p][lane] = wi;
    }
  }
  C::sync();
  T out[27];
  if constexpr (VISC) {
    T rxs[27], rys[27];   // [az][ay][qx]: D_x and B_x still to come
#pragma unroll
    for (int qx = 0; qx < 3; ++qx) {
      T px[3][3], py[3][3], pz[3][3];   // [az][qy]
#pragma unroll
      for (int qy = 0; qy < 3; ++qy) {
        const T* f = &sm.ex[3 * c * 27 + qx + 3 * qy][lane];
        constexpr int S = 9 * C::CELLS, E = 27 * C::CELLS;   // next z point, next entry
        T o0[3], o1[3], o2[3];
        line_values_t<T, false>(f[0], f[S], f[2 * S], o0);
        line_values_t<T, false>(f[E], f[E + S], f[E + 2 * S], o1);
        line_derivs_t<T, false>(dz, f[2 * E], f[2 * E + S], f[2 * E + 2 * S], o2);
#pragma unroll
        for (int az = 0; az < 3; ++az) {
          px[az][qy] = o0[az];
          py[az][qy] = o1[az];
          pz[az][qy] = o2[az];
        }
      }
#pragma unroll
      for (int az = 0; az < 3; ++az) {
        T rx[3], ry[3];
        line_values_t<T, false>(px[az][0], px[az][1], px[az][2], rx);
        line_derivs_t<T, false>(dy, py[az][0], py[az][1], py[az][2], ry);
        line_values_t<T, true>(pz[az][0], pz[az][1], pz[az][2], ry);
#pragma unroll
        for (int ay = 0; ay < 3; ++ay) {
          rxs[(3 * az + ay) * 3 + qx] = rx[ay];
          rys[(3 * az + ay) * 3 + qx] = ry[ay];
        }
      }
    }
#pragma unroll
    for (int l = 0; l < 9; ++l) {
      T o[3];
      line_derivs_t<T, false>(dx, rxs[3 * l], rxs[3 * l + 1], rxs[3 * l + 2], o);
      line_values_t<T, true>(rys[3 * l], rys[3 * l + 1], rys[3 * l + 2], o);
#pragma unroll
      for (int q = 0; q < 3; ++q) out[3 * l + q] = o[q];
    }
  } else {
#pragma unroll
    for (int p = 0; p < 27; ++p) out[p] = sm.ex[c * 27 + p][lane];
    if (c == 0) derivative_bwd<T, 0>(dx, out);
    else if (c == 1) derivative_bwd<T, 1>(dy, out);
    else derivative_bwd<T, 2>(dz, out);
  }
  if (act) {
#pragma unroll
    for (int az = 0; az < 3; ++az)
#pragma unroll
      for (int ay = 0; ay < 3; ++ay) {
        // row layout (stage_row), summed per node by the gather
        T* e = ebuf + (long long)stage_row(g, c, ay, az, cy, cz) * (3 * g.n[0]) + 3 * cx;
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) e[ax] = out[(3 * az + ay) * 3 + ax];
      }
  }
  pdl_trigger();
}
template <typename T, int MODE, bool ZP>
__global__ void __launch_bounds__(Cells3<T, MODE>::THREADS, Cells3<T, MODE>::BLOCKS)
    k_apply_cells3(Geom g, CellConst<T> cc, const T* __restrict__ x, const T* __restrict__ coef,
                   const T* __restrict__ p_in, T* __restrict__ p_out, T* __restrict__ ebuf,
                   const T* __restrict__ winv, PatchIn<T> pin) {
  __shared__ typename Cells3<T, MODE>::Smem sm;
  apply_cells3_body<T, MODE, ZP>(blockIdx.x, g, cc, x, coef, p_in, p_out, ebuf, winv, pin, sm);
}

// ---------------------------------------------------------------------------
// 2D: two lanes per cell (lanes i and i + 16: the components of cell i of the warp)
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void cell2_from_stars(const Geom& g, const PatchIn<T>& pin, int c, int cx, int cy,
                                                 T (&u)[9]) {
#pragma unroll
  for (int ay = 0; ay < 3; ++ay) {
    const int nj = 2 * cy + ay, ncol = 3 * g.nv[0];
    const bool off = nj == 0 || nj == g.nn[1] - 1;
    T acc[3] = {T(0), T(0), T(0)};
#pragma unroll
    for (int ty = 0; ty < (ay == 1 ? 2 : 1); ++ty) {
      const int vy = ay == 1 ? cy + ty : cy + (ay >> 1), oy = ay == 1 ? 2 - 2 * ty : 1;
      const T* rp = pin.out + (long long)((c * 3 + oy) * g.nv[1] + vy) * ncol + 3 * cx;
      const T v1 = off ? T(0) : rp[1], v2 = off ? T(0) : rp[2], v3 = off ? T(0) : rp[3], v4 = off ? T(0) : rp[4];
      acc[0] += v1;
      acc[1] += v2 + v3;
      acc[2] += v4;
    }
    u[3 * ay] = cx == 0 ? T(0) : acc[0];
    u[3 * ay + 1] = acc[1];
    u[3 * ay + 2] = cx == g.n[0] - 1 ? T(0) : acc[2];
    const long long at = (long long)c * g.N + (long long)(unsigned)(g.nn[0] * nj) + 2 * cx;
    if (ay < 2 || cy == g.n[1] - 1) {
      pin.z[at] = u[3 * ay];
      pin.z[at + 1] = u[3 * ay + 1];
      if (cx == g.n[0] - 1) pin.z[at + 2] = u[3 * ay + 2];
    }
  }
}

// The cell's contribution from its nodal values un (component c; the other lane of the pair holds
// the other one); store(ay, o) takes the outputs at the nodes (0..2, ay).  Every lane of the warp calls.
template <typename T, bool TENSOR, int MODE, typename Store>
__device__ __forceinline__ void cell2_contribution(const CellConst<T>& cc, bool act, int c, int cell, const T (&un)[9],
                                                   const T* mu, const T* __restrict__ coef,
                                                   const T* __restrict__ p_in, T* __restrict__ p_out,
                                                   const T* __restrict__ winv, Store store) {
  constexpr bool VISC = (MODE & OP_VISC) != 0;
  constexpr bool NEED_U = (MODE & (OP_VISC | OP_AL | OP_B)) != 0;
  constexpr bool NEED_FLUX = (MODE & (OP_VISC | OP_AL | OP_BT)) != 0;
  const DerivTab<T> dx = deriv_tab<T>(cc.s[0]), dy = deriv_tab<T>(cc.s[1]);
  // Only differences of u count: in FP32 those to the cell's middle node are taken first, so that what
  // follows rounds relative to them and not to u.
  T u[9];
#pragma unroll
  for (int a = 0; a < 9; ++a) u[a] = sizeof(T) == 4 ? un[a] - un[4] : un[a];
  T gd[9], gs[9], od[9];   // d u_c / d x_c; d u_c / d x_(1-c), then the shear sum; the other component's diagonal
#pragma unroll
  for (int q = 0; q < 9; ++q) gd[q] = gs[q] = od[q] = T(0);
  if constexpr (NEED_U) {
    T bu[3][3], du[3][3];   // [qx][ay]
#pragma unroll
    for (int ay = 0; ay < 3; ++ay) {
      T o0[3], o1[3];
      line_values<T>(u[3 * ay], u[3 * ay + 1], u[3 * ay + 2], o0);
      line_derivs<T>(dx, u[3 * ay], u[3 * ay + 1], u[3 * ay + 2], o1);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        bu[q][ay] = o0[q];
        du[q][ay] = o1[q];
      }
    }
#pragma unroll
    for (int qx = 0; qx < 3; ++qx) {
      T gx[3], gy[3];
      line_values<T>(du[qx][0], du[qx][1], du[qx][2], gx);
      line_derivs<T>(dy, bu[qx][0], bu[qx][1], bu[qx][2], gy);
#pragma unroll
      for (int qy = 0; qy < 3; ++qy) {
        gd[qx + 3 * qy] = c == 0 ? gx[qy] : gy[qy];
        gs[qx + 3 * qy] = c == 0 ? gy[qy] : gx[qy];
      }
    }
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      od[q] = __shfl_xor_sync(0xffffffffu, gd[q], 16);
      if constexpr (VISC) gs[q] += __shfl_xor_sync(0xffffffffu, gs[q], 16);
    }
  }
  if (act) {
    T pi[3] = {T(0), T(0), T(0)};
    if constexpr ((MODE & (OP_AL | OP_B)) != 0) {
      T m[3] = {T(0), T(0), T(0)};
#pragma unroll
      for (int q = 0; q < 9; ++q) {
        const T dv = (cc.wdet * (Ref<T>::W(q % 3) * Ref<T>::W(q / 3))) * (gd[q] + od[q]);
        m[0] += dv;
        m[1] += Ref<T>::G(q % 3) * dv;
        m[2] += Ref<T>::G(q / 3) * dv;
      }
      if constexpr ((MODE & OP_B) != 0) {
        if (c == 0) {
#pragma unroll
          for (int k = 0; k < 3; ++k) p_out[(long long)cell * 3 + k] = -m[k];
        }
      }
      if constexpr ((MODE & OP_AL) != 0) {
        if (winv) {
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            T s = T(0);
#pragma unroll
            for (int k = 0; k < 3; ++k) s += winv[((long long)cell * 3 + q) * 3 + k] * m[k];
            pi[q] = cc.gamma * s;
          }
        } else {
#pragma unroll
          for (int q = 0; q < 3; ++q) pi[q] = cc.gamma * m[q] * (q == 0 ? cc.inv_m0 : cc.inv_m1);
        }
      }
    }
    if constexpr (NEED_FLUX) {
      if constexpr ((MODE & OP_BT) != 0) {
#pragma unroll
        for (int q = 0; q < 3; ++q) pi[q] -= p_in[(long long)cell * 3 + q];
      }
      // fluxes |J| w_q sigma_ck (2 / h_k is in the transposed derivative): gd <- sigma_cc, gs <- sigma_01
#pragma unroll
      for (int q = 0; q < 9; ++q) {
        const T iso = pi[0] + pi[1] * Ref<T>::G(q % 3) + pi[2] * Ref<T>::G(q / 3);
        const T w = cc.wdet * (Ref<T>::W(q % 3) * Ref<T>::W(q / 3));
        if constexpr (VISC && TENSOR) {
          // Mandel vector (e00, e11, r2 e01) and rows c and 2 of C, packed upper triangle
          const T* C = coef + ((long long)cell * 9 + q) * Sz<2>::NC;
          const T ir2 = T(0.70710678118654752440), es = ir2 * gs[q];
          const T ec = gd[q], eo = od[q];
          const T c2 = c == 0 ? C[2] : C[4], co = c == 0 ? C[4] : C[2];
          const T sc = (c == 0 ? C[0] : C[3]) * ec + C[1] * eo + c2 * es;
          const T ss = (c2 * ec + co * eo + C[5] * es) * ir2;
          gd[q] = w * (sc + iso);
          gs[q] = w * ss;
        } else if constexpr (VISC) {
          gd[q] = w * (mu[q] * (gd[q] + gd[q]) + iso);
          gs[q] = w * (mu[q] * gs[q]);
        } else {
          gd[q] = w * iso;
        }
      }
      T rx[3][3], ry[3][3];   // [ay][qx]
#pragma unroll
      for (int qx = 0; qx < 3; ++qx) {
        T f0[3], f1[3], o0[3], o1[3];
#pragma unroll
        for (int qy = 0; qy < 3; ++qy) {
          f0[qy] = c == 0 ? gd[qx + 3 * qy] : (VISC ? gs[qx + 3 * qy] : T(0));
          f1[qy] = c == 0 ? (VISC ? gs[qx + 3 * qy] : T(0)) : gd[qx + 3 * qy];
        }
        line_values_t<T, false>(f0[0], f0[1], f0[2], o0);
        line_derivs_t<T, false>(dy, f1[0], f1[1], f1[2], o1);
#pragma unroll
        for (int ay = 0; ay < 3; ++ay) {
          rx[ay][qx] = o0[ay];
          ry[ay][qx] = o1[ay];
        }
      }
#pragma unroll
      for (int ay = 0; ay < 3; ++ay) {
        T o[3];
        line_derivs_t<T, false>(dx, rx[ay][0], rx[ay][1], rx[ay][2], o);
        line_values_t<T, true>(ry[ay][0], ry[ay][1], ry[ay][2], o);
        store(ay, o);
      }
    }
  }
}

// warp: index of the warp among those of this apply
template <typename T, bool TENSOR, int MODE, bool STAGED, bool ZP>
__device__ __forceinline__ void apply_cells2_body(unsigned warp, const Geom& g, const Colour& col,
                                                  const CellConst<T>& cc, const T* __restrict__ x, T* __restrict__ y,
                                                  const T* __restrict__ coef, const T* __restrict__ p_in,
                                                  T* __restrict__ p_out, long long vstride, T* __restrict__ ebuf,
                                                  const T* __restrict__ winv, const PatchIn<T>& pin) {
  constexpr bool RAW = (MODE & OP_RAW) != 0;
  constexpr bool VISC = (MODE & OP_VISC) != 0;
  constexpr bool NEED_U = (MODE & (OP_VISC | OP_AL | OP_B)) != 0;
  x += blockIdx.y * vstride;
  y += blockIdx.y * vstride;
  const int lane = threadIdx.x & 31, c = lane >> 4;
  int cx = 0, cy = 0, cz = 0;
  const bool act = colour_cell(col, (long long)warp * 16 + (lane & 15), cx, cy, cz);
  const int cell = cx + g.n[0] * cy;
  pdl_wait();
  // the viscosities (constant) are in flight beside the nodal values
  T mu[VISC && !TENSOR ? 9 : 1];
  if constexpr (VISC && !TENSOR) {
#pragma unroll
    for (int q = 0; q < 9; ++q) mu[q] = act ? coef[(long long)cell * 9 + q] : T(0);
  }
  T u[9];
#pragma unroll
  for (int a = 0; a < 9; ++a) u[a] = T(0);
  if constexpr (NEED_U) {
    if (act) {
      if constexpr (ZP) {
        cell2_from_stars<T>(g, pin, c, cx, cy, u);
      } else {
#pragma unroll
        for (int a = 0; a < 9; ++a) {
          const int ni = 2 * cx + a % 3, nj = 2 * cy + a / 3;
          if (RAW || !on_boundary(g, ni, nj, 0)) u[a] = x[c * g.N + (ni + g.nn[0] * nj)];
        }
      }
    }
  }
  cell2_contribution<T, TENSOR, MODE>(cc, act, c, cell, u, mu, coef, p_in, p_out, winv, [&](int ay, const T(&o)[3]) {
    if constexpr (STAGED) {
      T* e = ebuf + (long long)stage_row(g, c, ay, 0, cy, 0) * (3 * g.n[0]) + 3 * cx;
#pragma unroll
      for (int ax = 0; ax < 3; ++ax) e[ax] = o[ax];
    } else {
#pragma unroll
      for (int ax = 0; ax < 3; ++ax) {
        const int ni = 2 * cx + ax, nj = 2 * cy + ay;
        if (RAW || !on_boundary(g, ni, nj, 0)) y[c * g.N + (ni + g.nn[0] * nj)] += o[ax];
      }
    }
  });
  pdl_trigger();
}
constexpr int C2_THREADS = 64, C2_CELLS = C2_THREADS / 2;
template <typename T, bool TENSOR, int MODE, bool STAGED, bool ZP>
__global__ void __launch_bounds__(C2_THREADS) k_apply_cells2(Geom g, Colour col, CellConst<T> cc,
                                                             const T* __restrict__ x, T* __restrict__ y,
                                                             const T* __restrict__ coef, const T* __restrict__ p_in,
                                                             T* __restrict__ p_out, long long vstride,
                                                             T* __restrict__ ebuf, const T* __restrict__ winv,
                                                             PatchIn<T> pin) {
  apply_cells2_body<T, TENSOR, MODE, STAGED, ZP>(blockIdx.x * (C2_THREADS / 32) + threadIdx.x / 32, g, col, cc, x, y,
                                                 coef, p_in, p_out, vstride, ebuf, winv, pin);
}
