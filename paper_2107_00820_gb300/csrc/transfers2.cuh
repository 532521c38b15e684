// Tiled 2D FP32 operations beside the Arnoldi step (arnoldi2.cuh): the residual that starts a
// smoothing, and the robust transfers, one launch each.
//
// Included by tiles2.cu inside namespace als, after arnoldi2.cuh.
//
// As separate kernels a residual is two launches (cells, gather) and a transfer four (interior
// solves, cells, gather, interpolation), each a chain of latencies with little work.  The
// transfers are local to coarse cells: A_K^-1 acts on the 3 x 3 nodes inside coarse cell K, G couples
// those only to nodes of K's four fine cells, and the quadratic interpolation stays in K.  So a
// prolongation needs nothing from outside its coarse cells, and a restriction the coarse cells
// around its coarse nodes.  A block takes 8 x 8 fine cells (4 x 4 coarse ones); a restriction
// repeats a ring on two sides, 5 x 5 coarse cells.  One cycle, us, separate / tiled: 16^2 two levels
// 128 / 116, 128^2 five levels 478 / 397 (105 and 354 with what came after).
#pragma once

// u on a tile of nodes [component][node], W nodes a row, first node at a cell's corner -> the outputs of
// its CN x CN cells, se [component][3 ay + ax][cell] (CP cells apart); cell (0, 0) is (bx, by) of the
// level; cells outside it are left out
template <int MODE, bool TENSOR, int CN, int CP, int W>
__device__ __forceinline__ void cells2_tile(const Geom& g, const CellConst<float>& cc, int bx, int by, const float* nt,
                                            const float* smu, const float* __restrict__ coef,
                                            const float* __restrict__ winv, float* se) {
  const int lane = threadIdx.x & 31, c = lane >> 4;
  for (int w = threadIdx.x >> 5; w * 16 < CN * CN; w += RED_THREADS / 32) {
    const int ci = w * 16 + (lane & 15), ly = ci / CN, lx = ci - ly * CN, cx = bx + lx, cy = by + ly;
    const bool act = ci < CN * CN && cx >= 0 && cx < g.n[0] && cy >= 0 && cy < g.n[1];
    float u[9], mu[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) u[k] = act ? nt[(c * W + 2 * ly + k / 3) * W + 2 * lx + k % 3] : 0.f;
    if constexpr ((MODE & OP_VISC) != 0 && !TENSOR) {
#pragma unroll
      for (int k = 0; k < 9; ++k) mu[k] = act ? smu[k * CP + ci] : 0.f;
    }
    cell2_contribution<float, TENSOR, MODE>(cc, act, c, cx + g.n[0] * cy, u, mu, coef, nullptr, nullptr, winv,
                                            [&](int ay, const float(&o)[3]) {
                                              float* e = se + (c * 9 + 3 * ay) * CP + ci;
#pragma unroll
                                              for (int ax = 0; ax < 3; ++ax) e[ax * CP] = o[ax];
                                            });
  }
}
// their sum at node (px, py) of the tile, not on its rim; e: the component's outputs
template <int CN, int CP>
__device__ __forceinline__ float tile_sum2(const float* e, int px, int py) {
  const int cx = (px >> 1) - (px & 1 ? 0 : 1), cy = (py >> 1) - (py & 1 ? 0 : 1);   // the first of its cells
  return node_sum2<CN, CP>(e + cy * CN + cx, px & 1, py & 1);
}

// V_0 = b - A x (b - x at Dirichlet nodes) and the partials of its norm
struct Residual2Args {
  Geom g;
  CellConst<float> cc;
  const float* coef;
  const float* winv;
  const float* x;
  const float* b;
  float* y;
  GmresDev st;
};
template <bool TENSOR>
__device__ __forceinline__ void residual2_body(unsigned bx, const Residual2Args& a) {
  constexpr int T = 8, CN = T + 1, CP = 96, W = 2 * CN + 1;
  __shared__ float nt[2 * W * W], se[2 * 9 * CP], smu[9 * CP];
  const Geom& g = a.g;
  const int tid = threadIdx.x, tx = tiles2_x(g), ty = (int)bx / tx, cx0 = ((int)bx - ty * tx) * T, cy0 = ty * T;
  if constexpr (!TENSOR) {
    for (int e = tid; e < 9 * CN * CN; e += RED_THREADS) {
      const int ci = e / 9, k = e - 9 * ci, ly = ci / CN, cx = cx0 - 1 + ci - ly * CN, cy = cy0 - 1 + ly;
      smu[k * CP + ci] =
          cx >= 0 && cx < g.n[0] && cy >= 0 && cy < g.n[1] ? __ldg(a.coef + (long long)(cx + g.n[0] * cy) * 9 + k) : 0.f;
    }
  }
  constexpr int NQ = (2 * W * W + RED_THREADS - 1) / RED_THREADS;
  int at[NQ], flag[NQ];   // flag: 1 own, 2 free
  float xv[NQ], bv[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int e = tid + q * RED_THREADS, c = e >= W * W ? 1 : 0, f = e - c * W * W, py = f / W, px = f - W * py;
    const int x = 2 * cx0 - 2 + px, y = 2 * cy0 - 2 + py;
    const bool there = e < 2 * W * W && x >= 0 && x < g.nn[0] && y >= 0 && y < g.nn[1];
    at[q] = there ? c * (int)g.N + x + g.nn[0] * y : -1;
    const bool own = there && px >= 2 && (px < 2 + 2 * T || x == g.nn[0] - 1) && py >= 2 && (py < 2 + 2 * T || y == g.nn[1] - 1);
    flag[q] = (own ? 1 : 0) | (there && !on_boundary(g, x, y, 0) ? 2 : 0);
  }
  pdl_wait();
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    xv[q] = at[q] >= 0 ? __ldcg(a.x + at[q]) : 0.f;
    bv[q] = flag[q] & 1 ? __ldcg(a.b + at[q]) : 0.f;
  }
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int e = tid + q * RED_THREADS;
    if (e < 2 * W * W) nt[e] = flag[q] & 2 ? xv[q] : 0.f;
  }
  pdl_trigger();
  __syncthreads();
  cells2_tile<OP_VISC | OP_AL, TENSOR, CN, CP, W>(g, a.cc, cx0 - 1, cy0 - 1, nt, smu, a.coef, a.winv, se);
  __syncthreads();
  float acc[KMAXB] = {0.f};
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    if (!(flag[q] & 1)) continue;
    const int e = tid + q * RED_THREADS, c = e >= W * W ? 1 : 0, f = e - c * W * W, py = f / W, px = f - W * py;
    const float v = bv[q] - (flag[q] & 2 ? tile_sum2<CN, CP>(se + c * 9 * CP, px, py) : xv[q]);
    a.y[at[q]] = v;
    acc[0] += v * v;
  }
  store_partials<float>(a.st, 1, 1, acc, bx, tiles2(g));
}

// robust transfers between a level (gf) and the next coarser one (gc = gf / 2)
struct Transfer2Args {
  Geom gf, gc;
  CellConst<float> cc;
  const float* winv;
  const float* inv;    // block-packed inverses of every vertex of gf
  const float* in;     // restriction: rf;  prolongation: x_c
  float* out;          // restriction: r_c; prolongation: += (add) or =
  int add;
  DevStatus* status;
  int wait_polls;
};

// The local solves on coarse cells K of a tile, KN x KN of them, first (kx0, ky0): inverses copied to
// mats ahead of the wait (issue), the products of a star's blocks by two warps (products); part
// [role][component][entry][K]: y = part[1 - c][c] + part[c][c], the order of star2_store
template <int KN, int KP>
struct Interior2 {
  static constexpr int STRIDE = block_stride<float>(18);
  static_assert(KN * KN <= 32 && KP >= KN * KN, "a lane per star");
  static __device__ __forceinline__ bool vertex(const Geom& gc, int kx0, int ky0, int k, int& v, int nv0) {
    const int ly = k / KN, kx = kx0 + k - ly * KN, ky = ky0 + ly;
    v = (2 * kx + 1) + nv0 * (2 * ky + 1);
    return k < KN * KN && kx >= 0 && kx < gc.n[0] && ky >= 0 && ky < gc.n[1];
  }
  // one warp
  static __device__ __forceinline__ void issue(const Transfer2Args& a, int kx0, int ky0, float* mats, uint64_t* bar) {
    const int lane = threadIdx.x & 31;
    int v;
    const bool have = vertex(a.gc, kx0, ky0, lane, v, a.gf.nv[0]);
    const int n = __popc(__ballot_sync(0xffffffffu, have));
    if (lane == 0) tma::mbar_expect_tx(bar, (uint32_t)(n * STRIDE * 4));
    __syncwarp();
    if (have) tma::bulk_load(mats + lane * STRIDE, a.inv + (long long)v * STRIDE, STRIDE * 4, bar);
  }
  // warps 0 and 1; r(c, o, k): entry o of component c of star k
  template <typename R>
  static __device__ __forceinline__ void products(const Transfer2Args& a, int kx0, int ky0, const float* mats, R r,
                                                  float* part) {
    const int lane = threadIdx.x & 31, role = threadIdx.x >> 5;
    int v;
    if (!vertex(a.gc, kx0, ky0, lane, v, a.gf.nv[0])) return;
    float r0[9], r1[9], p0[9], p1[9];
#pragma unroll
    for (int o = 0; o < 9; ++o) {
      r0[o] = r(0, o, lane);
      r1[o] = r(1, o, lane);
    }
    star2_products<false, float>(mats + lane * STRIDE, role, r0, r1, p0, p1);
#pragma unroll
    for (int o = 0; o < 9; ++o) {
      part[((role * 2 + 0) * 9 + o) * KP + lane] = p0[o];
      part[((role * 2 + 1) * 9 + o) * KP + lane] = p1[o];
    }
  }
  static __device__ __forceinline__ float y(const float* part, int c, int o, int k) {
    return part[(((1 - c) * 2 + c) * 9 + o) * KP + k] + part[((c * 2 + c) * 9 + o) * KP + k];
  }
};

// every thread: wait for the copies; false (after the default limit for those in flight) on a timeout
__device__ __forceinline__ bool tile_copies_done(uint64_t* bar, int polls, DevStatus* status, unsigned bx, int* s_fail) {
  if (!tma::mbar_wait(bar, 0, polls)) {
    report(status, 7 /* ALS_ETIMEOUT */, bx);
    *s_fail = 1;
  }
  __syncthreads();
  if (!*s_fail) return true;
  if (threadIdx.x == 0) tma::mbar_wait(bar, 0);
  return false;
}

// r_c = P_H^T (r_f - G sum_K E_K A_K^-1 E_K^T r_f): 8 x 8 coarse nodes a block
__device__ __forceinline__ void restrict2_body(unsigned bx, const Transfer2Args& a) {
  constexpr int KN = 5, KP = 32, CN = 2 * KN, CP = 104, W = 4 * KN + 1, NN = 2 * W * W;
  using I2 = Interior2<KN, KP>;
  __shared__ __align__(128) float mats[KN * KN * I2::STRIDE];
  __shared__ float fr[NN], nt[NN], part[2 * 2 * 9 * KP], se[2 * 9 * CP];
  __shared__ __align__(8) uint64_t bar;
  __shared__ int s_fail;
  const Geom &gf = a.gf, &gc = a.gc;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int tx = (gc.n[0] + 3) >> 2, ty = (int)bx / tx, kx0 = 4 * ((int)bx - ty * tx) - 1, ky0 = 4 * ty - 1;
  if (tid == 0) {
    s_fail = 0;
    tma::mbar_init(&bar, 1);
    tma::fence_init();
  }
  __syncthreads();
  if (warp == 0) I2::issue(a, kx0, ky0, mats, &bar);
  constexpr int NQ = (NN + RED_THREADS - 1) / RED_THREADS;
  int at[NQ];   // -1 where r_f counts as 0: outside, or a Dirichlet node
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int e = tid + q * RED_THREADS, c = e >= W * W ? 1 : 0, f = e - c * W * W, py = f / W, px = f - W * py;
    const int x = 4 * kx0 + px, y = 4 * ky0 + py;
    at[q] = e < NN && x > 0 && x < gf.nn[0] - 1 && y > 0 && y < gf.nn[1] - 1 ? c * (int)gf.N + x + gf.nn[0] * y : -1;
  }
  pdl_wait();
  float v[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) v[q] = at[q] >= 0 ? __ldcg(a.in + at[q]) : 0.f;
#pragma unroll
  for (int q = 0; q < NQ; ++q)
    if (tid + q * RED_THREADS < NN) fr[tid + q * RED_THREADS] = v[q];
  pdl_trigger();
  if (!tile_copies_done(&bar, a.wait_polls, a.status, bx, &s_fail)) return;
  if (warp < 2)
    I2::products(a, kx0, ky0, mats,
                 [&](int c, int o, int k) { return fr[(c * W + 4 * (k / KN) + 1 + o / 3) * W + 4 * (k % KN) + 1 + o % 3]; },
                 part);
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int e = tid + q * RED_THREADS, c = e >= W * W ? 1 : 0, f = e - c * W * W, py = f / W, px = f - W * py;
    if (e < NN)
      nt[e] = at[q] >= 0 && (px & 3) && (py & 3) ? I2::y(part, c, (px & 3) - 1 + 3 * ((py & 3) - 1), (py >> 2) * KN + (px >> 2)) : 0.f;
  }
  __syncthreads();
  cells2_tile<OP_AL, false, CN, CP, W>(gf, a.cc, 2 * kx0, 2 * ky0, nt, nullptr, nullptr, a.winv, se);
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int e = tid + q * RED_THREADS, c = e >= W * W ? 1 : 0, f = e - c * W * W, py = f / W, px = f - W * py;
    if (at[q] >= 0 && px > 0 && px < W - 1 && py > 0 && py < W - 1) fr[e] = v[q] - tile_sum2<CN, CP>(se + c * 9 * CP, px, py);
  }
  __syncthreads();
  // coarse node (i, j) of the block's 8 x 8, and the last column and row of the level (Dirichlet)
  for (int e = tid; e < 2 * 81; e += RED_THREADS) {
    const int c = e >= 81 ? 1 : 0, f = e - c * 81, j = f / 9, i = f - 9 * j;
    const int mx = 2 * (kx0 + 1) + i, my = 2 * (ky0 + 1) + j;
    if (mx >= gc.nn[0] || my >= gc.nn[1] || (i == 8 && mx != gc.nn[0] - 1) || (j == 8 && my != gc.nn[1] - 1)) continue;
    float acc = 0.f;
    if (!on_boundary(gc, mx, my, 0)) {
      const float* p = fr + (c * W + 2 * j + 4) * W + 2 * i + 4;
      const bool ox = mx & 1, oy = my & 1;
      const float wx = ox ? 0.75f : 0.375f, wy = oy ? 0.75f : 0.375f;
#pragma unroll
      for (int t = 0; t < 5; ++t) {
        if (oy && t >= 3) continue;
        const float* r = p + (t == 0 ? 0 : t == 1 ? -1 : t == 2 ? 1 : t == 3 ? -3 : 3) * W;
        float s = 0.f;
        s += r[0];
        s += wx * r[-1];
        s += wx * r[1];
        if (!ox) {
          s += -0.125f * r[-3];
          s += -0.125f * r[3];
        }
        acc += (t == 0 ? 1.f : t < 3 ? wy : -0.125f) * s;
      }
    }
    a.out[c * (int)gc.N + mx + gc.nn[0] * my] = acc;
  }
}

// x (+)= (I - sum_K E_K A_K^-1 E_K^T G) P_H x_c: the fine nodes of 4 x 4 coarse cells a block
__device__ __forceinline__ void prolong2_body(unsigned bx, const Transfer2Args& a) {
  constexpr int KN = 4, KP = 17, CN = 2 * KN, CP = 72, W = 4 * KN + 1, NN = 2 * W * W, WC = 2 * KN + 1, NC = 2 * WC * WC;
  using I2 = Interior2<KN, KP>;
  __shared__ __align__(128) float mats[KN * KN * I2::STRIDE];
  __shared__ float cs[NC], nt[NN], rs[2 * 9 * KP], part[2 * 2 * 9 * KP], se[2 * 9 * CP];
  __shared__ __align__(8) uint64_t bar;
  __shared__ int s_fail;
  const Geom &gf = a.gf, &gc = a.gc;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int tx = (gc.n[0] + 3) >> 2, ty = (int)bx / tx, kx0 = 4 * ((int)bx - ty * tx), ky0 = 4 * ty;
  if (tid == 0) {
    s_fail = 0;
    tma::mbar_init(&bar, 1);
    tma::fence_init();
  }
  __syncthreads();
  if (warp == 0) I2::issue(a, kx0, ky0, mats, &bar);
  constexpr int NQ = (NN + RED_THREADS - 1) / RED_THREADS;
  int at[NQ], own = 0;   // -1 outside; own: bit q, a free node that this block writes
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int e = tid + q * RED_THREADS, c = e >= W * W ? 1 : 0, f = e - c * W * W, py = f / W, px = f - W * py;
    const int x = 4 * kx0 + px, y = 4 * ky0 + py;
    const bool there = e < NN && x < gf.nn[0] && y < gf.nn[1];
    at[q] = there ? c * (int)gf.N + x + gf.nn[0] * y : -1;
    if (there && (px < W - 1 || x == gf.nn[0] - 1) && (py < W - 1 || y == gf.nn[1] - 1)) own |= 1 << q;
  }
  int ca = -1;   // NC <= RED_THREADS: a coarse value a thread
  static_assert(NC <= RED_THREADS, "one coarse value a thread");
  if (tid < NC) {
    const int c = tid >= WC * WC ? 1 : 0, f = tid - c * WC * WC, j = f / WC, i = f - WC * j;
    const int mx = 2 * kx0 + i, my = 2 * ky0 + j;
    if (mx > 0 && mx < gc.nn[0] - 1 && my > 0 && my < gc.nn[1] - 1) ca = c * (int)gc.N + mx + gc.nn[0] * my;
  }
  pdl_wait();
  const float cv = ca >= 0 ? __ldcg(a.in + ca) : 0.f;
  float xv[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) xv[q] = a.add && (own >> q & 1) ? __ldcg(a.out + at[q]) : 0.f;
  if (tid < NC) cs[tid] = cv;
  pdl_trigger();
  if (!tile_copies_done(&bar, a.wait_polls, a.status, bx, &s_fail)) return;
  float tv[NQ];   // P_H x_c
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int e = tid + q * RED_THREADS, c = e >= W * W ? 1 : 0, f = e - c * W * W, py = f / W, px = f - W * py;
    tv[q] = 0.f;
    if (at[q] >= 0 && !on_boundary(gf, 4 * kx0 + px, 4 * ky0 + py, 0)) {
      // the taps one after another (y, then x) as in prolong_body of transfer.cu, with its products: the correction
      // that follows amplifies a change of rounding here by gamma / mu
      const int ix = px & 1 ? 2 * (px >> 2) : px >> 1, iy = py & 1 ? 2 * (py >> 2) : py >> 1;
      const float ax = (px & 3) == 1 ? 0.375f : -0.125f, bx2 = (px & 3) == 1 ? -0.125f : 0.375f;
      const float ay = (py & 3) == 1 ? 0.375f : -0.125f, by2 = (py & 3) == 1 ? -0.125f : 0.375f;
      const float* p = cs + (c * WC + iy) * WC + ix;
      float t = 0.f;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        if (k > 0 && !(py & 1)) continue;
        const float w = !(py & 1) ? 1.f : k == 0 ? ay : k == 1 ? 0.75f : by2;   // dyadic: every product of weights is exact
        const float* r = p + k * WC;
        if (px & 1) {
          t += (ax * w) * r[0];
          t += (0.75f * w) * r[1];
          t += (bx2 * w) * r[2];
        } else {
          t += w * r[0];
        }
      }
      tv[q] = t;
    }
    if (e < NN) nt[e] = tv[q];
  }
  __syncthreads();
  cells2_tile<OP_AL, false, CN, CP, W>(gf, a.cc, 2 * kx0, 2 * ky0, nt, nullptr, nullptr, a.winv, se);
  __syncthreads();
  for (int e = tid; e < KN * KN * 18; e += RED_THREADS) {
    const int k = e & (KN * KN - 1), i = e / (KN * KN), c = i / 9, o = i - 9 * c;
    rs[i * KP + k] = tile_sum2<CN, CP>(se + c * 9 * CP, 4 * (k % KN) + 1 + o % 3, 4 * (k / KN) + 1 + o / 3);
  }
  __syncthreads();
  if (warp < 2) I2::products(a, kx0, ky0, mats, [&](int c, int o, int k) { return rs[(c * 9 + o) * KP + k]; }, part);
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    if (!(own >> q & 1)) continue;
    const int e = tid + q * RED_THREADS, c = e >= W * W ? 1 : 0, f = e - c * W * W, py = f / W, px = f - W * py;
    float r = xv[q] + tv[q];
    if ((px & 3) && (py & 3)) r -= I2::y(part, c, (px & 3) - 1 + 3 * ((py & 3) - 1), (py >> 2) * KN + (px >> 2));
    a.out[at[q]] = r;
  }
}

template <bool TENSOR>
__global__ void __launch_bounds__(RED_THREADS) k_residual2(const __grid_constant__ Residual2Args a) {
  residual2_body<TENSOR>(blockIdx.x, a);
}
__global__ void __launch_bounds__(RED_THREADS) k_restrict2(const __grid_constant__ Transfer2Args a) {
  restrict2_body(blockIdx.x, a);
}
__global__ void __launch_bounds__(RED_THREADS) k_prolong2(const __grid_constant__ Transfer2Args a) {
  prolong2_body(blockIdx.x, a);
}
// merged launches (batch.cuh)
__global__ void __launch_bounds__(RED_THREADS) k_residual2_b(const __grid_constant__ BatchTab<Residual2Args> tb) {
  const int i = batch_slot(tb, blockIdx.x);
  residual2_body<false>(blockIdx.x - tb.start[i], tb.a[i]);
}
__global__ void __launch_bounds__(RED_THREADS) k_restrict2_b(const __grid_constant__ BatchTab<Transfer2Args> tb) {
  const int i = batch_slot(tb, blockIdx.x);
  restrict2_body(blockIdx.x - tb.start[i], tb.a[i]);
}
__global__ void __launch_bounds__(RED_THREADS) k_prolong2_b(const __grid_constant__ BatchTab<Transfer2Args> tb) {
  const int i = batch_slot(tb, blockIdx.x);
  prolong2_body(blockIdx.x - tb.start[i], tb.a[i]);
}

static Residual2Args residual2_args(const LevelDev& L, double gamma, const void* x, const void* b, void* y,
                                    const GmresDev& st) {
  return Residual2Args{L.g, cell_const<float>(L.g, gamma), L.coef32, L.winv32, (const float*)x, (const float*)b,
                       (float*)y, st};
}
void tiled_residual(const LevelDev& L, double gamma, const void* x, const void* b, void* y, const GmresDev& st,
                    cudaStream_t s) {
  const Residual2Args a = residual2_args(L, gamma, x, b, y, st);
  if (L.tensor) launch_pdl(k_residual2<true>, (unsigned)tiles2(L.g), RED_THREADS, 0, s, a);
  else launch_pdl(k_residual2<false>, (unsigned)tiles2(L.g), RED_THREADS, 0, s, a);
  count_launch(1);
}
int batch_tiled_residual(const std::vector<BApply>& items, cudaStream_t s) {
  std::vector<Residual2Args> a;
  std::vector<unsigned> nb;
  for (const BApply& it : items) {
    a.push_back(residual2_args(*it.L, it.gamma, it.x, it.e.b, it.y, it.e.st));
    nb.push_back((unsigned)tiles2(it.L->g));
  }
  const int n = launch_batch(k_residual2_b, a, nb, RED_THREADS, 0, s);
  count_launch(n);
  return n;
}

// Tiled transfers: as the tiled steps, with the inverses in float
bool transfer_tiled(const LevelDev& fine, int prec) { return arnoldi_tiled(fine, prec) && !fine.inv16; }

static Transfer2Args transfer2_args(const LevelDev& coarse, const LevelDev& fine, double gamma, const void* in, void* out,
                                    int add) {
  return Transfer2Args{fine.g, coarse.g, cell_const<float>(fine.g, gamma), fine.winv32, fine.inv32, (const float*)in,
                       (float*)out, add, fine.status, fine.wait_polls};
}
static unsigned transfer2_blocks(const Geom& gc) { return (unsigned)(((gc.n[0] + 3) >> 2) * ((gc.n[1] + 3) >> 2)); }

void tiled_restrict(const LevelDev& coarse, const LevelDev& fine, double gamma, const void* rf, void* rc, cudaStream_t s) {
  launch_pdl(k_restrict2, transfer2_blocks(coarse.g), RED_THREADS, 0, s, transfer2_args(coarse, fine, gamma, rf, rc, 0));
  count_launch(1);
}
void tiled_prolong(const LevelDev& coarse, const LevelDev& fine, double gamma, const void* xc, void* x, int add,
                   cudaStream_t s) {
  launch_pdl(k_prolong2, transfer2_blocks(coarse.g), RED_THREADS, 0, s, transfer2_args(coarse, fine, gamma, xc, x, add));
  count_launch(1);
}
static int batch_transfer2(void (*k)(BatchTab<Transfer2Args>), const std::vector<BTiledTransfer>& items, cudaStream_t s) {
  std::vector<Transfer2Args> a;
  std::vector<unsigned> nb;
  for (const BTiledTransfer& it : items) {
    a.push_back(transfer2_args(*it.coarse, *it.fine, it.gamma, it.in, it.out, 1));
    nb.push_back(transfer2_blocks(it.coarse->g));
  }
  const int n = launch_batch(k, a, nb, RED_THREADS, 0, s);
  count_launch(n);
  return n;
}
int batch_tiled_restrict(const std::vector<BTiledTransfer>& items, cudaStream_t s) {
  return batch_transfer2(k_restrict2_b, items, s);
}
int batch_tiled_prolong(const std::vector<BTiledTransfer>& items, cudaStream_t s) {
  return batch_transfer2(k_prolong2_b, items, s);
}
