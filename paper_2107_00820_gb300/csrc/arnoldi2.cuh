// A whole Arnoldi step of the 2D FP32 smoother in one launch.
//
// Included by tiles2.cu inside namespace als, after apply_cells.cuh.
//
// Step j:  V_j = w / hn - sum_i V_i coef_i  (Gram-Schmidt of the previous step, see k_gm_orth),
// Z_j = D^-1 V_j (star products and their node sums), w' = A Z_j, and the block partials of
// |V_j|^2 and V_i . w', i <= j.  As separate kernels (Gram-Schmidt, stars, cells, gather) a step is four
// launches, each 3 us of dependent latencies on levels this small: a 128^2 five-level cycle has 29 us of
// bytes to move and took 678.  Here a block owns the nodes of 8 x 8 cells and forms
// for itself what these depend on: V_j at the 21 x 21 nodes of the 10 x 10 stars that reach
// its cells, those stars' products (1.56 of its own number) and the outputs of 9 x 9 cells (1.27); only
// the sums cross blocks, and they go through the partials of the next launch.  The stars'
// inverses (69 KB) are copied to shared memory before the wait on the predecessor, so their
// transfer is hidden by it.  Sums within stars, nodes and cells run in the order of the separate
// kernels.  One cycle, us, separate / tiled: 16^2 two levels 166 / 128, 128^2 five levels
// 678 / 478 (112 / 106 and 375 / 351 when the column loops got the length KM, after the other steps; 105 and
// 354 with the state and the combinations of columns in double-float, see reduce.cuh).
//
// w goes through two buffers in turn (a block reads its neighbours' nodes of w while others write
// w'), and so do the partials; the last step's w' goes to column s for k_gm_orth.
// Blocks: one per tile, and for j > 0 one more for the one-thread bookkeeping of the step before.
#pragma once

struct ArnoldiArgs {
  Geom g;
  CellConst<float> cc;
  const float* coef;
  const float* winv;
  const void* inv;     // block-packed inverses of every vertex
  int j;
  int store;           // store V_j and the partials of its norm (all but a column 0 that is there already)
  const float* src;    // j = 0: V_0 or what it is a copy of; else w
  float* wout;
  float* z;
  float* V;
  long long ld;
  GmresDev st;
  DevStatus* status;
  int wait_polls;
};

template <typename TS>
struct Tile2 {
  static constexpr int T = 8, THREADS = RED_THREADS;
  static constexpr int S = T + 2, STARS = S * S;       // stars per axis, first vertex at cell - 1
  static constexpr int C = T + 1, CELLS = C * C;       // cells per axis, first cell - 1
  static constexpr int W = 2 * T + 5;                  // nodes per axis, first node 2 cell - 3
  static constexpr int FRAME = W * W - 4 * T * T;      // of them not in the square of the own ones
  static constexpr int SP = 128, CP = 96;              // padded star and cell counts in shared memory
  static constexpr int STRIDE = block_stride<TS>(18);
  static constexpr size_t inv_bytes = (size_t)STARS * STRIDE * sizeof(TS);
  static constexpr size_t y_bytes = 2 * 9 * SP * sizeof(float), r_bytes = 2 * W * W * sizeof(float);
  static constexpr size_t mu_bytes = 9 * CP * sizeof(float);
  // barrier | inverses, then cell outputs | y | V_j | viscosities
  static constexpr size_t smem = 128 + inv_bytes + y_bytes + r_bytes + mu_bytes;
  static_assert(THREADS == 4 * T * T && 2 * FRAME <= 2 * THREADS && STARS <= SP && CELLS <= CP, "tile shape");
  static_assert(2 * 9 * CP * sizeof(float) <= inv_bytes && inv_bytes % 16 == 0 && (STRIDE * sizeof(TS)) % 16 == 0, "shared memory");
};

__host__ __device__ __forceinline__ int tiles2_x(const Geom& g) { return (g.n[0] + 7) >> 3; }
__host__ __device__ __forceinline__ int tiles2(const Geom& g) { return tiles2_x(g) * ((g.n[1] + 7) >> 3); }

// the sum, rounded once, of the outputs [3 ay + ax][cell] (CN cells a row, CP apart) of the one, two or four cells
// of a node, e at the first of them; odd_x, odd_y: the node is in the middle of its cell along the axis
template <int CN, int CP>
__device__ __forceinline__ float node_sum2(const float* e, bool odd_x, bool odd_y) {
  const float* f = e + ((odd_y ? 3 : 6) + (odd_x ? 1 : 2)) * CP;
  const DF64 a = df_two_sum(f[0], odd_x ? 0.f : e[(odd_y ? 3 : 6) * CP + 1]);
  if (odd_y) return a.hi;   // (a sum of two is rounded once as it is)
  const DF64 b = df_two_sum(e[CN + (odd_x ? 1 : 2) * CP], odd_x ? 0.f : e[CN + 1]);
  const DF64 c = df_two_sum(a.hi, b.hi);
  return __fadd_rn(c.hi, __fadd_rn(__fadd_rn(a.lo, b.lo), c.lo));
}

// KM: the most columns before column j that this instance handles (the column loops are of that length)
template <typename TS, bool TENSOR, int KM>
__device__ __forceinline__ void arnoldi2_body(unsigned bx, const ArnoldiArgs& a, unsigned char* smraw) {
  using C = Tile2<TS>;
  constexpr int T = C::T, W = C::W;
  __shared__ float sh[RED_THREADS / 32][KMAXB];
  __shared__ DF64 coef[KMAXB], s_inv;
  __shared__ int s_fail;
  const Geom& g = a.g;
  const GmresDev& sd = a.st;
  const GmresView<DF64> st = gmres_view<float>(sd);
  const int j = KM == 0 ? 0 : a.j, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tx = tiles2_x(g), ntiles = tiles2(g);
  float acc[KMAXB];
  if ((int)bx == ntiles) {   // the bookkeeping block
    pdl_wait();
    pdl_trigger();
    sum_rows<float>(norm_rows<float>(sd, j - 1), norm_count(sd, j - 1, a.ld), 1, acc);
    const float v = block_total<float>(acc, 1, sh);
    if (tid == 0) {
      if (j == 1) gmres_start(st, to_small(v));
      else gmres_step(st, j - 2, to_small(v));
    }
    return;
  }
  uint64_t* bar = reinterpret_cast<uint64_t*>(smraw);
  TS* mats = reinterpret_cast<TS*>(smraw + 128);
  float* se = reinterpret_cast<float*>(smraw + 128);   // [component][3 ay + ax][cell], when the stars are done
  float* sy = reinterpret_cast<float*>(smraw + 128 + C::inv_bytes);   // [component][entry][star]
  float* rt = reinterpret_cast<float*>(smraw + 128 + C::inv_bytes + C::y_bytes);   // [component][node]
  float* smu = rt + 2 * W * W;                          // [point][cell]
  const int ty = (int)bx / tx, cx0 = ((int)bx - ty * tx) * T, cy0 = ty * T;
  if (tid == 0) {
    s_fail = 0;
    tma::mbar_init(bar, 1);
    tma::fence_init();
  }
  __syncthreads();
  if (warp == 0) {   // a copy per row of stars
    const int vx0 = cx0 > 0 ? cx0 - 1 : 0, vx1 = min(cx0 + T, g.n[0]);
    const int vy0 = cy0 > 0 ? cy0 - 1 : 0, vy1 = min(cy0 + T, g.n[1]);
    const uint32_t bytes = (uint32_t)((vx1 - vx0 + 1) * C::STRIDE * sizeof(TS));
    if (lane == 0) tma::mbar_expect_tx(bar, (uint32_t)(vy1 - vy0 + 1) * bytes);
    __syncwarp();
    const int vy = vy0 + lane;
    if (vy <= vy1)
      tma::bulk_load(mats + ((vy - cy0 + 1) * C::S + (vx0 - cx0 + 1)) * C::STRIDE,
                     static_cast<const TS*>(a.inv) + (long long)(vx0 + g.nv[0] * vy) * C::STRIDE, bytes, bar);
  }
  if constexpr (!TENSOR) {
    for (int e = tid; e < 9 * C::CELLS; e += C::THREADS) {
      const int ci = e / 9, k = e - 9 * ci, ly = ci / C::C, cx = cx0 - 1 + ci - ly * C::C, cy = cy0 - 1 + ly;
      smu[k * C::CP + ci] =
          cx >= 0 && cx < g.n[0] && cy >= 0 && cy < g.n[1] ? __ldg(a.coef + (long long)(cx + g.n[0] * cy) * 9 + k) : 0.f;
    }
  }
  // The thread's nodes: 0, 1 = the two components of a node of the tile's square, 2, 3 = of the frame
  // around it (the halo, and the last node column and row of the level, which their tile owns)
  int at[4], pos[4];
  bool own[4], in[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    int c = q, px, py;
    if (q < 2) {
      px = 3 + (tid & (2 * T - 1));
      py = 3 + tid / (2 * T);
    } else {
      int f = tid + (q - 2) * C::THREADS;
      c = f >= C::FRAME ? 1 : 0;
      f -= c * C::FRAME;
      if (f < 3 * W) {
        py = f / W;
        px = f - W * py;
      } else if (f < 5 * W) {
        py = (f - 3 * W) / W;
        px = (f - 3 * W) - W * py;
        py += 3 + 2 * T;
      } else {
        f -= 5 * W;
        py = f / 5;
        px = f - 5 * py;
        px += px < 3 ? 0 : 2 * T;
        py += 3;
      }
    }
    const int x = 2 * cx0 - 3 + px, y = 2 * cy0 - 3 + py;
    const bool slot = q < 2 || tid + (q - 2) * C::THREADS < 2 * C::FRAME;
    const bool there = slot && x >= 0 && x < g.nn[0] && y >= 0 && y < g.nn[1];
    at[q] = there ? c * (int)g.N + x + g.nn[0] * y : -1;
    pos[q] = slot ? (c * W + py) * W + px : -1;
    own[q] = there && px >= 3 && (px < 3 + 2 * T || x == g.nn[0] - 1) && py >= 3 && (py < 3 + 2 * T || y == g.nn[1] - 1);
    in[q] = there && x > 0 && x < g.nn[0] - 1 && y > 0 && y < g.nn[1] - 1;
  }
  // columns 0 .. j-2 come from kernels before the predecessor (complete before this launch began)
  constexpr int KA = KM > 0 ? KM : 1;
  float vc[4][KA];
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int c = 0; c < KM; ++c) vc[q][c] = c < j - 1 && at[q] >= 0 ? __ldcg(a.V + (long long)c * a.ld + at[q]) : 0.f;
  pdl_wait();
  pdl_trigger();
  // everything that the predecessor wrote is loaded at once: w, V_{j-1}, the partials (the first 256
  // blocks' here), 1 / hn
  float val[4], d[KA], dn = 0.f;
  DF64 rh{};
#pragma unroll
  for (int q = 0; q < 4; ++q) val[q] = at[q] >= 0 ? __ldcg(a.src + at[q]) : 0.f;
  if (j > 0) {
    const float *rows = dot_rows<float>(sd, j - 1), *nrows = norm_rows<float>(sd, j - 1);
    const int nbn = norm_count(sd, j - 1, a.ld);
#pragma unroll
    for (int c = 0; c < KM; ++c) d[c] = c < j && tid < sd.nbd ? __ldcg(rows + c * sd.nbd + tid) : 0.f;
    if (tid < nbn) dn = __ldcg(nrows + tid);
    if (lane < j - 1) rh = load_small(st.rhn + lane);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float last = at[q] >= 0 ? __ldcg(a.V + (long long)(j - 1) * a.ld + at[q]) : 0.f;
#pragma unroll
      for (int c = 0; c < KM; ++c)
        if (c == j - 1) vc[q][c] = last;
    }
    for (int b = tid + RED_THREADS; b < max(sd.nbd, nbn); b += RED_THREADS) {
#pragma unroll
      for (int c = 0; c < KM; ++c)
        if (c < j && b < sd.nbd) d[c] += __ldcg(rows + c * sd.nbd + b);
      if (b < nbn) dn += __ldcg(nrows + b);
    }
#pragma unroll
    for (int c = 0; c < KMAXB; ++c) acc[c] = c == j ? dn : c < KM ? d[c < KM ? c : 0] : 0.f;
    const float v = block_total<float>(acc, j + 1, sh);
    if (warp == 0) {
      DF64 nrm, inv;
      sqrt_recip(to_small(__shfl_sync(0xffffffffu, v, j)), nrm, inv);
      if (lane < j) {
        const DF64 rhni = lane == j - 1 ? inv : rh, h = to_small(v) * rhni * inv;
        coef[lane] = h * rhni;
        if (bx == 0) {
          st.H[(long long)(j - 1) * st.ldh + lane] = h;
          if (lane == j - 1) st.rhn[lane] = inv;
        }
      }
      if (lane == 0) s_inv = inv;
    }
    __syncthreads();
    const DF64 inv = s_inv;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      LinComb<float> sum(val[q]);
      sum.scale(inv);
#pragma unroll
      for (int c = 0; c < KM; ++c)
        if (c < j) sum.sub(vc[q][c], coef[c]);
      val[q] = sum.value();
    }
  }
  float nrm = 0.f;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (pos[q] >= 0) rt[pos[q]] = in[q] ? val[q] : 0.f;
    if (own[q] && a.store) {
      a.V[(long long)j * a.ld + at[q]] = val[q];
      nrm += val[q] * val[q];
    }
  }
  __syncthreads();
  // stars: 32 a warp pair, the two warps share the blocks of a star (see patches.cu)
  {
    const int role = warp & 1, s = (warp >> 1) * 32 + lane;
    const int sx = s % C::S, sr = s / C::S, vx = cx0 - 1 + sx, vy = cy0 - 1 + sr;
    const bool have = s < C::STARS && vx >= 0 && vx <= g.n[0] && vy >= 0 && vy <= g.n[1];
    float r0[9], r1[9], first[9], second[9];
#pragma unroll
    for (int o = 0; o < 9; ++o) {
      const int p = (2 * sr + o / 3) * W + 2 * sx + o % 3;
      r0[o] = have ? rt[p] : 0.f;
      r1[o] = have ? rt[W * W + p] : 0.f;
    }
    if (!tma::mbar_wait(bar, 0, a.wait_polls)) {
      report(a.status, 7 /* ALS_ETIMEOUT */, bx);
      s_fail = 1;
    }
    float* mine = sy + role * (9 * C::SP) + s;        // component `role` of star s
    float* other = sy + (1 - role) * (9 * C::SP) + s;
    if (have) {
      float p0[9], p1[9];   // to components 0 and 1
      star2_products<false, TS>(mats + (size_t)s * C::STRIDE, role, r0, r1, p0, p1);
#pragma unroll
      for (int o = 0; o < 9; ++o) {
        second[o] = role == 0 ? p0[o] : p1[o];
        other[o * C::SP] = role == 0 ? p1[o] : p0[o];
      }
    }
    __syncthreads();
    if (s_fail) {   // wait, at the default limit, for the copies in flight
      if (tid == 0) tma::mbar_wait(bar, 0);
      return;
    }
    if (have) {
#pragma unroll
      for (int o = 0; o < 9; ++o) first[o] = mine[o * C::SP];
#pragma unroll
      for (int o = 0; o < 9; ++o) mine[o * C::SP] = first[o] + second[o];
    }
  }
  // the older columns at the own nodes, for the dots: in flight over the cells
  float vd[2][KA];
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int c = 0; c < KM; ++c) vd[q][c] = c < j && own[q] ? __ldcg(a.V + (long long)c * a.ld + at[q]) : 0.f;
  __syncthreads();
  // cells: 16 a warp, the lanes i and i + 16 hold the components of cell i
  {
    const int ci = warp * 16 + (lane & 15), c = lane >> 4, ly = ci / C::C, lx = ci - ly * C::C;
    const int cx = cx0 - 1 + lx, cy = cy0 - 1 + ly;
    const bool act = ci < C::CELLS && cx >= 0 && cx < g.n[0] && cy >= 0 && cy < g.n[1];
    const int cell = cx + g.n[0] * cy;
    float mu[TENSOR ? 1 : 9];
    if constexpr (!TENSOR) {
#pragma unroll
      for (int q = 0; q < 9; ++q) mu[q] = act ? smu[q * C::CP + ci] : 0.f;
    }
    float u[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) u[k] = 0.f;
    if (act) {
      const float* ys = sy + c * (9 * C::SP) + ly * C::S + lx;
#pragma unroll
      for (int ay = 0; ay < 3; ++ay) {
        const int nj = 2 * cy + ay;
        const bool off = nj == 0 || nj == g.nn[1] - 1;
        float t[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int k = 0; k < (ay == 1 ? 2 : 1); ++k) {
          const int oy = ay == 1 ? 2 - 2 * k : 1;
          const float* p = ys + (ay == 1 ? k : ay >> 1) * C::S + 3 * oy * C::SP;
          t[0] += p[C::SP];
          t[1] += p[2 * C::SP] + p[1];
          t[2] += p[C::SP + 1];
        }
        u[3 * ay] = off || cx == 0 ? 0.f : t[0];
        u[3 * ay + 1] = off ? 0.f : t[1];
        u[3 * ay + 2] = off || cx == g.n[0] - 1 ? 0.f : t[2];
        if (lx > 0 && ly > 0 && (ay < 2 || cy == g.n[1] - 1)) {   // an own cell stores the nodes it owns
          float* z = a.z + (c * (int)g.N + g.nn[0] * nj + 2 * cx);
          z[0] = u[3 * ay];
          z[1] = u[3 * ay + 1];
          if (cx == g.n[0] - 1) z[2] = u[3 * ay + 2];
        }
      }
    }
    if (warp * 16 < C::CELLS) {
      cell2_contribution<float, TENSOR, OP_VISC | OP_AL>(
          a.cc, act, c, cell, u, mu, a.coef, nullptr, nullptr, a.winv, [&](int ay, const float(&o)[3]) {
            float* e = se + (c * 9 + 3 * ay) * C::CP + ci;
#pragma unroll
            for (int ax = 0; ax < 3; ++ax) e[ax * C::CP] = o[ax];
          });
    }
  }
  __syncthreads();
  // node sums, the dots and the norm
#pragma unroll
  for (int c = 0; c < KMAXB; ++c) acc[c] = 0.f;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (!own[q]) continue;
    float w = 0.f;
    if (q < 2 && in[q]) {
      const int lx = tid & (2 * T - 1), ly = tid / (2 * T);
      w = node_sum2<C::C, C::CP>(se + q * 9 * C::CP + ((ly + 1) >> 1) * C::C + ((lx + 1) >> 1), lx & 1, ly & 1);
    }
    a.wout[at[q]] = w;
    if (q < 2) {
#pragma unroll
      for (int c = 0; c <= KM; ++c) {
        if (c < KM && c < j) acc[c] += vd[q][c < KM ? c : 0] * w;
        if (c == j) acc[c] += val[q] * w;
      }
    }
  }
  const bool room = j + 1 < KMAXB;
#pragma unroll
  for (int c = 1; c < KMAXB; ++c)
    if (c == j + 1) acc[c] = nrm;
  const float v = block_total<float>(acc, room ? j + 2 : j + 1, sh);
  if (tid <= j) dot_rows<float>(sd, j)[tid * ntiles + bx] = v;
  if (room && tid == j + 1 && a.store) norm_rows<float>(sd, j)[bx] = v;
  if (!room && a.store) {
    __syncthreads();
    acc[0] = nrm;
    const float t = block_total<float>(acc, 1, sh);
    if (tid == 0) norm_rows<float>(sd, j)[bx] = t;
  }
}

template <typename TS, bool TENSOR, int KM>
__global__ void __launch_bounds__(RED_THREADS, 2) k_arnoldi2(const __grid_constant__ ArnoldiArgs a) {
  extern __shared__ __align__(128) unsigned char arnoldi_smem[];
  arnoldi2_body<TS, TENSOR, KM>(blockIdx.x, a, arnoldi_smem);
}
// merged launch (batch.cuh)
template <int KM>
__global__ void __launch_bounds__(RED_THREADS, 2) k_arnoldi2_b(const __grid_constant__ BatchTab<ArnoldiArgs> tb) {
  extern __shared__ __align__(128) unsigned char arnoldi_smem[];
  const int i = batch_slot(tb, blockIdx.x);
  arnoldi2_body<float, false, KM>(blockIdx.x - tb.start[i], tb.a[i], arnoldi_smem);
}
// the instance for step j: KM = 0, 2, 4 or 7
constexpr int kArnoldiKM = 4;
static int arnoldi_km(int j) { return j == 0 ? 0 : j <= 2 ? 1 : j <= 4 ? 2 : 3; }
template <typename TS, bool TENSOR>
static auto arnoldi_kernel(int i) {
  static constexpr decltype(&k_arnoldi2<TS, TENSOR, 0>) f[kArnoldiKM] = {
      k_arnoldi2<TS, TENSOR, 0>, k_arnoldi2<TS, TENSOR, 2>, k_arnoldi2<TS, TENSOR, 4>, k_arnoldi2<TS, TENSOR, 7>};
  return f[i];
}
static auto arnoldi_kernel_b(int i) {
  static constexpr decltype(&k_arnoldi2_b<0>) f[kArnoldiKM] = {k_arnoldi2_b<0>, k_arnoldi2_b<2>, k_arnoldi2_b<4>, k_arnoldi2_b<7>};
  return f[i];
}

// Which levels take their Arnoldi steps tiled: 2D, order 2, FP32, every vertex's inverse in one
// array, fewer than kTiledVertices vertices.  The repeated stars and cells cost more than the launches from about
// there on: one FP32 cycle, us, whose finest level takes tiles / separate kernels: 192^2 542 / 560, 256^2 740 / 666,
// 384^2 1652 / 1169 (16^2 and 128^2 above).
constexpr long long kTiledVertices = 32768;
bool arnoldi_tiled(const LevelDev& L, int prec) {
  return L.k == 2 && L.g.dim == 2 && prec == PREC_F32 && !L.split && L.g.nverts < kTiledVertices;
}
int arnoldi_tiles(const LevelDev& L) { return tiles2(L.g); }

static ArnoldiArgs arnoldi_args(const LevelDev& L, double gamma, const ArnoldiStep& e) {
  ArnoldiArgs a{};
  a.g = L.g;
  a.cc = cell_const<float>(L.g, gamma);
  a.coef = L.coef32;
  a.winv = L.winv32;
  a.inv = L.inv16 ? L.inv16 : (const void*)L.inv32;
  a.j = e.j;
  a.store = e.store;
  a.src = (const float*)e.src;
  a.wout = (float*)e.wout;
  a.z = (float*)e.z;
  a.V = (float*)e.V;
  a.ld = e.ld;
  a.st = e.st;
  a.status = L.status;
  a.wait_polls = L.wait_polls;
  return a;
}

// shared-memory opt-ins (before any capture)
void arnoldi_prepare() {
  const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
  const int f = (int)Tile2<float>::smem, h = (int)Tile2<__nv_bfloat16>::smem;
  for (int i = 0; i < kArnoldiKM; ++i) {
    cudaFuncSetAttribute(arnoldi_kernel<float, false>(i), at, f);
    cudaFuncSetAttribute(arnoldi_kernel<float, true>(i), at, f);
    cudaFuncSetAttribute(arnoldi_kernel<__nv_bfloat16, false>(i), at, h);
    cudaFuncSetAttribute(arnoldi_kernel<__nv_bfloat16, true>(i), at, h);
    cudaFuncSetAttribute(arnoldi_kernel_b(i), at, f);
  }
}

void arnoldi_step(const LevelDev& L, double gamma, const ArnoldiStep& e, cudaStream_t s) {
  const ArnoldiArgs a = arnoldi_args(L, gamma, e);
  const unsigned blocks = (unsigned)(tiles2(L.g) + (e.j > 0 ? 1 : 0));
  const size_t f = Tile2<float>::smem, h = Tile2<__nv_bfloat16>::smem;
  const int i = arnoldi_km(e.j);
  if (L.inv16) {
    if (L.tensor) launch_pdl(arnoldi_kernel<__nv_bfloat16, true>(i), blocks, RED_THREADS, h, s, a);
    else launch_pdl(arnoldi_kernel<__nv_bfloat16, false>(i), blocks, RED_THREADS, h, s, a);
  } else {
    if (L.tensor) launch_pdl(arnoldi_kernel<float, true>(i), blocks, RED_THREADS, f, s, a);
    else launch_pdl(arnoldi_kernel<float, false>(i), blocks, RED_THREADS, f, s, a);
  }
  count_launch(1);
}

int batch_arnoldi_step(const std::vector<BArnoldi>& items, cudaStream_t s) {
  std::vector<ArnoldiArgs> a;
  std::vector<unsigned> nb;
  for (const BArnoldi& it : items) {
    a.push_back(arnoldi_args(*it.L, it.gamma, it.e));
    nb.push_back((unsigned)(tiles2(it.L->g) + (it.e.j > 0 ? 1 : 0)));
  }
  const int n = launch_batch(arnoldi_kernel_b(arnoldi_km(items[0].e.j)), a, nb, RED_THREADS, Tile2<float>::smem, s);
  count_launch(n);
  return n;
}
