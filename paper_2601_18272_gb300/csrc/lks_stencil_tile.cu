// Tiled forms of the D2Q9 predictor and its transpose for grids too small to fill the chip with long
// strips (lks_stencil.cu states the method and holds the strip forms).
//
// A strip of two rows, all that a small grid leaves a warp, works on six rows to write two, one after
// the other. Here a CTA takes a tile of TX x TY cells: its threads stage the tile with a halo of two
// in shared memory, form the nine f_i^eq (or the six moments of the transpose) on the halo of one,
// one node each, and gather the outputs. The halo costs (1 + 2/TX)(1 + 2/TY) instead of three, and
// the chain is three phases long. In FP64, where a warp instruction costs its scheduler 64 cycles,
// small tiles also spread the work over all schedulers.
//
// Boundary nodes take the values of the interior node their rule copies from: the gather is made at
// the node clamped to the interior, then walls zero u, then the open planes prescribe their part.
#include "lks_kernels.h"
#include "lks_stencil_common.cuh"

namespace lks {

namespace {

template <typename T>
__device__ __forceinline__ T third() { return T(1.0 / 3.0); }

// Tile of this CTA: first column and row of the cells it stages for (the last tile is moved back onto
// the grid so that every boundary node has its inward neighbours in the tile), and of those it writes.
template <int TX, int TY>
struct Tile {
  int x0, y0, ox, oy;
  __device__ __forceinline__ explicit Tile(const Geo& g) {
    ox = blockIdx.x * TX;
    oy = blockIdx.y * TY;
    x0 = min(ox, max(0, g.n[0] - TX));
    y0 = min(oy, max(0, g.n[1] - TY));
  }
};

// Grid index of node (x, y), wrapped on periodic axes; false off the grid.
__device__ __forceinline__ bool grid_node(const Geo& g, int& x, int& y) {
  if (g.bc[0] == BC_PERIODIC) x = wrapi(x, g.n[0]);
  if (g.bc[1] == BC_PERIODIC) y = wrapi(y, g.n[1]);
  return x >= 0 && x < g.n[0] && y >= 0 && y < g.n[1];
}

__device__ __forceinline__ int clamp_interior(int bc, int n, int v) {
  return bc == BC_PERIODIC ? v : min(max(v, 1), n - 2);
}

template <typename T, int TX, int TY, int NT>
__global__ void __launch_bounds__(NT) k_tile2d_fwd(Geo g, Slots<T> S, const Ctrl* __restrict__ ctrl, int di) {
  constexpr int RX = TX + 4, RY = TY + 4, FX = TX + 2, FY = TY + 2;
  __shared__ T u[2][RY * RX];
  __shared__ T f[9][FY * FX];
  const int t = ctrl->t0 + di, base = ctrl->base, tid = threadIdx.x;
  const T* __restrict__ src = slot_ptr(S, t - 1, base);
  T* __restrict__ dst = slot_ptr(S, t, base);
  const Tile<TX, TY> tl(g);
  const int nx = g.n[0], ny = g.n[1];
  const long long N = g.N;
  for (int q = tid; q < RX * RY; q += NT) {  // u under the ghost rule
    int x = tl.x0 - 2 + q % RX, y = tl.y0 - 2 + q / RX, sg = 1;
    const bool ok = ghost_axis(g.bc[0], nx, &x, &sg) && ghost_axis(g.bc[1], ny, &y, &sg);
    const long long n = ok ? x + (long long)nx * y : 0;
    u[0][q] = ok ? T(sg) * src[N + n] : T(0);
    u[1][q] = ok ? T(sg) * src[2 * N + n] : T(0);
  }
  const T K = two_a<T>(g) * T(1.0 / 6.0);
  __syncthreads();
  for (int q = tid; q < FX * FY; q += NT) {
    const int ci = q % FX, cj = q / FX;
    int x = tl.x0 - 1 + ci, y = tl.y0 - 1 + cj;
    if (!grid_node(g, x, y)) continue;  // (no interior node reads it)
    const T p = src[x + (long long)nx * y];
    const T* a = &u[0][cj * RX + ci];  // row below, shifted one column left
    const T* b = &u[1][cj * RX + ci];
    const T ux = a[RX + 1], uy = b[RX + 1];
    // 6 G_xx, 6 G_yy, 6 (G_xy + G_yx) as raw stencil sums
    const T ne = a[2 * RX + 2], nw = a[2 * RX], se = a[2], sw = a[0];
    const T gxx = ((ne - nw) + (se - sw)) + (a[RX + 2] - a[RX]);
    const T gxy = ((ne - se) + (nw - sw)) + (a[2 * RX + 1] - a[1]);
    const T me = b[2 * RX + 2], mw = b[2 * RX], oe = b[2], ow = b[0];
    const T gyy = ((me - oe) + (mw - ow)) + (b[2 * RX + 1] - b[1]);
    const T gyx = ((me - mw) + (oe - ow)) + (b[RX + 2] - b[RX]);
    // with d = 3p + 3 |u|^2 + K (Gxx + Gyy), qxy = 9 ux uy + K (Gxy + Gyx):
    //   f0 = 4/9 a, f1,3 = 1/9 (a + 9/2 ux^2 + K Gxx) +- ux/3, f5..8 = 1/36 (d +- qxy) + (+-ux +-uy)/12
    const T ux2 = ux * ux, uy2 = uy * uy, s2 = ux2 + uy2, p3 = T(3) * p;
    const T kxx = K * gxx, kyy = K * gyy, kxy = K * (gxy + gyx);
    const T e = fma(T(-1.5), s2, p3);
    const T h1 = T(1.0 / 9.0) * (fma(T(4.5), ux2, e) + kxx), v1 = T(1.0 / 3.0) * ux;
    const T h2 = T(1.0 / 9.0) * (fma(T(4.5), uy2, e) + kyy), v2 = T(1.0 / 3.0) * uy;
    const T d36 = T(1.0 / 36.0) * (fma(T(3), s2, p3) + kxx + kyy);
    const T q36 = T(1.0 / 36.0) * fma(T(9) * ux, uy, kxy);
    const T bx = T(1.0 / 12.0) * ux, by = T(1.0 / 12.0) * uy;
    const T e1 = d36 + q36, e2 = d36 - q36, s1 = bx + by, sm = bx - by;
    f[0][q] = T(4.0 / 9.0) * e;
    f[1][q] = h1 + v1;
    f[3][q] = h1 - v1;
    f[2][q] = h2 + v2;
    f[4][q] = h2 - v2;
    f[5][q] = e1 + s1;
    f[7][q] = e1 - s1;
    f[6][q] = e2 - sm;
    f[8][q] = e2 + sm;
  }
  __syncthreads();
  for (int q = tid; q < TX * TY; q += NT) {
    const int x = tl.x0 + q % TX, y = tl.y0 + q / TX;
    if (x < tl.ox || y < tl.oy || x >= nx || y >= ny) continue;
    const int xc = clamp_interior(g.bc[0], nx, x), yc = clamp_interior(g.bc[1], ny, y);
    const int c = (yc - tl.y0 + 1) * FX + (xc - tl.x0 + 1);
    const T f1 = f[1][c - 1], f3 = f[3][c + 1], f2 = f[2][c - FX], f4 = f[4][c + FX];
    const T f5 = f[5][c - FX - 1], f6 = f[6][c - FX + 1], f7 = f[7][c + FX + 1], f8 = f[8][c + FX - 1];
    const T s57 = f5 + f7, s68 = f6 + f8, d57 = f5 - f7, d86 = f8 - f6;
    T P = third<T>() * ((f[0][c] + (f1 + f3) + (f2 + f4)) + (s57 + s68));
    T X = (f1 - f3) + (d57 + d86), Y = (f2 - f4) + (d57 - d86);
    if (yc != y) X = Y = T(0);  // no-slip wall
    if (xc != x) {
      if (x != 0) {
        P = T(0);
      } else if (g.bc[0] == BC_INFLOW_OUTFLOW) {
        X = T(g.u_in);
        Y = T(0);
      } else {
        P = T(g.dp);
      }
    }
    const long long n = x + (long long)nx * y;
    dst[n] = P;
    dst[N + n] = X;
    dst[2 * N + n] = Y;
  }
}

// Adjoint of (p*, u*) at grid node (x, y) with the boundary rules reversed: zero on boundary nodes,
// what the rules copied from the node added to it.
template <typename T>
__device__ __forceinline__ void routed(const Geo& g, const T* __restrict__ L, int x, int y, T* p, T* a, T* b) {
  const long long N = g.N;
  const int nx = g.n[0], ny = g.n[1];
  *p = *a = *b = T(0);
  if (!interior_axis(g.bc[0], nx, x) || !interior_axis(g.bc[1], ny, y)) return;
  auto ld = [&](int plane, int xx, int yy) { return L[plane * N + xx + (long long)nx * yy]; };
  *p = ld(0, x, y);
  *a = ld(1, x, y);
  *b = ld(2, x, y);
  const int bx = g.bc[0];
  const bool inl = bx == BC_INFLOW_OUTFLOW && x == 1;
  if (inl) *p += ld(0, 0, y);
  if (g.bc[1] == BC_WALL && (y == 1 || y == ny - 2)) {
    const int yw = (y == 1) ? 0 : ny - 1;
    *p += ld(0, x, yw);
    if (inl) *p += ld(0, 0, yw);
  }
  if (bx != BC_PERIODIC && x == nx - 2) {
    *a += ld(1, nx - 1, y);
    *b += ld(2, nx - 1, y);
  }
  if (bx == BC_PRESSURE && x == 1) {
    *a += ld(1, 0, y);
    *b += ld(2, 0, y);
  }
}

template <typename T, int TX, int TY, int NT>
__global__ void __launch_bounds__(NT) k_tile2d_adj(Geo g, Slots<T> S, T* Lb, long long lstride,
                                                   const Ctrl* __restrict__ ctrl, int di) {
  constexpr int RX = TX + 4, RY = TY + 4, FX = TX + 2, FY = TY + 2;
  __shared__ T l[3][RY * RX];  // lam_p* / 3, lam_u*
  __shared__ T m[6][FY * FX];  // P, Ux, Uy, Sxx, Syy, Sxy
  const int t = ctrl->t0 - di, base = ctrl->base, tid = threadIdx.x;
  const T* __restrict__ Lcur = Lb + (long long)(t & 1) * lstride;
  T* __restrict__ Lnext = Lb + (long long)((t - 1) & 1) * lstride;
  const T* __restrict__ su = slot_ptr(S, t - 1, base);
  const Tile<TX, TY> tl(g);
  const int nx = g.n[0], ny = g.n[1];
  const long long N = g.N;
  for (int q = tid; q < RX * RY; q += NT) {
    int x = tl.x0 - 2 + q % RX, y = tl.y0 - 2 + q / RX;
    T p = T(0), a = T(0), b = T(0);
    if (grid_node(g, x, y)) routed(g, Lcur, x, y, &p, &a, &b);
    l[0][q] = third<T>() * p;
    l[1][q] = a;
    l[2][q] = b;
  }
  __syncthreads();
  for (int q = tid; q < FX * FY; q += NT) {
    const int ci = q % FX, cj = q / FX;
    int x = tl.x0 - 1 + ci, y = tl.y0 - 1 + cj;
    const bool ok = grid_node(g, x, y);
    const int c = (cj + 1) * RX + ci + 1;
    auto tp = [&](int o) { return l[0][c + o]; };
    auto la = [&](int o) { return l[1][c + o]; };
    auto lb = [&](int o) { return l[2][c + o]; };
    const T g1 = tp(1) + la(1), g3 = tp(-1) - la(-1), g2 = tp(RX) + lb(RX), g4 = tp(-RX) - lb(-RX);
    const T g5 = tp(RX + 1) + (la(RX + 1) + lb(RX + 1)), g7 = tp(-RX - 1) - (la(-RX - 1) + lb(-RX - 1));
    const T g6 = tp(RX - 1) - (la(RX - 1) - lb(RX - 1)), g8 = tp(-RX + 1) + (la(-RX + 1) - lb(-RX + 1));
    const T w0 = T(4.0 / 9.0), w1 = T(1.0 / 9.0), w5 = T(1.0 / 36.0);
    const T s57 = g5 + g7, s68 = g6 + g8, d57 = g5 - g7, d86 = g8 - g6;
    const T sd = w5 * (s57 + s68), sx = fma(w1, g1 + g3, sd), ax = w1 * (g2 + g4);
    m[0][q] = ok ? fma(w0, tp(0), sx + ax) : T(0);
    m[1][q] = ok ? fma(w1, g1 - g3, w5 * (d57 + d86)) : T(0);
    m[2][q] = ok ? fma(w1, g2 - g4, w5 * (d57 - d86)) : T(0);
    m[3][q] = ok ? sx : T(0);  // (S is zero off the grid)
    m[4][q] = ok ? ax + sd : T(0);
    m[5][q] = ok ? w5 * (s57 - s68) : T(0);
  }
  const T kA = two_a<T>(g) * T(1.0 / 6.0);
  __syncthreads();
  for (int q = tid; q < TX * TY; q += NT) {
    const int x = tl.x0 + q % TX, y = tl.y0 + q / TX;
    if (x < tl.ox || y < tl.oy || x >= nx || y >= ny) continue;
    const int c = (y - tl.y0 + 1) * FX + (x - tl.x0 + 1);
    const T *xx = m[3], *yy = m[4], *xy = m[5];
    // h_a(z) = sum_j c_j . S_a(z - c_j)
    const T hx0 = (xx[c - 1] - xx[c + 1]) + (xy[c - FX] - xy[c + FX]);
    const T hy0 = (xy[c - 1] - xy[c + 1]) + (yy[c - FX] - yy[c + FX]);
    const int sw = c - FX - 1, se = c - FX + 1, nw = c + FX - 1, ne = c + FX + 1;
    T hx = hx0 + ((xx[sw] - xx[ne]) + (xy[sw] - xy[ne])) + ((xx[nw] - xx[se]) - (xy[nw] - xy[se]));
    T hy = hy0 + ((xy[sw] - xy[ne]) + (yy[sw] - yy[ne])) + ((xy[nw] - xy[se]) - (yy[nw] - yy[se]));
    // the gradient's ghost nodes: an open plane's copies the boundary node, a wall's reflects with a
    // sign flip onto the next row; their h folds back onto the node
    const bool gx = g.bc[0] != BC_PERIODIC && (x == 0 || x == nx - 1);
    const bool gy = g.bc[1] == BC_WALL && (y == 1 || y == ny - 2);
    if (gx || gy) {
      auto ghost = [&](int zx, int zy, T sg) {
        for (int j = 0; j < 8; ++j) {
          const int cx = j < 4 ? (j == 0) - (j == 2) : ((j == 4 || j == 7) ? 1 : -1);
          const int cy = j < 4 ? (j == 1) - (j == 3) : (j < 6 ? 1 : -1);
          const int qx = zx - cx - tl.x0 + 1, qy = zy - cy - tl.y0 + 1;
          if (qx < 0 || qx >= FX || qy < 0 || qy >= FY) continue;  // (off the grid there: S = 0)
          const int o = qy * FX + qx;
          hx += sg * (T(cx) * xx[o] + T(cy) * xy[o]);
          hy += sg * (T(cx) * xy[o] + T(cy) * yy[o]);
        }
      };
      const int zx = x == 0 ? -1 : nx, zy = y == 1 ? -1 : ny;
      if (gx) ghost(zx, y, T(1));
      if (gy) ghost(x, zy, T(-1));
      if (gx && gy) ghost(zx, zy, T(-1));
    }
    const long long n = x + (long long)nx * y;
    const T ux = su[N + n], uy = su[2 * N + n];
    const T P = m[0][c], P3 = T(3) * P;
    Lnext[n] = P3;
    Lnext[N + n] = fma(kA, hx, fma(T(9), xx[c] * ux + xy[c] * uy, T(3) * m[1][c] - ux * P3));
    Lnext[2 * N + n] = fma(kA, hy, fma(T(9), xy[c] * ux + yy[c] * uy, T(3) * m[2][c] - uy * P3));
  }
}

template <typename T, int TX, int TY, int NT>
void fwd_shape(const Geo& g, const Slots<T>& S, const Ctrl* ctrl, int di, cudaStream_t st) {
  launch(k_tile2d_fwd<T, TX, TY, NT>, dim3((g.n[0] + TX - 1) / TX, (g.n[1] + TY - 1) / TY), NT, 0, st, g, S, ctrl, di);
}
template <typename T, int TX, int TY, int NT>
void adj_shape(const Geo& g, const Slots<T>& S, T* Lb, long long lstride, const Ctrl* ctrl, int di, cudaStream_t st) {
  launch(k_tile2d_adj<T, TX, TY, NT>, dim3((g.n[0] + TX - 1) / TX, (g.n[1] + TY - 1) / TY), NT, 0, st, g, S, Lb,
         lstride, ctrl, di);
}

}  // namespace

// Tiles pay while the strips of the other form are short: a strip of L rows works on L + 4. FP64
// (instruction count decides): the predictor below 4 rows, the transpose, whose strips do more per row, below
// 12. Strips -> tiles, predictor / transpose in us: 80x40 25 / 42 -> 7 / 7; 600x100 24 / 42 -> 17 / 19; 1024x512
// 149 / 258 -> 102 / 101; 2600x1300 712 / 1168 -> 623 / 603; 3000x1500 (3 rows) 840 / 1315 -> 827 / 795; 3300x1700
// (4) 969 / 1497 -> 1030 / 994; 4096x2048 (7) 1305 / 1915 -> 1524 / 1468; 5000x2500 (10) 1799 / 2547 -> 2281 / 2193.
// FP32 (the tile's loads cost more): only where strips have two or three rows,
// and the predictor, whose chain is shorter, only on the smallest grids: 512x256 7 / 11 -> 6 / 7,
// 1024x512 12.4 / 18 -> 13 / 13.5, 2048x1024 21 / 32 -> 40 / 44 us. (Events around each launch, less
// their 3.5 us.)
bool stencil_tile_pays(const Geo& g, int rows, bool fp64, bool transpose) {
  if (fp64) return rows < (transpose ? 12 : 4);
  return rows < 4 && g.N <= (transpose ? 1LL << 20 : 1LL << 18);
}

template <typename T>
void launch_stencil_tile_fwd(const Geo& g, const Slots<T>& S, const Ctrl* ctrl, int di, cudaStream_t st) {
  const bool small = g.N <= 152 * 4 * 64;  // a CTA of 8 x 8 cells per scheduler or fewer
  if (small)
    fwd_shape<T, 8, 8, 128>(g, S, ctrl, di, st);
  else
    fwd_shape<T, 32, 8, 352>(g, S, ctrl, di, st);
}
template <typename T>
void launch_stencil_tile_adj(const Geo& g, const Slots<T>& S, T* Lb, long long lstride, const Ctrl* ctrl, int di,
                             cudaStream_t st) {
  const bool small = g.N <= 152 * 4 * 64;
  if (small)
    adj_shape<T, 8, 8, 128>(g, S, Lb, lstride, ctrl, di, st);
  else
    adj_shape<T, 32, 8, 352>(g, S, Lb, lstride, ctrl, di, st);
}

#define LKS_TILE_INST(T)                                                                                     \
  template void launch_stencil_tile_fwd<T>(const Geo&, const Slots<T>&, const Ctrl*, int, cudaStream_t);     \
  template void launch_stencil_tile_adj<T>(const Geo&, const Slots<T>&, T*, long long, const Ctrl*, int, cudaStream_t);
LKS_TILE_INST(float)
LKS_TILE_INST(double)

}  // namespace lks
