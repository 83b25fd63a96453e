// Reverse of a coupling iteration of a freely rotating body in FP32 with the cosine kernel, on tiles of
// 8 x 8 x 8 cells: the cell phase (adj_cell_work of lks_body.cu) and the design-point phase
// (adj_design_point there, which FP64 and the bilinear kernel take).
//
// A cell's gather takes the 64 or so design points within the support of it. Found from the cell (the
// support cube pulled back to the design frame, its rows clipped to the cube: gather_free_lanes in
// lks_device.cuh) they lie in about 37 rows of one or two points each, so most instructions went into
// rows. Here a CTA first sorts the design points of its tile's reach (11^3 cells) by the cell that
// holds them: a thread takes a row of the design grid, clips it to the tile's reach and puts its points
// into bins; the bins' starts follow from a scan, and the points of a bin are ordered by their index,
// so that sums do not depend on the order the bins were filled in. A cell then visits the 16 runs of
// four bins along x around it. A point's weights at the four cells of its window are (1 -+ sin)/4 and
// (1 +- cos)/4 of one angle per axis, which are stored with it: a pair costs three shared loads and about
// twenty instructions. 256x128x128 body of 96^3 (ball), per iteration on GB300: cell phase 205 -> 106 us,
// design-point phase 230 -> 131 us.
//
// The forward keeps the per-cell gather (k_couple): the tiled one took 135 us against 257, but its other
// rounding moves values of reduced-precision snapshots across a rounding step of 1/512, and with that
// single gradient entries by up to 8e-4 of their rms (BF16, 12 steps), where no more than that is wanted.
#include <algorithm>
#include <climits>

#include "lks_body_common.cuh"
#include "lks_free.cuh"

namespace lks {

namespace {

constexpr int TE = kFreeTile;      // tile edge in cells
constexpr int BE = TE + 3;         // bins per axis: a cell's window holds points of four cells
constexpr int NB = BE * BE * BE;
constexpr int NT = TE * TE * TE;   // threads: one per cell
// Design points in a cube of edge 11: each lies in a unit cube of its own within the cube grown by
// the unit cube's half diagonal, at most (11 + sqrt 3)^3 = 2064.
constexpr int CAP = 2080;

struct Smem {
  float4 a[CAP];   // cos, sin along x; cos, sin along y   (of pi/2 times the fraction)
  float4 b[CAP];   // cos, sin along z; kappa; lever x
  float2 c[CAP];   // lever y, z
  int point[CAP];             // design points in the order they were found
  int fill[NB];
  unsigned short order[CAP];  // their places in that list, by bin
  unsigned short bin[CAP];    // their bins
  unsigned short start[NB + 1];
  unsigned char bx[CAP];      // bin's x of the sorted points
  int total, sums[NT / 32];
};

static_assert(sizeof(Smem) + 2048 <= 113 * 1024, "two CTAs per SM");

// Tile of this CTA: first cell (unwrapped coordinates), this thread's cell in the box.
struct FreeCell {
  int x0[3], j[3];
  bool in;  // inside the box
};
__device__ __forceinline__ FreeCell free_cell(const Geo& g, const int (&lo)[3]) {
  FreeCell c;
  const int t = threadIdx.x;
  const int e[3] = {t % TE, (t / TE) % TE, t / (TE * TE)};
  const int bid[3] = {(int)blockIdx.x, (int)blockIdx.y, (int)blockIdx.z};
  c.in = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    c.j[a] = bid[a] * TE + e[a];
    c.x0[a] = lo[a] + bid[a] * TE;
    c.in = c.in && c.j[a] < g.B[a];
  }
  return c;
}

// x^ref - floor(x^G) of a design point along axis a: one fixed sequence of roundings, so that the cell
// found for a point and its fraction there always belong together. The part without x of the row:
__device__ __forceinline__ float row_part(const float (&R)[9], int a, float ry, float rz) {
  return fmaf(R[3 * a + 1], ry, __fmul_rn(R[3 * a + 2], rz));
}
__device__ __forceinline__ float place(const float (&R)[9], int a, float rx, float xf, float part) {
  return fmaf(R[3 * a], rx, __fadd_rn(xf, part));
}

// Sorts the design points of the tile's reach into s. Returns their number (0: no cell of the tile is
// reached). All threads of the block call it.
__device__ __forceinline__ int sort_points(const Geo& g, const float* __restrict__ kref, const Dof& sk, const int (&x0)[3],
                                           Smem& s) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float R[9], xf[3];
  int off[3];  // bin coordinate of floor(x^G) (bin 0 is cell x0 - 2)
#pragma unroll
  for (int i = 0; i < 9; ++i) R[i] = sk.Rf[i];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    xf[a] = sk.xf[a];
    off[a] = sk.xi[a] - x0[a] + 2;
  }
  for (int q = tid; q < NB; q += NT) s.fill[q] = 0;
  if (tid == 0) s.total = 0;
  // design box of the reach: bin coordinates in [0, 11)^3, widened by the rounding of positions
  const float half = 0.5f * BE + 2e-3f, pad = 1e-3f, tiny = 1e-6f;
  float ctr[3], xi[3];
  int lo[3], hi[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) ctr[a] = 0.5f * BE - (float)off[a] - xf[a];  // centre - x^G
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    xi[d] = R[d] * ctr[0] + R[3 + d] * ctr[1] + R[6 + d] * ctr[2] + g.xicf[d];
    const float h = half * (fabsf(R[d]) + fabsf(R[3 + d]) + fabsf(R[6 + d])) + pad;
    lo[d] = max(0, (int)ceilf(xi[d] - h));
    hi[d] = min(g.nd[d] - 1, (int)floorf(xi[d] + h));
  }
  const int nyr = hi[1] - lo[1] + 1, nzr = hi[2] - lo[2] + 1;
  if (hi[0] < lo[0] || nyr <= 0 || nzr <= 0) return 0;  // (uniform)
  __syncthreads();
  for (int q = tid; q < nyr * nzr; q += NT) {
    const int iy = lo[1] + q % nyr, iz = lo[2] + q / nyr;
    const int qyz = dsq(iy, g.nd[1]) + dsq(iz, g.nd[2]);
    if (qyz > g.rad4) continue;
    const float ey = (float)iy - xi[1], ez = (float)iz - xi[2];
    float e0 = -1e6f, e1 = 1e6f;
    bool empty = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float cw = R[3 * a + 1] * ey + R[3 * a + 2] * ez, r = R[3 * a];
      if (fabsf(r) > tiny) {
        const float inv = 1.0f / r, p0 = (-half - cw) * inv, p1 = (half - cw) * inv;
        e0 = fmaxf(e0, fminf(p0, p1));
        e1 = fminf(e1, fmaxf(p0, p1));
      } else if (fabsf(cw) >= half) {
        empty = true;
      }
    }
    if (empty) continue;
    const int j0 = max(lo[0], (int)ceilf(xi[0] + e0 - pad)), j1 = min(hi[0], (int)floorf(xi[0] + e1 + pad));
    const float ry = (float)iy - g.xicf[1], rz = (float)iz - g.xicf[2];
    const float part[3] = {row_part(R, 0, ry, rz), row_part(R, 1, ry, rz), row_part(R, 2, ry, rz)};
    for (int ix = j0; ix <= j1; ++ix) {
      if (qyz + dsq(ix, g.nd[0]) > g.rad4) continue;
      const float rx = (float)ix - g.xicf[0];
      const int f0 = (int)floorf(place(R, 0, rx, xf[0], part[0])) + off[0];
      const int f1 = (int)floorf(place(R, 1, rx, xf[1], part[1])) + off[1];
      const int f2 = (int)floorf(place(R, 2, rx, xf[2], part[2])) + off[2];
      if ((unsigned)f0 >= (unsigned)BE || (unsigned)f1 >= (unsigned)BE || (unsigned)f2 >= (unsigned)BE) continue;
      const int bin = (f2 * BE + f1) * BE + f0, at = atomicAdd(&s.total, 1);
      if (at < CAP) {
        atomicAdd(&s.fill[bin], 1);
        s.point[at] = ix + g.nd[0] * (iy + g.nd[1] * iz);
        s.bin[at] = (unsigned short)bin;
      }
    }
  }
  __syncthreads();
  const int n = min(s.total, CAP);
  if (n == 0) return 0;
  // starts: exclusive scan of the bins' counts, three bins a thread
  constexpr int PER = (NB + NT - 1) / NT;
  int cnt[PER], sum = 0;
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const int bin = tid * PER + q;
    cnt[q] = bin < NB ? s.fill[bin] : 0;
    sum += cnt[q];
  }
  int inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += v;
  }
  if (lane == 31) s.sums[warp] = inc;
  __syncthreads();
  int base = inc - sum;
  for (int w = 0; w < warp; ++w) base += s.sums[w];
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const int bin = tid * PER + q;
    if (bin < NB) {
      s.start[bin] = (unsigned short)base;
      s.fill[bin] = base;
    }
    base += cnt[q];
  }
  if (tid == 0) s.start[NB] = (unsigned short)n;
  __syncthreads();
  for (int q = tid; q < n; q += NT) s.order[atomicAdd(&s.fill[s.bin[q]], 1)] = (unsigned short)q;
  __syncthreads();
  for (int q = tid; q < n; q += NT) {  // each point to its place by index within its bin
    const int m = s.point[q], bin = s.bin[q], s0 = s.start[bin], s1 = s.start[bin + 1];
    int at = s0;
    for (int p = s0; p < s1; ++p) at += s.point[s.order[p]] < m;
    const int iz = m / (g.nd[0] * g.nd[1]), r = m - iz * g.nd[0] * g.nd[1], iy = r / g.nd[0], ix = r - iy * g.nd[0];
    const float rx = (float)ix - g.xicf[0], ry = (float)iy - g.xicf[1], rz = (float)iz - g.xicf[2];
    float l[3], c[3], sn[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float part = row_part(R, a, ry, rz), p = place(R, a, rx, xf[a], part), fr = p - floorf(p);
      l[a] = fmaf(R[3 * a], rx, part);
      c[a] = __cosf(1.57079632679f * fr);
      sn[a] = __sinf(1.57079632679f * fr);
    }
    s.a[at] = make_float4(c[0], sn[0], c[1], sn[1]);
    s.b[at] = make_float4(c[2], sn[2], __ldg(kref + m), l[0]);
    s.c[at] = make_float2(l[1], l[2]);
    s.bx[at] = (unsigned char)(bin % BE);
  }
  __syncthreads();
  return n;
}

// Sums over the sorted points for this thread's cell: phi, kappa, P = sum W l, L = sum W kappa l (world
// levers l = R r).
struct FreeSums {
  float phi, kap, P[3], L[3];
};
__device__ __forceinline__ void free_sums(const Smem& s, FreeSums& o) {
  const int t = threadIdx.x, cx = t % TE, cy = (t / TE) % TE, cz = t / (TE * TE);
  o.phi = o.kap = 0.0f;
#pragma unroll
  for (int a = 0; a < 3; ++a) o.P[a] = o.L[a] = 0.0f;
#pragma unroll 1
  for (int jz = 0; jz < 4; ++jz) {
#pragma unroll
    for (int jy = 0; jy < 4; ++jy) {
      // window place 3 - j along the axis: weight (1 - c)/4, (1 + s)/4, (1 + c)/4, (1 - s)/4 for j = 0..3
      const int row = ((cz + jz) * BE + cy + jy) * BE + cx;
      const int e = s.start[row + 4];
      for (int i = s.start[row]; i < e; ++i) {
        const float4 A = s.a[i], B = s.b[i];
        const float2 C = s.c[i];
        const int jx = s.bx[i] - cx;
        const float tx = (jx & 1) ? A.y : A.x, ty = (jy & 1) ? A.w : A.z, tz = (jz & 1) ? B.y : B.x;
        const float wx = (jx == 0 || jx == 3) ? 1.0f - tx : 1.0f + tx;
        const float wy = (jy == 0 || jy == 3) ? 1.0f - ty : 1.0f + ty;
        const float wz = (jz == 0 || jz == 3) ? 1.0f - tz : 1.0f + tz;
        const float W = wx * wy * wz, K = W * B.z;
        o.phi += W;
        o.kap += K;
        o.P[0] = fmaf(W, B.w, o.P[0]);
        o.P[1] = fmaf(W, C.x, o.P[1]);
        o.P[2] = fmaf(W, C.y, o.P[2]);
        o.L[0] = fmaf(K, B.w, o.L[0]);
        o.L[1] = fmaf(K, C.x, o.L[1]);
        o.L[2] = fmaf(K, C.y, o.L[2]);
      }
    }
  }
  constexpr float f = 1.0f / 64.0f;
  o.phi *= f;
  o.kap *= f;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    o.P[a] *= f;
    o.L[a] *= f;
  }
}

// Cell phase of the reverse of iteration k (adj_cell_work).
__global__ void __launch_bounds__(NT, 2) k_adj_cell_free(Geo g, const Ctrl* ctrl, const Dof* it,
                                                         const float* __restrict__ kref,
                                                         const float* __restrict__ boxstore, int nbox, float* Lb,
                                                         long long lstride, float* __restrict__ acc,
                                                         float* __restrict__ scratch, int k, int di) {
  extern __shared__ __align__(16) unsigned char raw[];
  Smem& s = *reinterpret_cast<Smem*>(raw);
  const int t = ctrl->t0 - di, base = ctrl->base, K = g.K;
  const Dof* row = it + (long long)(t - 1) * (K + 1);
  const Dof& sk = row[k - 1];
  int lo[3];
  box_origin<3>(g, row[0], lo[0], lo[1], lo[2]);
  const FreeCell cc = free_cell(g, lo);
  const int n = sort_points(g, kref, sk, cc.x0, s);
  if (!cc.in) return;
  const long long N = g.N, BC = g.box_cells;
  const long long bl = cc.j[0] + (long long)g.B[0] * (cc.j[1] + (long long)g.B[1] * cc.j[2]);
  long long m = 0;
  if (!cell_index<3>(g, lo[0] + cc.j[0], lo[1] + cc.j[1], lo[2] + cc.j[2], m)) {
#pragma unroll
    for (int q = 0; q < 7; ++q) scratch[q * BC + bl] = 0.0f;
    return;
  }
  FreeSums A;
  A.phi = A.kap = 0.0f;
#pragma unroll
  for (int a = 0; a < 3; ++a) A.P[a] = A.L[a] = 0.0f;
  if (n > 0) free_sums(s, A);
  float* Lcur = Lb + (long long)(t & 1) * lstride;
  const float* bs = boxstore + (long long)((t - base - 1) % nbox) * BC * 3;
  const float lT[3] = {ctrl->lam_Tf[0], ctrl->lam_Tf[1], ctrl->lam_Tf[2]};
  const float om[3] = {sk.omf[0], sk.omf[1], sk.omf[2]};
  float rv[3], extra[3];
  cross3(om, A.P, rv);
  cross3(lT, A.L, extra);
  const float inv = 1.0f / (1.0f + A.kap);
  float lkap = 0.0f;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float us = sk.ug[a] * A.phi + rv[a];
    const float uk = (bs[a * BC + bl] + A.kap * us) * inv;
    float lu = A.kap * ctrl->lam_Ff[a] + extra[a];
    if (k == K) lu += Lcur[(a + 1) * N + m];
    const float accv = (k == K ? 0.0f : acc[a * BC + bl]) + lu * inv;
    if (k == 1)
      Lcur[(a + 1) * N + m] = accv;
    else
      acc[a * BC + bl] = accv;
    lkap += lu * (us - uk) * inv;
    scratch[a * BC + bl] = uk;
    scratch[(4 + a) * BC + bl] = lu * A.kap * inv;
  }
  scratch[3 * BC + bl] = lkap;
}

// Design-point phase of the reverse of iteration k (adj_design_point): a CTA takes tiles of 8^3 cells
// in turn, brings the seven scratch values of the tile and its window's halo to shared memory as one
// 32-byte record a cell, lists the design points that lie in the tile's cells, and gives each to one
// thread. Reading the windows through L1 (64 cells by seven scattered loads a point) bound the form
// with four lanes a point: 230 us an iteration on the 96^3 ball. The window is summed by rows along x:
// the row's sums of the seven values and of the combination q that multiplies the weights' derivatives,
// then the row's y and z weights.
constexpr int DT = 256;      // threads
constexpr int DCAP = 928;    // design points in the tile: at most (8 + sqrt 3)^3 = 922
struct DesignSmem {
  float4 f[2 * NB];  // u x, y, z, dJ/dkappa_n; dJ/du^S x, y, z, -
  int point[DCAP];
  int sums[DT / 32];
};
__global__ void __launch_bounds__(DT, 2) k_adj_design_free(Geo g, Ctrl* ctrl, const Dof* it,
                                                           const float* __restrict__ kref,
                                                           const float* __restrict__ scratch,
                                                           double* __restrict__ dkref, float2* partials, int k, int di) {
  constexpr int NV = 18;
  extern __shared__ __align__(16) unsigned char raw[];
  DesignSmem& s = *reinterpret_cast<DesignSmem*>(raw);
  __shared__ double red[32 * NV];
  const int t = ctrl->t0 - di, K = g.K, tid = threadIdx.x;
  const Dof* row = it + (long long)(t - 1) * (K + 1);
  const Dof& sk = row[k - 1];
  int lo[3];
  box_origin<3>(g, row[0], lo[0], lo[1], lo[2]);
  float R[9], xf[3], om[3], ug[3], lF[3], lT[3];
  int xi[3];
#pragma unroll
  for (int i = 0; i < 9; ++i) R[i] = sk.Rf[i];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    xf[a] = sk.xf[a];
    xi[a] = sk.xi[a];
    om[a] = sk.omf[a];
    ug[a] = sk.ug[a];
    lF[a] = ctrl->lam_Ff[a];
    lT[a] = ctrl->lam_Tf[a];
  }
  float v[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) v[i] = 0.0f;
  const long long BC = g.box_cells;
  const int n0 = (g.B[0] + TE - 1) / TE, n1 = (g.B[1] + TE - 1) / TE, n2 = (g.B[2] + TE - 1) / TE;
  for (int tile = blockIdx.x; tile < n0 * n1 * n2; tile += gridDim.x) {
    const int org[3] = {(tile % n0) * TE, (tile / n0 % n1) * TE, tile / (n0 * n1) * TE};  // in the box
    __syncthreads();
    // the design points whose cell lies in the tile, found as in sort_points
    const float half = 0.5f * TE + 2e-3f, pad = 1e-3f, tiny = 1e-6f;
    int off[3], dlo[3], dhi[3];
    float ctr[3], xd[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      off[a] = xi[a] - lo[a] - org[a];  // tile coordinate of floor(x^G)
      ctr[a] = 0.5f * TE - (float)off[a] - xf[a];
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      xd[d] = R[d] * ctr[0] + R[3 + d] * ctr[1] + R[6 + d] * ctr[2] + g.xicf[d];
      const float h = half * (fabsf(R[d]) + fabsf(R[3 + d]) + fabsf(R[6 + d])) + pad;
      dlo[d] = max(0, (int)ceilf(xd[d] - h));
      dhi[d] = min(g.nd[d] - 1, (int)floorf(xd[d] + h));
    }
    const int nyr = dhi[1] - dlo[1] + 1, nzr = dhi[2] - dlo[2] + 1;
    if (dhi[0] < dlo[0] || nyr <= 0 || nzr <= 0) continue;  // (uniform)
    // a thread marks its row's points, a scan over the rows places them: a fixed order, on which the
    // threads' sums depend
    int n = 0;
    for (int q0 = 0; q0 < nyr * nzr; q0 += DT) {
      const int q = q0 + tid, iy = dlo[1] + q % nyr, iz = dlo[2] + q / nyr;
      const int qyz = dsq(iy, g.nd[1]) + dsq(iz, g.nd[2]);
      const float ey = (float)iy - xd[1], ez = (float)iz - xd[2];
      float e0 = -1e6f, e1 = 1e6f;
      bool empty = q >= nyr * nzr || qyz > g.rad4;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const float cw = R[3 * a + 1] * ey + R[3 * a + 2] * ez, r = R[3 * a];
        if (fabsf(r) > tiny) {
          const float inv = 1.0f / r, p0 = (-half - cw) * inv, p1 = (half - cw) * inv;
          e0 = fmaxf(e0, fminf(p0, p1));
          e1 = fminf(e1, fmaxf(p0, p1));
        } else if (fabsf(cw) >= half) {
          empty = true;
        }
      }
      unsigned mask = 0;  // a row's points in the tile's cube: at most 8 sqrt 3 + 1 of them
      int j0 = 0;
      if (!empty) {
        j0 = max(dlo[0], (int)ceilf(xd[0] + e0 - pad));
        const int j1 = min(min(dhi[0], (int)floorf(xd[0] + e1 + pad)), j0 + 31);
        const float ry = (float)iy - g.xicf[1], rz = (float)iz - g.xicf[2];
        const float part[3] = {row_part(R, 0, ry, rz), row_part(R, 1, ry, rz), row_part(R, 2, ry, rz)};
        for (int ix = j0; ix <= j1; ++ix) {
          const float rx = (float)ix - g.xicf[0];
          bool in = qyz + dsq(ix, g.nd[0]) <= g.rad4;
#pragma unroll
          for (int a = 0; a < 3; ++a)
            in = in && (unsigned)((int)floorf(place(R, a, rx, xf[a], part[a])) + off[a]) < (unsigned)TE;
          if (in) mask |= 1u << (ix - j0);
        }
      }
      const int cnt = __popc(mask), lane = tid & 31, warp = tid >> 5;
      int inc = cnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += x;
      }
      if (lane == 31) s.sums[warp] = inc;
      __syncthreads();
      int at = n + inc - cnt;
#pragma unroll
      for (int w = 0; w < DT / 32; ++w) {
        if (w < warp) at += s.sums[w];
        n += s.sums[w];
      }
      const int m0 = j0 + g.nd[0] * (iy + g.nd[1] * iz);
      for (; mask; mask &= mask - 1, ++at)
        if (at < DCAP) s.point[at] = m0 + __ffs(mask) - 1;
      __syncthreads();
    }
    n = min(n, DCAP);
    if (n == 0) continue;  // (uniform)
    // the cells of the tile and its halo (one below, two above); off the box: zeros
    for (int q = tid; q < NB; q += DT) {
      const int j[3] = {org[0] - 1 + q % BE, org[1] - 1 + q / BE % BE, org[2] - 1 + q / (BE * BE)};
      float x[7] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
      if (j[0] >= 0 && j[0] < g.B[0] && j[1] >= 0 && j[1] < g.B[1] && j[2] >= 0 && j[2] < g.B[2]) {
        const long long bl = j[0] + (long long)g.B[0] * (j[1] + (long long)g.B[1] * j[2]);
#pragma unroll
        for (int c = 0; c < 7; ++c) x[c] = __ldg(scratch + c * BC + bl);
      }
      s.f[2 * q] = make_float4(x[0], x[1], x[2], x[3]);
      s.f[2 * q + 1] = make_float4(x[4], x[5], x[6], 0.0f);
    }
    __syncthreads();
    for (int q = tid; q < n; q += DT) {
      const int m = s.point[q];
      const int iz = m / (g.nd[0] * g.nd[1]), rm = m - iz * g.nd[0] * g.nd[1], iy = rm / g.nd[0], ix = rm - iy * g.nd[0];
      const float r[3] = {(float)ix - g.xicf[0], (float)iy - g.xicf[1], (float)iz - g.xicf[2]};
      const float km = __ldg(kref + m);
      float l[3], w[3][4], dw[3][4], oxl[3], rotl[3], usr[3], luref[3];
      int f[3];
      bool outside = false;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const float part = row_part(R, a, r[1], r[2]), p = place(R, a, r[0], xf[a], part), fl = floorf(p), fr = p - fl;
        l[a] = fmaf(R[3 * a], r[0], part);
        f[a] = (int)fl + off[a];  // tile coordinate of the point's cell, 0 .. 7: window f .. f + 3 of the halo
        const float c = __cosf(1.57079632679f * fr), sn = __sinf(1.57079632679f * fr);
        w[a][0] = 0.25f * (1.0f - sn);
        w[a][1] = 0.25f * (1.0f + c);
        w[a][2] = 0.25f * (1.0f + sn);
        w[a][3] = 0.25f * (1.0f - c);
        const float h = 0.392699081699f;  // w' = -pi/8 sin(pi/2 (q - 1 - fr))
        dw[a][0] = h * c;
        dw[a][1] = h * sn;
        dw[a][2] = -h * c;
        dw[a][3] = -h * sn;
        const int b0 = org[a] + f[a] - 1;
        outside = outside || b0 < 0 || b0 + 3 - (fr == 0.0f) >= g.B[a];
      }
      if (outside) atomicOr(&ctrl->status, ST_BOX_OVERFLOW);
      cross3(om, l, oxl);
      cross3(lT, l, rotl);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        usr[a] = ug[a] + oxl[a];
        luref[a] = km * (lF[a] + rotl[a]);
      }
      float uref[3] = {0.0f, 0.0f, 0.0f}, slus[3] = {0.0f, 0.0f, 0.0f}, slk = 0.0f, lxr[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll 1
      for (int qz = 0; qz < 4; ++qz) {
        const float wz = qz == 0 ? w[2][0] : qz == 1 ? w[2][1] : qz == 2 ? w[2][2] : w[2][3];
        const float dz = qz == 0 ? dw[2][0] : qz == 1 ? dw[2][1] : qz == 2 ? dw[2][2] : dw[2][3];
#pragma unroll
        for (int qy = 0; qy < 4; ++qy) {
          const float4* F = s.f + 2 * (((f[2] + qz) * BE + f[1] + qy) * BE + f[0]);
          float S[7] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f}, D = 0.0f;
#pragma unroll
          for (int qx = 0; qx < 4; ++qx) {
            const float4 A = F[2 * qx], B = F[2 * qx + 1];
            const float x[7] = {A.x, A.y, A.z, A.w, B.x, B.y, B.z};
            const float wx = w[0][qx];
#pragma unroll
            for (int c = 0; c < 7; ++c) S[c] = fmaf(wx, x[c], S[c]);
            const float qv = km * x[3] + luref[0] * x[0] + luref[1] * x[1] + luref[2] * x[2] + usr[0] * x[4] +
                             usr[1] * x[5] + usr[2] * x[6];
            D = fmaf(dw[0][qx], qv, D);
          }
          const float Q = km * S[3] + luref[0] * S[0] + luref[1] * S[1] + luref[2] * S[2] + usr[0] * S[4] +
                          usr[1] * S[5] + usr[2] * S[6];
          const float wyz = w[1][qy] * wz;
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            uref[a] = fmaf(wyz, S[a], uref[a]);
            slus[a] = fmaf(wyz, S[4 + a], slus[a]);
          }
          slk = fmaf(wyz, S[3], slk);
          // dW/dx^ref_e = -w'(x_e - x^ref_e) prod_{a != e} w
          lxr[0] = fmaf(-wyz, D, lxr[0]);
          lxr[1] = fmaf(-dw[1][qy] * wz, Q, lxr[1]);
          lxr[2] = fmaf(-w[1][qy] * dz, Q, lxr[2]);
        }
      }
      float Dl[3], lxD[3], DxT[3], lusr[3], lxu[3], uxo[3], dk = slk;
#pragma unroll
      for (int a = 0; a < 3; ++a) Dl[a] = uref[a] - usr[a];
      cross3(l, Dl, lxD);
      cross3(Dl, lT, DxT);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        dk += lF[a] * Dl[a] + lT[a] * lxD[a];
        lusr[a] = -luref[a] + slus[a];
      }
      dkref[m] += (double)dk;
      cross3(l, lusr, lxu);
      cross3(lusr, om, uxo);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        v[i] += lxr[i];
        v[3 + i] += lusr[i];
        v[6 + i] += lxu[i];
        const float gl = lxr[i] + km * DxT[i] + uxo[i];  // dJ/d(R r_m)
#pragma unroll
        for (int j = 0; j < 3; ++j) v[9 + 3 * i + j] += gl * r[j];
      }
    }
  }
  __syncthreads();
  block_sum_partial<NV, 1>(v, partials + blockIdx.x * NV, red);
}

dim3 free_grid(const Geo& g) {
  return dim3((g.B[0] + TE - 1) / TE, (g.B[1] + TE - 1) / TE, (g.B[2] + TE - 1) / TE);
}

}  // namespace

bool prepare_free3d() {
  const int bytes = (int)sizeof(Smem);
  return cudaFuncSetAttribute(k_adj_cell_free, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess &&
         cudaFuncSetAttribute(k_adj_design_free, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)sizeof(DesignSmem)) == cudaSuccess;
}

int free_tiles(const Geo& g) {
  const dim3 n = free_grid(g);
  return (int)(n.x * n.y * n.z);
}

// Where the tiles pay. Few tiles leave the chip idle for the whole of a tile's sort and sums (about 22 us for
// the cell phase), and a box-shaped body leaves the corners of its box, a tile each, without design points.
// GB300, us per iteration, per point or cell -> tiles:
//   cell phase        ball, box of 40^3 cells 21.8 -> 22.7, 44^3 25.0 -> 22.9, 52^3 37.4 -> 30.5;
//                     solid, 42^3 18.8 -> 22.7, 48^3 21.5 -> 21.3, 56^3 29.5 -> 22.8, 90^3 97.8 -> 49.4
//   design points     ball, 36^3 46.6 -> 47.3, 40^3 53.9 -> 46.3, 52^3 70.6 -> 57.1;
//                     solid, 56^3 46.7 -> 49.6, 90^3 75.3 -> 79.7, 104^3 95.4 -> 80.2
bool free_cell_pays(const Geo& g) { return g.box_cells >= 80000; }
bool free_design_pays(const Geo& g) { return g.box_cells >= (g.rad4 != INT_MAX ? 55000 : 1000000); }

int free_design_ctas(const Geo& g) { return std::min(free_tiles(g), kFreeDesignCtas); }

void launch_adj_cell_free(const Geo& g, const Ctrl* ctrl, const Dof* it, const float* kref, const float* boxstore, int nbox,
                          float* Lb, long long lstride, float* acc, float* scratch, int k, int di, cudaStream_t st) {
  launch(k_adj_cell_free, free_grid(g), NT, sizeof(Smem), st, g, ctrl, it, kref, boxstore, nbox, Lb, lstride, acc, scratch,
         k, di);
}
void launch_adj_design_free(const Geo& g, Ctrl* ctrl, const Dof* it, const float* kref, const float* scratch, double* dkref,
                            void* partials, int k, int di, cudaStream_t st) {
  launch(k_adj_design_free, free_design_ctas(g), DT, sizeof(DesignSmem), st, g, ctrl, it, kref, scratch, dkref,
         (float2*)partials, k, di);
}

}  // namespace lks
