// 3D body kernels for one rotation axis that treat a column of cells along the axis together.
//
// About one axis a cell and a design point meet through an in-plane weight w_b w_c and an axial one.
// The in-plane part (which columns of design points reach a column of cells, their weights and levers)
// is the same for every plane, and the axial weights are the same four numbers for every cell, since
// design points and cells are both one apart. So a lane takes one in-plane position and ZC
// consecutive planes: it finds the reaching design columns once (a list in shared memory), and per
// column loads ZC + 3 values of kappa, forms ZC axial sums from them and adds those to the planes'
// sums. A cell's gather of 64 pairs costs it about 16 (1 load, 7 multiply-adds), where the form with
// one cell per four lanes (lks_device.cuh) ran every candidate test and weight again for every plane.
// Loads are issued one design column ahead (the kernels wait on L2 otherwise: a quarter of their time).
// Measured on GB300, FP32, per step of the 128x64x64 / 48^3 body: coupling 250 -> 73 us (five iterations),
// recompute 27 -> 11, reverse sums 107 -> 73, dJ/dkappa^ref 95 -> 43 (against one cell per four lanes and
// one design point per four lanes).
//
//   k_couple_axis3d  the N_itr coupling iterations of a step, sums and iterate exchanged through
//                    flagged words (lks_flag.cuh), one cooperative launch
//   k_apply_axis3d   recompute of a step's Brinkman update
//   k_coef_axis3d    the sums of the reverse by linear maps (k_rev_coef of lks_reverse.cu)
//   k_design_axis3d  its dJ/dkappa^ref: a lane takes one column of design points and ZD of them
#include <climits>
#include <type_traits>

#include "lks_flag.cuh"
#include "lks_reverse.cuh"

namespace lks {

namespace {

constexpr int kListMax = 30;  // lattice points in an open square of side 4: at most (4 + sqrt 2)^2 = 29.3
constexpr int kPadPts = 3;    // taps beyond the first of the axial window

// Planes per lane.
template <typename T>
struct Planes {
  static constexpr int ZC = sizeof(T) == 4 ? 8 : 4;  // forward sums: 3 (6 with a ball) per plane
  static constexpr int ZR = sizeof(T) == 4 ? 4 : 2;  // reverse sums: 14 per plane
};

// Box units: 32 in-plane positions (a warp's lanes) by Z planes. The in-plane axis that is x runs fastest.
template <int AX>
struct InPlane {
  static constexpr int B = Axes<AX>::B, C = Axes<AX>::C, A = Axes<AX>::A;
  static constexpr bool b_fast = C != 0;
};
template <int AX>
__host__ __device__ inline int plane_tiles(const Geo& g) {
  return (g.B[InPlane<AX>::B] * g.B[InPlane<AX>::C] + 31) / 32;
}
template <int AX>
__host__ __device__ inline long long plane_units(const Geo& g, int Z) {
  return (long long)plane_tiles<AX>(g) * ((g.B[InPlane<AX>::A] + Z - 1) / Z);
}

// A lane's in-plane position in the box (jb, jc) and its first plane ja.
struct LanePos {
  int j[3];
  bool ok;  // inside the box in the plane
};
template <int AX>
__device__ __forceinline__ LanePos lane_pos(const Geo& g, int unit, int tiles, int Z, int lane) {
  using P = InPlane<AX>;
  LanePos p;
  const int tile = unit % tiles, q = tile * 32 + lane;
  const int fast = g.B[P::b_fast ? P::B : P::C];
  const int r = q / fast, f = q - r * fast;
  p.j[P::B] = P::b_fast ? f : r;
  p.j[P::C] = P::b_fast ? r : f;
  p.j[P::A] = (unit / tiles) * Z;
  p.ok = r < g.B[P::b_fast ? P::C : P::B];
  return p;
}

// List of the design columns (ib, ic) whose in-plane offset from the cell at d lies within the
// support, packed in 16 bits each, into list[0 .. count)[lane]. Bounds in FP32 (widened), test in T.
template <typename T, int AX>
__device__ __forceinline__ int column_list(const Geo& g, const T (&d)[3], T cs, T sn, bool active,
                                           unsigned (*list)[32], int lane) {
  constexpr int b = Axes<AX>::B, c = Axes<AX>::C;
  const T S = (T)g.s;
  const T xib = dot2(cs, d[b], sn, d[c]) + pivot<T>(g, b), xic = dot2(cs, d[c], -sn, d[b]) + pivot<T>(g, c);
  const float csf = (float)cs, snf = (float)sn, pad = 2e-3f, Sp = (float)g.s + pad;
  const float xibf = (float)xib, xicf = (float)xic, h = Sp * (fabsf(csf) + fabsf(snf)) + pad;
  const int ib0 = max(0, (int)ceilf(xibf - h)), ib1 = active ? min(g.nd[b] - 1, (int)floorf(xibf + h)) : -1;
  const int ic0 = max(0, (int)ceilf(xicf - h)), ic1 = min(g.nd[c] - 1, (int)floorf(xicf + h));
  const float tiny = 1e-6f;
  const float ics = fabsf(csf) > tiny ? 1.0f / csf : 0.0f, isn = fabsf(snf) > tiny ? 1.0f / snf : 0.0f;
  int n = 0;
  if (ib0 > ib1) return 0;
  for (int ic = ic0; ic <= ic1; ++ic) {
    const float ecf = (float)ic - xicf;
    float lo = -1e6f, hi = 1e6f;
    if (ics != 0.0f) {
      const float e1 = (snf * ecf - Sp) * ics, e2 = (snf * ecf + Sp) * ics;
      lo = fmaxf(lo, fminf(e1, e2));
      hi = fminf(hi, fmaxf(e1, e2));
    }
    if (isn != 0.0f) {
      const float e1 = (-Sp - csf * ecf) * isn, e2 = (Sp - csf * ecf) * isn;
      lo = fmaxf(lo, fminf(e1, e2));
      hi = fminf(hi, fmaxf(e1, e2));
    }
    const int j0 = max(ib0, (int)ceilf(xibf + lo - pad)), j1 = min(ib1, (int)floorf(xibf + hi + pad));
    const T ec = (T)ic - xic;
    for (int ib = j0; ib <= j1; ++ib) {
      const T eb = (T)ib - xib;
      if (fabs(dot2(cs, eb, -sn, ec)) < S && fabs(dot2(sn, eb, cs, ec)) < S && n < kListMax)
        list[n++][lane] = (unsigned)ib | ((unsigned)ic << 16);
    }
  }
  return n;
}

// In-plane geometry of a listed column: its offset x^ref - x_n in the plane and lever R r.
template <typename T, int AX>
struct Column {
  int ib, ic;
  T ob, oc, lb, lc;
  __device__ __forceinline__ Column(const Geo& g, unsigned e, T xib, T xic, T cs, T sn, const T (&d)[3]) {
    constexpr int b = Axes<AX>::B, c = Axes<AX>::C;
    ib = (int)(e & 0xffffu);
    ic = (int)(e >> 16);
    const T eb = (T)ib - xib, ec = (T)ic - xic;
    ob = dot2(cs, eb, -sn, ec);
    oc = dot2(sn, eb, cs, ec);
    lb = ob + d[b];
    lc = oc + d[c];
  }
};

// The axial window of a lane's planes: weights of the four taps (the same for each plane), the first
// plane's first tap ia0, strides.
template <typename T, int AX>
struct Axial {
  T w[4], dw[4];
  bool in[4];  // the tap lies within the support
  int ia0;
  __device__ __forceinline__ Axial(const Geo& g, T da) {
    constexpr int a = Axes<AX>::A;
    const T S = (T)g.s, xia = da + pivot<T>(g, a), fl = floor(xia), fr = xia - fl;
    ia0 = (int)fl - g.s + 1;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const T o = fr + (T)(g.s - 1 - q);  // x_n - x^ref along the axis
      w[q] = dw[q] = T(0);
      in[q] = q < 2 * g.s && fabs(o) < S;
      if (in[q]) {
        if constexpr (sizeof(T) == 8) {
          if (g.wk == W_COS4) {
            double s, c;
            sincospi(0.5 * o, &s, &c);
            w[q] = 0.25 * (1.0 + c);
            dw[q] = -0.125 * 3.141592653589793 * s;
            continue;
          }
        }
        w[q] = wfun(g.wk, o);
        dw[q] = dwfun(g.wk, o);
      }
    }
  }
};
template <int AX>
__device__ __forceinline__ void design_strides(const Geo& g, int& sb, int& sc, int& sa) {
  const int s[3] = {1, g.nd[0], g.nd[0] * g.nd[1]};
  sb = s[Axes<AX>::B];
  sc = s[Axes<AX>::C];
  sa = s[Axes<AX>::A];
}

// Z + 3 values of kappa of a listed column from the axial window's first tap, zero off the design grid.
// The window is the same for a warp's lanes, so the test for one inside the grid does not diverge.
template <typename T, int Z>
__device__ __forceinline__ void load_window(const T* __restrict__ kc, int ia0, int na, int sa, T (&kv)[Z + kPadPts]) {
  const T* p = kc + (long long)ia0 * sa;
  if (ia0 >= 0 && ia0 + Z + kPadPts <= na) {
#pragma unroll
    for (int m = 0; m < Z + kPadPts; ++m) kv[m] = __ldg(p + m * sa);
  } else {
#pragma unroll
    for (int m = 0; m < Z + kPadPts; ++m) kv[m] = (ia0 + m >= 0 && ia0 + m < na) ? __ldg(p + m * sa) : T(0);
  }
}

// Sums of ZC planes of one in-plane position: phi, kappa, P = sum W l, L = sum W kappa l (in the plane).
template <typename T, int Z>
struct PlaneSums {
  T phi[Z], kap[Z], Pb[Z], Pc[Z], Lb[Z], Lc[Z];
};
// visit (a test export): called with the plane and the linear index of each design point that is summed.
struct NoPlaneVisit {};
template <typename T, int AX, bool BALL, int Z, typename Visit = NoPlaneVisit>
__device__ __forceinline__ void plane_sums(const Geo& g, const T* __restrict__ kref, const T (&d)[3], T cs, T sn, int n,
                                           const unsigned (*list)[32], int lane, PlaneSums<T, Z>& o,
                                           Visit visit = Visit()) {
  constexpr int b = Axes<AX>::B, c = Axes<AX>::C, a = Axes<AX>::A;
  const T xib = dot2(cs, d[b], sn, d[c]) + pivot<T>(g, b), xic = dot2(cs, d[c], -sn, d[b]) + pivot<T>(g, c);
  const Axial<T, AX> ax(g, d[a]);
  int sb, sc, sa;
  design_strides<AX>(g, sb, sc, sa);
  T f2 = T(0), pb2 = T(0), pc2 = T(0);
#pragma unroll
  for (int j = 0; j < Z; ++j) o.phi[j] = o.kap[j] = o.Pb[j] = o.Pc[j] = o.Lb[j] = o.Lc[j] = T(0);
  auto column_at = [&](unsigned e) { return kref + (int)(e & 0xffffu) * sb + (int)(e >> 16) * sc; };
  // the next column's kappa is loaded while this one's is used
  T kn[Z + kPadPts];
  unsigned en = n > 0 ? list[0][lane] : 0;
  if (n > 0) load_window<T, Z>(column_at(en), ax.ia0, g.nd[a], sa, kn);
  for (int i = 0; i < n; ++i) {
    const Column<T, AX> q(g, en, xib, xic, cs, sn, d);
    T kv[Z + kPadPts];
#pragma unroll
    for (int m = 0; m < Z + kPadPts; ++m) kv[m] = kn[m];
    if (i + 1 < n) {
      en = list[i + 1][lane];
      load_window<T, Z>(column_at(en), ax.ia0, g.nd[a], sa, kn);
    }
    const T w2 = mul_(wfun(g.wk, q.ob), wfun(g.wk, q.oc));
    const T wb = mul_(w2, q.lb), wc = mul_(w2, q.lc);
    int left = 0;
    if (BALL) left = g.rad4 - dsq(q.ib, g.nd[b]) - dsq(q.ic, g.nd[c]);
    if constexpr (!std::is_same_v<Visit, NoPlaneVisit>)
      for (int j = 0; j < Z; ++j)
        for (int m = 0; m < 4; ++m) {
          const int ia = ax.ia0 + j + m;
          if (ax.in[m] && ia >= 0 && ia < g.nd[a] && (!BALL || dsq(ia, g.nd[a]) <= left))
            visit(j, q.ib * sb + q.ic * sc + ia * sa);
        }
    if (!BALL) {
      f2 += w2;
      pb2 += wb;
      pc2 += wc;
    }
#pragma unroll
    for (int j = 0; j < Z; ++j) {
      const T s = fma_(ax.w[3], kv[j + 3], fma_(ax.w[2], kv[j + 2], dot2(ax.w[1], kv[j + 1], ax.w[0], kv[j])));
      o.kap[j] = fma_(w2, s, o.kap[j]);
      o.Lb[j] = fma_(wb, s, o.Lb[j]);
      o.Lc[j] = fma_(wc, s, o.Lc[j]);
      if (BALL) {  // the points of the design domain only (kappa is zero off it)
        T s1 = T(0);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const int ia = ax.ia0 + j + m;
          if (ia >= 0 && ia < g.nd[a] && dsq(ia, g.nd[a]) <= left) s1 += ax.w[m];
        }
        o.phi[j] = fma_(w2, s1, o.phi[j]);
        o.Pb[j] = fma_(wb, s1, o.Pb[j]);
        o.Pc[j] = fma_(wc, s1, o.Pc[j]);
      }
    }
  }
  if (!BALL)
#pragma unroll
    for (int j = 0; j < Z; ++j) {
      T s1 = T(0);
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const int ia = ax.ia0 + j + m;
        if (ia >= 0 && ia < g.nd[a]) s1 += ax.w[m];
      }
      o.phi[j] = mul_(f2, s1);
      o.Pb[j] = mul_(pb2, s1);
      o.Pc[j] = mul_(pc2, s1);
    }
}

// Grid indices of a lane's Z cells: the in-plane part once, the axial one stepped (wrapped on a periodic
// axis). ok: bit j set if cell j is in the box and on the grid; forb: it may not be touched by the body.
template <int AX, int Z>
struct LaneCells {
  long long n0;
  int pa, na, sa;  // first axial coordinate (wrapped if periodic), extent, stride
  unsigned box, ok, forb;
  bool per;
  __device__ __forceinline__ LaneCells(const Geo& g, const int (&lo)[3], const LanePos& lp) {
    constexpr int b = Axes<AX>::B, c = Axes<AX>::C, a = Axes<AX>::A;
    const int st[3] = {1, g.n[0], g.n[0] * g.n[1]};
    bool in = lp.ok, fb = false;
    n0 = 0;
#pragma unroll
    for (int e = 0; e < 3; ++e) {
      if (e == a) continue;
      int p = lo[e] + lp.j[e];
      if (g.bc[e] == BC_PERIODIC) {
        p = wrapi(p, g.n[e]);
      } else {
        fb = fb || p < 2 || p > g.n[e] - 3;
        in = in && p >= 0 && p < g.n[e];
      }
      n0 += (long long)p * st[e];
    }
    per = g.bc[a] == BC_PERIODIC;
    na = g.n[a];
    sa = st[a];
    pa = lo[a] + lp.j[a];
    if (per) pa = wrapi(pa, na);
    box = ok = forb = 0;
#pragma unroll
    for (int j = 0; j < Z; ++j) {
      const bool ib = lp.ok && lp.j[a] + j < g.B[a];
      if (ib) box |= 1u << j;
      if (ib && in && (per || (pa + j >= 0 && pa + j < na))) ok |= 1u << j;
      if (fb || (!per && (pa + j < 2 || pa + j > na - 3))) forb |= 1u << j;
    }
    (void)b;
    (void)c;
  }
  __device__ __forceinline__ long long at(int j) const {
    int p = pa + j;
    if (per && p >= na) p -= na;  // (the box fits the axis, so a chunk wraps at most once)
    return n0 + (long long)p * sa;
  }
};

// us of a cell from its sums.
template <typename T, int AX, typename U>
__device__ __forceinline__ T solid_velocity(int a, const U& ug, T om, T phi, T Pb, T Pc) {
  constexpr int b = Axes<AX>::B, c = Axes<AX>::C;
  return a == b ? dot2(ug[a], phi, -om, Pc) : (a == c ? dot2(ug[a], phi, om, Pb) : mul_(ug[a], phi));
}

template <typename T, int AX, bool BALL>
__global__ void __launch_bounds__(512, 1)
    k_couple_axis3d(Geo g, Slots<T> S, Ctrl* ctrl, Dof* it, const T* __restrict__ kref,
                    const Moments* __restrict__ mom, void* words, T* __restrict__ boxstore, int nbox, int di) {
  using V = typename SumOf<T>::type;
  constexpr int Z = Planes<T>::ZC, NV = 4, b = Axes<AX>::B, c = Axes<AX>::C, a3 = Axes<AX>::A;
  constexpr int DW = (int)(sizeof(Dof) / sizeof(double));
  extern __shared__ __align__(16) unsigned lists[];
  __shared__ V part[16 * NV];
  __shared__ Dof sd[2];  // CTA 0: s(t-1), the current iterate
  __shared__ Pose<T, 3> pose;
  __shared__ int gave_up;
  if (*(volatile int*)&ctrl->status & ST_SYNC_TIMEOUT) return;  // an earlier launch gave up
  const int t = ctrl->t0 + di, base = ctrl->base, K = g.K;
  Dof* row = it + (long long)(t - 1) * (K + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = (int)(blockDim.x >> 5);
  const int G = (int)gridDim.x - 1, cta = (int)blockIdx.x - 1;  // CTAs with cells
  const unsigned e0 = (unsigned)((long long)(t - 1) * K);
  if (tid < DW) {
    const double v = reinterpret_cast<const double*>(row)[tid];
    reinterpret_cast<double*>(sd)[tid] = v;
    reinterpret_cast<double*>(sd)[DW + tid] = v;
  }
  if (tid == 0) gave_up = 0;
  __syncthreads();
  if (cta < 0) {
    flag_root<T, 3, AX>(g, ctrl, row, mom, words, G, e0, (ctrl->sync_skip & 1) != 0, sd, gave_up);
    return;
  }
  if (tid == 0) pose.set(sd[0]);
  T* __restrict__ dst = slot_ptr(S, t, base);
  int lo[3];
  box_origin<3>(g, sd[0], lo[0], lo[1], lo[2]);
  T* bs = boxstore ? boxstore + (long long)((t - base - 1) % nbox) * g.box_cells * 3 : nullptr;
  const long long N = g.N;
  unsigned(*list)[32] = reinterpret_cast<unsigned(*)[32]>(lists + warp * kListMax * 32);
  const int tiles = plane_tiles<AX>(g), units = (int)plane_units<AX>(g, Z);
  __syncthreads();
  for (int k = 1; k <= K; ++k) {
    const bool last = k == K;
    const Pose<T, 3> P = pose;
    V v[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i].zero();
    for (int u0 = warp * G + cta; u0 < units; u0 += G * nw) {  // uniform per warp
      const LanePos lp = lane_pos<AX>(g, u0, tiles, Z, lane);
      const T d[3] = {P.rel(0, lo[0] + lp.j[0]), P.rel(1, lo[1] + lp.j[1]), P.rel(2, lo[2] + lp.j[2])};
      const int n = column_list<T, AX>(g, d, P.cs, P.sn, lp.ok, list, lane);
      PlaneSums<T, Z> A;
      plane_sums<T, AX, BALL, Z>(g, kref, d, P.cs, P.sn, n, list, lane, A);
      const LaneCells<AX, Z> lc(g, lo, lp);
      unsigned work = 0;  // cells the body reaches (the others keep u = u*)
#pragma unroll
      for (int j = 0; j < Z; ++j)
        if (A.phi[j] > T(0)) work |= 1u << j;
      if (work & (lc.forb | (lc.box & ~lc.ok))) atomicOr(&ctrl->status, ST_BODY_OUTSIDE);
      work &= lc.ok;
      const unsigned stored = last && bs ? lc.ok : work;
      const long long bl0 = lp.j[0] + (long long)g.B[0] * (lp.j[1] + (long long)g.B[1] * lp.j[2]);
      const int sbx = a3 == 0 ? 1 : (a3 == 1 ? g.B[0] : g.B[0] * g.B[1]);
      T us[Z][3];
#pragma unroll
      for (int j = 0; j < Z; ++j)
#pragma unroll
        for (int a = 0; a < 3; ++a) us[j][a] = (stored >> j & 1u) ? dst[(a + 1) * N + lc.at(j)] : T(0);
#pragma unroll
      for (int j = 0; j < Z; ++j) {
        const T inv = T(1) / (T(1) + A.kap[j]);
        T uu[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const T sv = solid_velocity<T, AX>(a, P.ug, P.om, A.phi[j], A.Pb[j], A.Pc[j]);
          uu[a] = brinkman(us[j][a], A.kap[j], sv, inv);
        }
        if (work >> j & 1u) {
#pragma unroll
          for (int a = 0; a < 3; ++a) run_add(v[a], A.kap[j] * uu[a]);
          run_add(v[3], A.Lb[j] * uu[c] - A.Lc[j] * uu[b]);
          if (last)
#pragma unroll
            for (int a = 0; a < 3; ++a) dst[(a + 1) * N + lc.at(j)] = uu[a];
        }
        if (last && bs && (stored >> j & 1u))
#pragma unroll
          for (int a = 0; a < 3; ++a) bs[a * g.box_cells + bl0 + (long long)j * sbx] = us[j][a];
      }
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      warp_total<1>(v[i]);
      if (lane == 0) part[warp * NV + i] = v[i];
    }
    __syncthreads();
    flag_exchange<T, 3>(words, e0 + (unsigned)k, cta, G, last, &ctrl->status, part, pose, gave_up);
    if (last) return;
    __syncthreads();
    if (gave_up) return;
  }
}

constexpr int kApplyWarps = 4;
template <typename T, int AX, bool BALL>
__global__ void __launch_bounds__(kApplyWarps * 32) k_apply_axis3d(Geo g, Slots<T> S, const Ctrl* ctrl, const Dof* it,
                                                                   const T* __restrict__ kref,
                                                                   T* __restrict__ boxstore, int nbox, int di) {
  constexpr int Z = Planes<T>::ZC, a3 = Axes<AX>::A;
  __shared__ unsigned lists[kApplyWarps][kListMax][32];
  const int t = ctrl->t0 + di, base = ctrl->base, K = g.K;
  const Dof* row = it + (long long)(t - 1) * (K + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int u0 = blockIdx.x * kApplyWarps + warp, tiles = plane_tiles<AX>(g);
  if (u0 >= plane_units<AX>(g, Z)) return;
  T* __restrict__ dst = slot_ptr(S, t, base);
  T* bs = boxstore + (long long)((t - base - 1) % nbox) * g.box_cells * 3;
  int lo[3];
  box_origin<3>(g, row[0], lo[0], lo[1], lo[2]);
  const DofView<T> P(row[K - 1]);
  const LanePos lp = lane_pos<AX>(g, u0, tiles, Z, lane);
  const T d[3] = {P.rel(0, lo[0] + lp.j[0]), P.rel(1, lo[1] + lp.j[1]), P.rel(2, lo[2] + lp.j[2])};
  const int n = column_list<T, AX>(g, d, P.cs, P.sn, lp.ok, lists[warp], lane);
  PlaneSums<T, Z> A;
  plane_sums<T, AX, BALL, Z>(g, kref, d, P.cs, P.sn, n, lists[warp], lane, A);
  const LaneCells<AX, Z> lc(g, lo, lp);
  const long long bl0 = lp.j[0] + (long long)g.B[0] * (lp.j[1] + (long long)g.B[1] * lp.j[2]);
  const int sbx = a3 == 0 ? 1 : (a3 == 1 ? g.B[0] : g.B[0] * g.B[1]);
  T us[Z][3];
#pragma unroll
  for (int j = 0; j < Z; ++j)
#pragma unroll
    for (int a = 0; a < 3; ++a) us[j][a] = (lc.ok >> j & 1u) ? dst[(a + 1) * g.N + lc.at(j)] : T(0);
#pragma unroll
  for (int j = 0; j < Z; ++j) {
    if (!(lc.ok >> j & 1u)) continue;
    const T inv = T(1) / (T(1) + A.kap[j]);
    const bool body = A.phi[j] > T(0);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const T sv = solid_velocity<T, AX>(a, P.ug, P.om, A.phi[j], A.Pb[j], A.Pc[j]);
      bs[a * g.box_cells + bl0 + (long long)j * sbx] = us[j][a];
      if (body) dst[(a + 1) * g.N + lc.at(j)] = brinkman(us[j][a], A.kap[j], sv, inv);
    }
  }
}

// The box of the iterate s, gathered as k_couple_axis3d does, with the accepted index sets as out[box cell][5].
template <typename T, int AX, bool BALL>
__global__ void __launch_bounds__(kApplyWarps * 32) k_support_axis3d(Geo g, Dof s, const T* __restrict__ kref,
                                                                     long long* __restrict__ out) {
  constexpr int Z = Planes<T>::ZC, a3 = Axes<AX>::A;
  __shared__ unsigned lists[kApplyWarps][kListMax][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int u0 = blockIdx.x * kApplyWarps + warp, tiles = plane_tiles<AX>(g);
  if (u0 >= plane_units<AX>(g, Z)) return;
  int lo[3];
  box_origin<3>(g, s, lo[0], lo[1], lo[2]);
  const DofView<T> P(s);
  const LanePos lp = lane_pos<AX>(g, u0, tiles, Z, lane);
  const T d[3] = {P.rel(0, lo[0] + lp.j[0]), P.rel(1, lo[1] + lp.j[1]), P.rel(2, lo[2] + lp.j[2])};
  const int n = column_list<T, AX>(g, d, P.cs, P.sn, lp.ok, lists[warp], lane);
  SetStats st[Z];
  PlaneSums<T, Z> A;
  auto visit = [&](int j, int m) { st[j].add(m); };
  plane_sums<T, AX, BALL, Z>(g, kref, d, P.cs, P.sn, n, lists[warp], lane, A, visit);
  const int sbx = a3 == 0 ? 1 : (a3 == 1 ? g.B[0] : g.B[0] * g.B[1]);
  const long long bl0 = lp.j[0] + (long long)g.B[0] * (lp.j[1] + (long long)g.B[1] * lp.j[2]);
  for (int j = 0; j < Z; ++j)
    if (lp.ok && lp.j[a3] + j < g.B[a3]) st[j].store(out, bl0 + (long long)j * sbx);
}

// The planes and sums of k_rev_coef (whole design domain; a ball takes that kernel). Sums over the
// design columns per plane, of kappa: with W, dW/db, dW/dc times 1, l_b, l_c, with dW/da likewise, and
// the rotation derivative times l_b, l_c; without kappa the planes share the in-plane sums.
// A thread's planes are added as pairs (packed FP32). FP32 runs two CTAs per SM (128 registers): with 22 more
// for the pairs, one CTA of 184 took 90 us a step of the 48^3 body (planes and matrices together) and left the
// chain's kernels no place beside it; two take 70, against 80 before the pairs (170 registers, FP32 sums).
template <typename T, int AX>
__global__ void __launch_bounds__(kRevThreads, sizeof(T) == 4 ? 2 : 1) k_coef_axis3d(Geo g, const Ctrl* ctrl, const Dof* it,
                                                             const T* __restrict__ kref,
                                                             const T* __restrict__ boxstore, int nbox,
                                                             T* __restrict__ slabs, long long slab,
                                                             typename Partial<T>::type* __restrict__ mpart, int di) {
  using RS = RevSums<3>;
  constexpr int Z = Planes<T>::ZR, b = Axes<AX>::B, c = Axes<AX>::C, a3 = Axes<AX>::A, NW = kRevThreads / 32;
  extern __shared__ __align__(16) unsigned char rev_smem[];
  unsigned(*list)[32] = reinterpret_cast<unsigned(*)[32]>(rev_smem) + (threadIdx.x >> 5) * kListMax;
  const int K = g.K, k = (int)blockIdx.y + 1, i = blockIdx.z;
  const int t = rev_step(ctrl, di, i), base = ctrl->base;
  const Dof* row = it + (long long)(t - 1) * (K + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int u0 = blockIdx.x * NW + warp, tiles = plane_tiles<AX>(g);
  typename SumOf<T>::type v[RS::N];
#pragma unroll
  for (int q = 0; q < RS::N; ++q) v[q].zero();
  if (u0 < plane_units<AX>(g, Z)) {
    int lo[3];
    box_origin<3>(g, row[0], lo[0], lo[1], lo[2]);
    const DofView<T> P(row[k - 1]);
    const LanePos lp = lane_pos<AX>(g, u0, tiles, Z, lane);
    const T d[3] = {P.rel(0, lo[0] + lp.j[0]), P.rel(1, lo[1] + lp.j[1]), P.rel(2, lo[2] + lp.j[2])};
    const int n = column_list<T, AX>(g, d, P.cs, P.sn, lp.ok, list, lane);
    const T xib = dot2(P.cs, d[b], P.sn, d[c]) + pivot<T>(g, b), xic = dot2(P.cs, d[c], -P.sn, d[b]) + pivot<T>(g, c);
    const Axial<T, AX> ax(g, d[a3]);
    int sb, sc, sa;
    design_strides<AX>(g, sb, sc, sa);
    // in-plane sums without kappa: [W, dW/db, dW/dc][1, l_b, l_c], and the rotation derivative's
    T f[3][3], fq[2];
    T s[Z][4][3], sq[Z][2];  // of kappa by plane: [W, dW/db, dW/dc, dW/da][1, l_b, l_c]
#pragma unroll
    for (int e = 0; e < 3; ++e) f[e][0] = f[e][1] = f[e][2] = T(0);
    fq[0] = fq[1] = T(0);
#pragma unroll
    for (int j = 0; j < Z; ++j) {
#pragma unroll
      for (int e = 0; e < 4; ++e) s[j][e][0] = s[j][e][1] = s[j][e][2] = T(0);
      sq[j][0] = sq[j][1] = T(0);
    }
    auto column_at = [&](unsigned e) { return kref + (int)(e & 0xffffu) * sb + (int)(e >> 16) * sc; };
    T kn[Z + kPadPts];
    unsigned en = n > 0 ? list[0][lane] : 0;
    if (n > 0) load_window<T, Z>(column_at(en), ax.ia0, g.nd[a3], sa, kn);
    for (int q0 = 0; q0 < n; ++q0) {
      const Column<T, AX> q(g, en, xib, xic, P.cs, P.sn, d);
      T kv[Z + kPadPts];
#pragma unroll
      for (int m = 0; m < Z + kPadPts; ++m) kv[m] = kn[m];
      if (q0 + 1 < n) {
        en = list[q0 + 1][lane];
        load_window<T, Z>(column_at(en), ax.ia0, g.nd[a3], sa, kn);
      }
      T wb, dwb, wc, dwc;
      w_dw(g.wk, -q.ob, &wb, &dwb);
      w_dw(g.wk, -q.oc, &wc, &dwc);
      const T w[3] = {wb * wc, dwb * wc, wb * dwc};
      const T rt = w[1] * q.lc - w[2] * q.lb, rb = rt * q.lb, rc = rt * q.lc;
      T wl[3][2];
#pragma unroll
      for (int e = 0; e < 3; ++e) {
        wl[e][0] = w[e] * q.lb;
        wl[e][1] = w[e] * q.lc;
        f[e][0] += w[e];
        f[e][1] += wl[e][0];
        f[e][2] += wl[e][1];
      }
      fq[0] += rb;
      fq[1] += rc;
#pragma unroll
      for (int j = 0; j < Z; ++j) {
        const T s0 = ax.w[0] * kv[j] + ax.w[1] * kv[j + 1] + ax.w[2] * kv[j + 2] + ax.w[3] * kv[j + 3];
        const T s1 = ax.dw[0] * kv[j] + ax.dw[1] * kv[j + 1] + ax.dw[2] * kv[j + 2] + ax.dw[3] * kv[j + 3];
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          s[j][e][0] += w[e] * s0;
          s[j][e][1] += wl[e][0] * s0;
          s[j][e][2] += wl[e][1] * s0;
        }
        s[j][3][0] += w[0] * s1;
        s[j][3][1] += wl[0][0] * s1;
        s[j][3][2] += wl[0][1] * s1;
        sq[j][0] += rb * s0;
        sq[j][1] += rc * s0;
      }
    }
    const T* bs = boxstore + (long long)((t - base - 1) % nbox) * g.box_cells * 3;
#pragma unroll
    for (int j = 0; j < Z; ++j) {
      int jj[3] = {lp.j[0], lp.j[1], lp.j[2]};
      jj[a3] += j;
      if (!lp.ok || jj[a3] >= g.B[a3]) continue;
      T a0 = T(0), a1 = T(0);  // the axial weights' sums over the taps on the design grid
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const int ia = ax.ia0 + j + m;
        if (ia >= 0 && ia < g.nd[a3]) {
          a0 += ax.w[m];
          a1 += ax.dw[m];
        }
      }
      long long m;
      const bool ing = cell_index<3>(g, lo[0] + jj[0], lo[1] + jj[1], lo[2] + jj[2], m);
      Moments1<T> A;
      auto put = [&](int at, const T (&f3)[3], T fa, const T (&k3)[3]) {
        A.phi[at] = ing ? f3[0] * fa : T(0);
        A.Pb[at] = ing ? f3[1] * fa : T(0);
        A.Pc[at] = ing ? f3[2] * fa : T(0);
        A.kap[at] = ing ? k3[0] : T(0);
        A.Lb[at] = ing ? k3[1] : T(0);
        A.Lc[at] = ing ? k3[2] : T(0);
      };
      put(0, f[0], a0, s[j][0]);
      put(1 + b, f[1], a0, s[j][1]);
      put(1 + c, f[2], a0, s[j][2]);
      put(1 + a3, f[0], a1, s[j][3]);
      A.qPb = ing ? fq[0] * a0 : T(0);
      A.qPc = ing ? fq[1] * a0 : T(0);
      A.qLb = ing ? sq[j][0] : T(0);
      A.qLc = ing ? sq[j][1] : T(0);
      const long long bl = jj[0] + (long long)g.B[0] * (jj[1] + (long long)g.B[1] * jj[2]);
      T one[RS::N];
      rev_cell<T, 3, AX>(g, P, A, ing, bs, bl, slabs + (long long)i * slab + bl, k, one);
#pragma unroll
      for (int q = 0; q < RS::N; q += 2) {
        if (j == 0) {
          v[q].set(one[q]);
          v[q + 1].set(one[q + 1]);
        } else {
          run_add2(v[q], v[q + 1], one[q], one[q + 1]);
        }
      }
    }
  }
  row_sums<RS::N>(v, reinterpret_cast<T*>(rev_smem),
                  mpart + (((long long)i * K + (k - 1)) * gridDim.x + blockIdx.x) * RS::N);
}

// dJ/dkappa^ref of ZD design points of a column along the axis: over the 4 x 4 in-plane window the
// axial sums of u and dJ/dkappa_n for the ZD points from ZD + 3 planes, then the in-plane weight.
template <typename T>
struct DesignCol {
  static constexpr int ZD = sizeof(T) == 4 ? 8 : 4;
};
template <typename T, int AX>
__global__ void __launch_bounds__(128) k_design_axis3d(Geo g, Ctrl* ctrl, const Dof* it, const T* __restrict__ slabs,
                                                       long long slab, const T* __restrict__ lamh,
                                                       double* __restrict__ dkp, int nsteps, int di) {
  using RP = RevPlanes<3>;
  constexpr int Z = DesignCol<T>::ZD, b = Axes<AX>::B, c = Axes<AX>::C, a3 = Axes<AX>::A;
  const int K = g.K;
  // the in-plane axis that is x runs fastest over the threads
  constexpr int fast = InPlane<AX>::b_fast ? b : c, slow = InPlane<AX>::b_fast ? c : b;
  const int cols = g.nd[b] * g.nd[c], chunks = (g.nd[a3] + Z - 1) / Z;
  const int th = blockIdx.x * 128 + threadIdx.x;
  const int ch = th / cols, q = th - ch * cols;
  if (ch >= chunks) return;
  int id[3];
  id[slow] = q / g.nd[fast];
  id[fast] = q - id[slow] * g.nd[fast];
  id[a3] = ch * Z;
  int np = min(Z, g.nd[a3] - id[a3]);  // points of this thread
  // A ball: only the column's points in the design domain (consecutive ones). The body box is sized to the
  // domain, so the window of a point off it may lie outside the box, and must not decide for the others.
  if (g.rad4 != INT_MAX) {
    const int left = g.rad4 - dsq(id[b], g.nd[b]) - dsq(id[c], g.nd[c]);
    while (np > 0 && dsq(id[a3] + np - 1, g.nd[a3]) > left) --np;
    while (np > 0 && dsq(id[a3], g.nd[a3]) > left) ++id[a3], --np;
    if (np == 0) return;
  }
  const T r[3] = {(T)id[0] - pivot<T>(g, 0), (T)id[1] - pivot<T>(g, 1), (T)id[2] - pivot<T>(g, 2)};
  const long long BC = g.box_cells;
  const int st[3] = {1, g.B[0], g.B[0] * g.B[1]}, S2 = 2 * g.s;
  bool inside = true;
  double acc[Z];
#pragma unroll
  for (int j = 0; j < Z; ++j) acc[j] = 0.0;
  for (int item = blockIdx.y; item < nsteps * K; item += gridDim.y) {
    const int i = item / K, k = K - item % K;
    const Dof* row = it + (long long)(rev_step(ctrl, di, i) - 1) * (K + 1);
    int lo[3];
    box_origin<3>(g, row[0], lo[0], lo[1], lo[2]);
    const DofView<T> V(row[k - 1]);
    T l[3], dl[3], fr[3], w[3][4];
    int f[3];
    rot<AX>(V.cs, V.sn, r, l);
    drot<AX>(V.cs, V.sn, r, dl);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      V.split(a, l[a], &f[a], &fr[a]);
      window_weights(g, fr[a], w[a]);
      f[a] += 1 - g.s - lo[a];
    }
    // cells with weight 0 (fr = 0 puts the window's last one on the support's edge) need not lie in the box
    bool in = true;
#pragma unroll
    for (int a = 0; a < 3; ++a)
      in = in && f[a] >= 0 && f[a] + S2 - 1 - (fr[a] == T(0)) + (a == a3 ? np - 1 : 0) < g.B[a];
    if (!in) {
      inside = false;
      continue;
    }
    const T* Pk = slabs + (long long)i * slab + (long long)(k - 1) * RP::per_itr * BC;
    const int o0 = f[0] * st[0] + f[1] * st[1] + f[2] * st[2];
    T sum[Z][4];  // u, dJ/dkappa_n
#pragma unroll
    for (int j = 0; j < Z; ++j) sum[j][0] = sum[j][1] = sum[j][2] = sum[j][3] = T(0);
    const int top = min(np + S2 - 1, g.B[a3] - f[a3]);  // planes of the window that are read
    auto weight = [&](int q2) {  // in-plane weight of window cell q2 = qb + S2 qc
      const int qc = q2 / S2, qb = q2 - qc * S2;
      const T wc = qc == 0 ? w[c][0] : (qc == 1 ? w[c][1] : (qc == 2 ? w[c][2] : w[c][3]));
      return wc * (qb == 0 ? w[b][0] : (qb == 1 ? w[b][1] : (qb == 2 ? w[b][2] : w[b][3])));
    };
    auto load = [&](int q2, int fl, bool on, T (&x)[Z + kPadPts]) {
      const int qc = q2 / S2, qb = q2 - qc * S2;
      const T* F = Pk + (fl < 3 ? RP::u + fl : RP::eps) * BC + (o0 + qb * st[b] + qc * st[c]);
#pragma unroll
      for (int m = 0; m < Z + kPadPts; ++m) x[m] = on && m < top ? __ldg(F + m * st[a3]) : T(0);
    };
    // each field's values are loaded while the one before is used
    T w2 = weight(0), wn = T(0), x[Z + kPadPts], xn[Z + kPadPts];
    load(0, 0, w2 != T(0), x);
#pragma unroll 1
    for (int q2 = 0; q2 < S2 * S2; ++q2) {
      const bool more = q2 + 1 < S2 * S2;
      wn = more ? weight(q2 + 1) : T(0);
#pragma unroll
      for (int fl = 0; fl < 4; ++fl) {
        if (fl < 3)
          load(q2, fl + 1, w2 != T(0), xn);
        else
          load(more ? q2 + 1 : q2, 0, wn != T(0), xn);
#pragma unroll
        for (int j = 0; j < Z; ++j)
          sum[j][fl] += w2 * (w[a3][0] * x[j] + w[a3][1] * x[j + 1] + w[a3][2] * x[j + 2] + w[a3][3] * x[j + 3]);
#pragma unroll
        for (int m = 0; m < Z + kPadPts; ++m) x[m] = xn[m];
      }
      w2 = wn;
    }
    const T* lam = lamh + ((long long)i * K + (k - 1)) * 4;
#pragma unroll
    for (int j = 0; j < Z; ++j) {
      T D[3], dk = sum[j][3];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        D[a] = sum[j][a] - (V.ug[a] + V.om * dl[a]);
        dk += lam[a] * D[a];
      }
      dk += lam[3] * (l[b] * D[c] - l[c] * D[b]);
      acc[j] += (double)dk;
    }
  }
  if (!inside) atomicOr(&ctrl->status, ST_BOX_OVERFLOW);
  const int sd[3] = {1, g.nd[0], g.nd[0] * g.nd[1]};
  const int m0 = id[0] * sd[0] + id[1] * sd[1] + id[2] * sd[2];
#pragma unroll
  for (int j = 0; j < Z; ++j)
    if (j < np) dkp[(long long)blockIdx.y * g.ND + m0 + j * sd[a3]] += acc[j];
}

constexpr size_t list_bytes(int warps) { return (size_t)warps * kListMax * 32 * sizeof(unsigned); }

template <typename T, int AX, bool BALL>
int couple_shape(const Geo& g, int* threads) {
  int dev = 0, sms = 0, per_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 2) return 0;
  const long long units = plane_units<AX>(g, Planes<T>::ZC);
  long long nw = (units + sms - 2) / (sms - 1);
  nw = nw < 5 ? 5 : (nw > 16 ? 16 : nw);  // four warps sum, the last one waits for the iterate
  auto* kernel = k_couple_axis3d<T, AX, BALL>;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)list_bytes(16)) != cudaSuccess) return 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, (int)nw * 32, list_bytes((int)nw)) != cudaSuccess) return 0;
  if (per_sm < 1) return 0;
  *threads = (int)nw * 32;
  const long long ctas = (units + nw - 1) / nw + 1, cap = sms < kFlagMaxCtas ? sms : kFlagMaxCtas;
  return (int)(ctas < cap ? ctas : cap);
}

// Dispatch on the axis and on whether the design domain is a ball.
#define LKS_AXIS_BALL(F, ...)                                                           \
  do {                                                                                  \
    const bool ball_ = g.rad4 != INT_MAX;                                               \
    if (g.ax == 0) { if (ball_) F<T, 0, true>(__VA_ARGS__); else F<T, 0, false>(__VA_ARGS__); } \
    else if (g.ax == 1) { if (ball_) F<T, 1, true>(__VA_ARGS__); else F<T, 1, false>(__VA_ARGS__); } \
    else { if (ball_) F<T, 2, true>(__VA_ARGS__); else F<T, 2, false>(__VA_ARGS__); }   \
  } while (0)

template <typename T, int AX, bool BALL>
void shape_ax(Geo* gp) { gp->flag_ctas = couple_shape<T, AX, BALL>(*gp, &gp->flag_threads); }
template <typename T>
void shape_any(Geo* gp) {
  const Geo& g = *gp;
  LKS_AXIS_BALL(shape_ax, gp);
}
template <typename T, int AX, bool BALL>
void couple_ax(const Geo& g, const Slots<T>& S, Ctrl* ctrl, Dof* it, const T* kref, const Moments* mom, void* words,
               T* boxstore, int nbox, int di, cudaStream_t st) {
  launch_coop(k_couple_axis3d<T, AX, BALL>, dim3((unsigned)g.flag_ctas), dim3((unsigned)g.flag_threads),
              list_bytes(g.flag_threads / 32), st, g, S, ctrl, it, kref, mom, words, boxstore, nbox, di);
}
template <typename T, int AX, bool BALL>
void apply_ax(const Geo& g, const Slots<T>& S, const Ctrl* ctrl, const Dof* it, const T* kref, T* boxstore, int nbox,
              int di, cudaStream_t st) {
  const long long units = plane_units<AX>(g, Planes<T>::ZC);
  launch(k_apply_axis3d<T, AX, BALL>, dim3((unsigned)((units + kApplyWarps - 1) / kApplyWarps)), kApplyWarps * 32, 0, st,
         g, S, ctrl, it, kref, boxstore, nbox, di);
}
template <typename T, int AX, bool BALL>
void support_ax(const Geo& g, const Dof& s, const T* kref, long long* out, cudaStream_t st) {
  const long long units = plane_units<AX>(g, Planes<T>::ZC);
  launch(k_support_axis3d<T, AX, BALL>, dim3((unsigned)((units + kApplyWarps - 1) / kApplyWarps)), kApplyWarps * 32, 0, st,
         g, s, kref, out);
}
template <typename T, int AX>
int coef_ctas_ax(const Geo& g) {
  const long long units = plane_units<AX>(g, Planes<T>::ZR);
  return (int)((units + kRevThreads / 32 - 1) / (kRevThreads / 32));
}
template <typename T, int AX>
void coef_ax(const Geo& g, const RevBuffers& R, const Ctrl* ctrl, const Dof* it, const T* kref, const T* boxstore, int nbox,
             int nsteps, int di, cudaStream_t st) {
  const size_t rows = row_bytes<T>(RevSums<3>::N, true), lists = list_bytes(kRevThreads / 32);
  launch(k_coef_axis3d<T, AX>, dim3((unsigned)coef_ctas_ax<T, AX>(g), g.K, nsteps), kRevThreads, rows > lists ? rows : lists,
         st, g, ctrl, it, kref, boxstore, nbox, (T*)R.slabs, R.slab, (typename Partial<T>::type*)R.mpart, di);
}
template <typename T, int AX>
void design_ax(const Geo& g, const RevBuffers& R, Ctrl* ctrl, const Dof* it, int nsteps, int di, cudaStream_t st) {
  constexpr int Z = DesignCol<T>::ZD;
  const long long n = (long long)(g.ND / g.nd[Axes<AX>::A]) * ((g.nd[Axes<AX>::A] + Z - 1) / Z);
  launch(k_design_axis3d<T, AX>, dim3((unsigned)((n + 127) / 128), R.splits), 128, 0, st, g, ctrl, it,
         (const T*)R.slabs, R.slab, (const T*)R.lamh, R.dkp, nsteps, di);
}
#define LKS_AXIS(F, ...)                        \
  do {                                          \
    if (g.ax == 0) F<T, 0>(__VA_ARGS__);        \
    else if (g.ax == 1) F<T, 1>(__VA_ARGS__);   \
    else F<T, 2>(__VA_ARGS__);                  \
  } while (0)

}  // namespace

bool axis3d_fits(const Geo& g) {
  return g.dim == 3 && g.ax != AX_FREE && g.nd[0] < 65536 && g.nd[1] < 65536 && g.nd[2] < 65536 &&
         g.box_cells < (1LL << 29);
}

// Small boxes leave each SM one warp, whose list and window loads then make the iteration's time: up to
// 40,000 cells (FP64, where the per-iteration kernels are slower per cell, 10,000) those are as fast or
// faster. Forward us per step at 5 iterations, per-iteration -> this: FP32 18^3 cells 85 -> 91, 32^3 99 ->
// 99, 52 x 52 x 38 178 -> 114, 56^3 248 -> 108; FP64 20^3 635 -> 700, 28 x 28 x 22 936 -> 626.
void setup_couple_axis3d(Geo* g, bool fp64) {
  if (!axis3d_fits(*g) || g->box_cells <= (fp64 ? 10000 : 40000)) return;
  if (fp64)
    shape_any<double>(g);
  else
    shape_any<float>(g);
}

template <typename T>
void launch_couple_axis3d(const Geo& g, const Slots<T>& S, Ctrl* ctrl, Dof* it, const T* kref, const Moments* mom,
                          void* words, T* boxstore, int nbox, int di, cudaStream_t st) {
  LKS_AXIS_BALL(couple_ax, g, S, ctrl, it, kref, mom, words, boxstore, nbox, di, st);
}

template <typename T>
void launch_apply_axis3d(const Geo& g, const Slots<T>& S, const Ctrl* ctrl, const Dof* it, const T* kref, T* boxstore,
                         int nbox, int di, cudaStream_t st) {
  LKS_AXIS_BALL(apply_ax, g, S, ctrl, it, kref, boxstore, nbox, di, st);
}

template <typename T>
void launch_support_axis3d(const Geo& g, const Dof& s, const T* kref, long long* out, cudaStream_t st) {
  LKS_AXIS_BALL(support_ax, g, s, kref, out, st);
}

bool coef_axis3d_fits(const Geo& g) { return axis3d_fits(g) && g.rad4 == INT_MAX; }
int coef_axis3d_ctas(const Geo& g, bool fp64) {
  if (fp64) return g.ax == 0 ? coef_ctas_ax<double, 0>(g) : g.ax == 1 ? coef_ctas_ax<double, 1>(g) : coef_ctas_ax<double, 2>(g);
  return g.ax == 0 ? coef_ctas_ax<float, 0>(g) : g.ax == 1 ? coef_ctas_ax<float, 1>(g) : coef_ctas_ax<float, 2>(g);
}
// FP32: the two CTAs per SM take 62 KB of shared memory; asking for the split that holds just them (64 KB)
// leaves L1 the rest (157x67x70 duct gradient 6.64 -> 6.55 ms, 128x64x64 10.54 -> 10.51).
void prepare_coef_axis3d(const Geo& g) {
  const void* k[3] = {(const void*)k_coef_axis3d<float, 0>, (const void*)k_coef_axis3d<float, 1>,
                      (const void*)k_coef_axis3d<float, 2>};
  cudaFuncSetAttribute(k[g.ax], cudaFuncAttributePreferredSharedMemoryCarveout, 28);  // % of 228 KB; a hint
  cudaGetLastError();
}
template <typename T>
void launch_coef_axis3d(const Geo& g, const RevBuffers& R, const Ctrl* ctrl, const Dof* it, const T* kref, const T* boxstore,
                        int nbox, int nsteps, int di, cudaStream_t st) {
  LKS_AXIS(coef_ax, g, R, ctrl, it, kref, boxstore, nbox, nsteps, di, st);
}
template <typename T>
void launch_design_axis3d(const Geo& g, const RevBuffers& R, Ctrl* ctrl, const Dof* it, int nsteps, int di,
                          cudaStream_t st) {
  LKS_AXIS(design_ax, g, R, ctrl, it, nsteps, di, st);
}

#define LKS_AXIS_INST(T)                                                                                              \
  template void launch_couple_axis3d<T>(const Geo&, const Slots<T>&, Ctrl*, Dof*, const T*, const Moments*, void*, T*, \
                                        int, int, cudaStream_t);                                                      \
  template void launch_apply_axis3d<T>(const Geo&, const Slots<T>&, const Ctrl*, const Dof*, const T*, T*, int, int,   \
                                       cudaStream_t);                                                                 \
  template void launch_support_axis3d<T>(const Geo&, const Dof&, const T*, long long*, cudaStream_t);                   \
  template void launch_coef_axis3d<T>(const Geo&, const RevBuffers&, const Ctrl*, const Dof*, const T*, const T*, int, \
                                      int, int, cudaStream_t);                                                        \
  template void launch_design_axis3d<T>(const Geo&, const RevBuffers&, Ctrl*, const Dof*, int, int, cudaStream_t);
LKS_AXIS_INST(float)
LKS_AXIS_INST(double)

}  // namespace lks
