// All N_itr coupling iterations of a 2D step in one launch whose CTAs exchange their force and
// torque sums and the iterate through flagged words (the default in 2D; lks_body.cu holds the forms
// with one launch per iteration and with grid barriers).
//
// An iteration is short (a gather over the box's cells, three sums, the EOM), so its time is the
// latency of the sums' way through the chip (lks_flag.cuh: how they travel).
//
// Warps are dealt over the box round robin, so the design-free corners of a rotating body's box are
// shared evenly between the CTAs. The launch is cooperative (all CTAs resident).
//
// What bounds it: the gather's slowest warps and two trips through L2 per iteration. Forward march
// measured on GB300, N_itr launches (or grid barriers) per step -> this kernel, us per step: 512x256
// body of 128^2 60 -> 37; 1024x512, 256^2 (grid barriers before) 100 -> 56; FP64 80x40, 16^2 290 -> 58;
// FP64 600x100, 20^2 500 -> 67 (40 and 60 with the tiled stencils of lks_stencil_tile.cu).
#include <climits>

#include "lks_flag.cuh"

namespace lks {

namespace {

constexpr int NVC = 3;  // force x, y and torque

// Lanes per cell (LC) and the largest CTA. FP32: the gather is bound by issue, and uneven rows and each
// lane's setup cost more with every lane, while fewer leave the chip idle on small boxes: 2 lanes split a
// cell's candidate rows while that gives each thread one cell, 1 beyond (forward us per step, 2 lanes
// and 1: 512x256 with 128x128 design points 37.4 and 39.7; 1024x512 with 256x256 57.9 and 55.8). FP64
// issues one warp instruction per 64 cycles and scheduler, so 16 lanes take one to four candidates each and a small box spreads over all SMs.
constexpr int kLanes64 = 16;
template <typename T>
constexpr int max_threads() { return sizeof(T) == 4 ? 640 : 512; }

// Sums over the design points of one cell, e = xi_m - xi(cell) the offset from the cell's image in
// the design frame: phi, kappa, sum W e, sum W kappa e; then moved to the pivot (sum W r).
template <typename T>
__device__ __forceinline__ void to_pivot(T xb, T xc, T eb, T ec, T kb, T kc, Acc<T>& o) {
  o.wr[0] = fma_(xb, o.phi, eb);
  o.wr[1] = fma_(xc, o.phi, ec);
  o.kr[0] = fma_(xb, o.kap, kb);
  o.kr[1] = fma_(xc, o.kap, kc);
  o.wr[2] = o.kr[2] = T(0);
}

// FP32. Lane cl takes the candidate rows cl, cl + LC, ...; within a row the interval of candidates
// follows from the two support bounds (linear in the offset), widened, and the exact test decides.
// Cosine kernel: with the rotation scaled by pi/2 the offsets are the cosines' arguments; the factor
// 1/16 of the two weights is applied to the sums.
template <int LC, typename Visit = NoVisit>
__device__ __forceinline__ void gather2d(const Geo& g, const float* __restrict__ kref, const float (&d)[2], float cs,
                                         float sn, int cl, bool active, Acc<float>& o, Visit visit = Visit()) {
  const float S = (float)g.s, pad = 1e-3f, tiny = 1e-6f;
  const float xb = dot2(cs, d[0], sn, d[1]), xc = dot2(cs, d[1], -sn, d[0]);
  const float xib = xb + g.xicf[0], xic = xc + g.xicf[1];
  const float h = S * (fabsf(cs) + fabsf(sn));
  const int nx = g.nd[0];
  const int ib0 = max(0, (int)ceilf(xib - h)), ib1 = min(nx - 1, (int)floorf(xib + h));
  const int ic0 = max(0, (int)ceilf(xic - h)), ic1 = min(g.nd[1] - 1, (int)floorf(xic + h));
  float phi = 0.0f, kap = 0.0f, sb = 0.0f, sc = 0.0f, kb = 0.0f, kc = 0.0f;
  if (active && ib0 <= ib1) {
    const bool cosine = g.wk == W_COS4, ball = g.rad4 != INT_MAX;
    const float sw = cosine ? 1.57079632679f : 1.0f, Sw = cosine ? 3.14159265359f : 1.0f;
    const float cw = sw * cs, nw = sw * sn;
    const float ics = fabsf(cs) > tiny ? 1.0f / cs : 0.0f, isn = fabsf(sn) > tiny ? 1.0f / sn : 0.0f;
    for (int ic = ic0 + cl; ic <= ic1; ic += LC) {
      const float ec = (float)ic - xic;
      float lo = -1e6f, hi = 1e6f;
      if (ics != 0.0f) {
        const float e1 = (sn * ec - S) * ics, e2 = (sn * ec + S) * ics;
        lo = fmaxf(lo, fminf(e1, e2));
        hi = fminf(hi, fmaxf(e1, e2));
      } else if (fabsf(sn * ec) >= S + pad) {
        continue;
      }
      if (isn != 0.0f) {
        const float e1 = (-S - cs * ec) * isn, e2 = (S - cs * ec) * isn;
        lo = fmaxf(lo, fminf(e1, e2));
        hi = fminf(hi, fmaxf(e1, e2));
      } else if (fabsf(cs * ec) >= S + pad) {
        continue;
      }
      const int j0 = max(ib0, (int)ceilf(xib + lo - pad)), j1 = min(ib1, (int)floorf(xib + hi + pad));
      if (j0 > j1) continue;
      // a chord of the rotated support square is at most 4 sqrt 2 long: six candidates, all taken at
      // once (masked) so that their loads and cosines overlap
      const float* kr = kref + (long long)ic * nx;
      float kv[6];
#pragma unroll
      for (int j = 0; j < 6; ++j) kv[j] = __ldg(kr + min(j0 + j, j1));
      const float ob0 = mul_(-nw, ec), oc0 = mul_(cw, ec);
      float ps = 0.0f, pk = 0.0f;
#pragma unroll
      for (int j = 0; j < 6; ++j) {
        const int ib = j0 + j;
        const float eb = (float)ib - xib;
        const float ob = fmaf(cw, eb, ob0), oc = fmaf(nw, eb, oc0);
        bool ok = ib <= j1 && fabsf(ob) < Sw && fabsf(oc) < Sw;
        if (ball) ok = ok && dsq(ib, nx) + dsq(ic, g.nd[1]) <= g.rad4;
        float w = cosine ? mul_(1.0f + __cosf(ob), 1.0f + __cosf(oc)) : mul_(1.0f - fabsf(ob), 1.0f - fabsf(oc));
        w = ok ? w : 0.0f;
        if (ok) visit(ib + ic * nx);
        const float wk = mul_(w, kv[j]);
        ps += w;
        pk += wk;
        sb = fmaf(w, eb, sb);
        kb = fmaf(wk, eb, kb);
      }
      phi += ps;
      kap += pk;
      sc = fmaf(ps, ec, sc);
      kc = fmaf(pk, ec, kc);
    }
    const float f = cosine ? 0.0625f : 1.0f;
    phi = mul_(phi, f);
    kap = mul_(kap, f);
    sb = mul_(sb, f);
    sc = mul_(sc, f);
    kb = mul_(kb, f);
    kc = mul_(kc, f);
  }
#pragma unroll
  for (int off = 1; off < LC; off <<= 1) {
    phi += __shfl_xor_sync(0xffffffffu, phi, off);
    kap += __shfl_xor_sync(0xffffffffu, kap, off);
    sb += __shfl_xor_sync(0xffffffffu, sb, off);
    sc += __shfl_xor_sync(0xffffffffu, sc, off);
    kb += __shfl_xor_sync(0xffffffffu, kb, off);
    kc += __shfl_xor_sync(0xffffffffu, kc, off);
  }
  o.phi = phi;
  o.kap = kap;
  to_pivot(xb, xc, sb, sc, kb, kc, o);
}

// FP64: lane (cl >> 2, cl & 3) takes every fourth row and column of the candidates' bounding
// square; the test against the support is made in FP32 first (widened by more than its rounding),
// so FP64 instructions are spent on accepted candidates only. The six sums of the 16 lanes are
// combined by halving (each level exchanges half of the values: 8 additions, not 24).
template <int LC, typename Visit = NoVisit>
__device__ __forceinline__ void gather2d(const Geo& g, const double* __restrict__ kref, const double (&d)[2],
                                         double cs, double sn, int cl, bool active, Acc<double>& o, Visit visit = Visit()) {
  static_assert(LC == kLanes64, "a 4 x 4 pattern of lanes");
  const double S = (double)g.s;
  const double xb = dot2(cs, d[0], sn, d[1]), xc = dot2(cs, d[1], -sn, d[0]);
  const double xib = xb + g.xic[0], xic = xc + g.xic[1];
  const float csf = (float)cs, snf = (float)sn, pad = 2e-3f, Sp = (float)g.s + pad;
  const float xibf = (float)xib, xicf = (float)xic;
  const float h = Sp * (fabsf(csf) + fabsf(snf)) + pad;
  const int ib0 = max(0, (int)ceilf(xibf - h)), ic0 = max(0, (int)ceilf(xicf - h));
  const int ib1 = active ? min(g.nd[0] - 1, (int)floorf(xibf + h)) : -1;
  const int ic1 = min(g.nd[1] - 1, (int)floorf(xicf + h));
  double v[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = 0.0;
  for (int ib = ib0 + (cl >> 2); ib <= ib1; ib += 4)
    for (int ic = ic0 + (cl & 3); ic <= ic1; ic += 4) {
      const float ebf = (float)ib - xibf, ecf = (float)ic - xicf;
      if (fabsf(csf * ebf - snf * ecf) >= Sp || fabsf(snf * ebf + csf * ecf) >= Sp) continue;
      if (dsq(ib, g.nd[0]) + dsq(ic, g.nd[1]) > g.rad4) continue;
      const double eb = (double)ib - xib, ec = (double)ic - xic;
      const double ob = dot2(-sn, ec, cs, eb), oc = dot2(cs, ec, sn, eb);  // (the products of eb leave the loop)
      if (fabs(ob) >= S || fabs(oc) >= S) continue;
      visit(ib + ic * g.nd[0]);
      const double w = mul_(wfun(g.wk, ob), wfun(g.wk, oc)), wk = mul_(w, kref[ib + ic * g.nd[0]]);
      v[0] += w;
      v[1] += wk;
      v[2] = fma_(w, eb, v[2]);
      v[3] = fma_(w, ec, v[3]);
      v[4] = fma_(wk, eb, v[4]);
      v[5] = fma_(wk, ec, v[5]);
    }
  // halving over lane bits 3, 2, 1 (value index bits 2, 1, 0), then the pair of bit 0
  const bool b3 = cl & 8, b2 = cl & 4, b1 = cl & 2;
  double a[4], b[2], c;
#pragma unroll
  for (int i = 0; i < 4; ++i) a[i] = (b3 ? v[4 + i] : v[i]) + __shfl_xor_sync(0xffffffffu, b3 ? v[i] : v[4 + i], 8);
#pragma unroll
  for (int i = 0; i < 2; ++i) b[i] = (b2 ? a[2 + i] : a[i]) + __shfl_xor_sync(0xffffffffu, b2 ? a[i] : a[2 + i], 4);
  c = (b1 ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, b1 ? b[0] : b[1], 2);
  c += __shfl_xor_sync(0xffffffffu, c, 1);
  o.phi = __shfl_sync(0xffffffffu, c, 0, 16);
  o.kap = __shfl_sync(0xffffffffu, c, 2, 16);
  const double sb = __shfl_sync(0xffffffffu, c, 4, 16), sc = __shfl_sync(0xffffffffu, c, 6, 16);
  const double kb = __shfl_sync(0xffffffffu, c, 8, 16), kc = __shfl_sync(0xffffffffu, c, 10, 16);
  to_pivot(xb, xc, sb, sc, kb, kc, o);
}

// u^S of a cell from its sums; returns 1 / (1 + kappa).
template <typename T>
__device__ __forceinline__ T solid_velocity(const Pose<T, 2>& P, const Acc<T>& A, T (&us)[2]) {
  const T dwr[2] = {-dot2(P.sn, A.wr[0], P.cs, A.wr[1]), dot2(P.cs, A.wr[0], -P.sn, A.wr[1])};
#pragma unroll
  for (int a = 0; a < 2; ++a) us[a] = dot2(P.ug[a], A.phi, P.om, dwr[a]);
  return T(1) / (T(1) + A.kap);
}

template <typename T, int LC>
__global__ void __launch_bounds__(max_threads<T>(), 1)
    k_couple_flag(Geo g, Slots<T> S, Ctrl* ctrl, Dof* it, const T* __restrict__ kref, const Moments* __restrict__ mom,
                  void* words, T* __restrict__ boxstore, int nbox, int di) {
  using V = typename SumOf<T>::type;
  constexpr int CPW = 32 / LC;  // cells per warp
  constexpr int DW = (int)(sizeof(Dof) / sizeof(double));
  __shared__ V part[32 * NVC];
  __shared__ Dof sd[2];  // CTA 0: s(t-1), the current iterate
  __shared__ Pose<T, 2> pose;
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
    flag_root<T, 2, 2>(g, ctrl, row, mom, words, G, e0, (ctrl->sync_skip & 1) != 0, sd, gave_up);
    return;
  }
  if (tid == 0) pose.set(sd[0]);
  T* __restrict__ dst = slot_ptr(S, t, base);
  int lo[3];
  box_origin<2>(g, sd[0], lo[0], lo[1], lo[2]);
  T* bs = boxstore ? boxstore + (long long)((t - base - 1) % nbox) * g.box_cells * 2 : nullptr;
  const long long N = g.N;
  const int BC = (int)g.box_cells, W = G * nw, sub = lane / LC, cl = lane % LC;
  const int first = (warp * G + cta) * CPW;
  // position, grid index and u* of this thread's first cell stay in registers through the iterations
  struct Cell {
    int px, py, n;  // n < 0: outside the grid
  };
  auto cell_of = [&](int bl) {
    Cell c{0, 0, -1};
    if (bl < BC) {
      const int j1 = bl / g.B[0];
      c.px = lo[0] + bl - j1 * g.B[0];
      c.py = lo[1] + j1;
      long long n;
      if (cell_index<2>(g, c.px, c.py, 0, n)) c.n = (int)n;
    }
    return c;
  };
  const Cell cell0 = cell_of(first + sub);
  T ust0[2] = {T(0), T(0)};
  if (cell0.n >= 0) {
    ust0[0] = dst[N + cell0.n];
    ust0[1] = dst[2 * N + cell0.n];
  }
  __syncthreads();
  for (int k = 1; k <= K; ++k) {
    const bool last = k == K;
    const unsigned e = e0 + (unsigned)k;
    const Pose<T, 2> P = pose;
    T v[NVC] = {T(0), T(0), T(0)};
    for (int c0 = first; c0 < BC; c0 += W * CPW) {  // uniform per warp
      const int bl = c0 + sub;
      const Cell cc = c0 == first ? cell0 : cell_of(bl);
      const int n = cc.n;
      const T d[2] = {P.rel(0, cc.px), P.rel(1, cc.py)};
      Acc<T> A;
      gather2d<LC>(g, kref, d, P.cs, P.sn, cl, bl < BC, A);
      if (bl >= BC || cl != 0) continue;
      if (A.phi == T(0)) {  // no design point in reach: u = u*
        if (last && bs && n >= 0) {
          bs[bl] = c0 == first ? ust0[0] : dst[N + n];
          bs[g.box_cells + bl] = c0 == first ? ust0[1] : dst[2 * N + n];
        }
        continue;
      }
      if (n < 0 || forbidden<2>(g, cc.px, cc.py, 0)) atomicOr(&ctrl->status, ST_BODY_OUTSIDE);
      if (n < 0) continue;
      T L[3], u[2], us[2];
      rot<2>(P.cs, P.sn, A.kr, L);
      const T inv = solid_velocity(P, A, us);
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        const T ustar = c0 == first ? ust0[a] : dst[(a + 1) * N + n];
        u[a] = brinkman(ustar, A.kap, us[a], inv);
        v[a] += A.kap * u[a];
        if (last) {
          if (bs) bs[a * g.box_cells + bl] = ustar;
          dst[(a + 1) * N + n] = u[a];
        }
      }
      v[2] += L[0] * u[1] - L[1] * u[0];
    }
    __syncwarp();
    // the lanes with cl = 0 hold the values: lane cl takes component cl of its cell (two components a
    // lane in FP32), so the trees over the cells run side by side
    constexpr int per = (NVC + LC - 1) / LC;
#pragma unroll
    for (int q = 0; q < per; ++q) {
      T x = T(0);
#pragma unroll
      for (int i = 0; i < NVC; ++i) {
        const T y = __shfl_sync(0xffffffffu, v[i], lane - cl);
        if (i == cl + q * LC) x = y;
      }
      V s;
      s.set(x);
      warp_total<LC>(s);
      if (lane + q * LC < NVC && lane < LC) part[warp * NVC + lane + q * LC] = s;
    }
    __syncthreads();
    flag_exchange<T, 2>(words, e, cta, G, last, &ctrl->status, part, pose, gave_up);
    if (last) return;
    __syncthreads();
    if (gave_up) return;
  }
}

// Recompute of one step's Brinkman update from the stored iterate s^(K-1), by the forward's gather with
// its lanes, so that the recomputed state is the forward's to the bit (k_apply of lks_body.cu sums a cell's
// points in another order and goes with k_couple).
constexpr int kApplyThreads = 128;
template <typename T, int LC>
__global__ void __launch_bounds__(kApplyThreads) k_apply_flag(Geo g, Slots<T> S, const Ctrl* ctrl, const Dof* it,
                                                              const T* __restrict__ kref, T* __restrict__ boxstore,
                                                              int nbox, int di) {
  const int t = ctrl->t0 + di, base = ctrl->base, K = g.K;
  const Dof* row = it + (long long)(t - 1) * (K + 1);
  Pose<T, 2> P;
  P.set(row[K - 1]);
  T* __restrict__ dst = slot_ptr(S, t, base);
  T* bs = boxstore + (long long)((t - base - 1) % nbox) * g.box_cells * 2;
  int lo[3];
  box_origin<2>(g, row[0], lo[0], lo[1], lo[2]);
  const long long N = g.N;
  const unsigned q = blockIdx.x * (unsigned)kApplyThreads + threadIdx.x;
  const int bl = (int)(q / LC), cl = (int)(q % LC);
  const bool in = bl < (int)g.box_cells;
  const int j1 = bl / g.B[0], px = lo[0] + bl - j1 * g.B[0], py = lo[1] + j1;
  long long n = 0;
  const bool ing = in && cell_index<2>(g, px, py, 0, n);
  T ust[2] = {T(0), T(0)};
  if (ing) {
    ust[0] = dst[N + n];
    ust[1] = dst[2 * N + n];
  }
  const T d[2] = {P.rel(0, px), P.rel(1, py)};
  Acc<T> A;
  gather2d<LC>(g, kref, d, P.cs, P.sn, cl, in, A);
  if (!ing || cl != 0) return;
  T us[2];
  const T inv = solid_velocity(P, A, us);
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    bs[a * g.box_cells + bl] = ust[a];
    if (A.phi != T(0)) dst[(a + 1) * N + n] = brinkman(ust[a], A.kap, us[a], inv);
  }
}

// The box of the iterate s, gathered as k_couple_flag does, with the accepted index sets as out[box cell][5].
template <typename T, int LC>
__global__ void __launch_bounds__(kApplyThreads) k_support_flag(Geo g, Dof s, const T* __restrict__ kref,
                                                                long long* __restrict__ out) {
  Pose<T, 2> P;
  P.set(s);
  int lo[3];
  box_origin<2>(g, s, lo[0], lo[1], lo[2]);
  const unsigned q = blockIdx.x * (unsigned)kApplyThreads + threadIdx.x;
  const int bl = (int)(q / LC), cl = (int)(q % LC), j1 = bl / g.B[0];
  const T d[2] = {P.rel(0, lo[0] + bl - j1 * g.B[0]), P.rel(1, lo[1] + j1)};
  SetStats st;
  Acc<T> A;
  gather2d<LC>(g, kref, d, P.cs, P.sn, cl, bl < (int)g.box_cells, A, StatVisit{&st});
  st.lanes<LC>();
  if (bl < (int)g.box_cells && cl == 0) st.store(out, bl);
}

// CTAs and threads of the kernel with LC lanes; *passes: cells per thread.
template <typename T, int LC>
int flag_shape(const Geo& g, int* threads, long long* passes) {
  int dev = 0, sms = 0, per_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 2) return 0;
  const long long want = g.box_cells * LC;
  // one CTA per SM, one SM for CTA 0: as few publishers as fill the chip, each with the threads its
  // share needs
  long long nt = (want + sms - 2) / (sms - 1);
  *passes = (nt + max_threads<T>() - 1) / max_threads<T>();
  nt = (nt + 31) / 32 * 32;
  if (nt < 128) nt = 128;  // a warp per scheduler; three sum, the fourth waits for the iterate
  if (nt > max_threads<T>()) nt = max_threads<T>();
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_couple_flag<T, LC>, (int)nt, 0) != cudaSuccess) return 0;
  if (per_sm < 1) return 0;
  const long long ctas = (want + nt - 1) / nt + 1;
  *threads = (int)nt;
  const long long cap = sms < kFlagMaxCtas ? sms : kFlagMaxCtas;
  return (int)(ctas < cap ? ctas : cap);
}

}  // namespace

void setup_couple_flag(Geo* g, bool fp64) {
  g->flag_ctas = g->flag_threads = 0;
  if (g->dim == 3) {
    setup_couple_axis3d(g, fp64);
  } else if (g->box_cells < (1LL << 27) && g->N < (1LL << 31)) {
    long long passes = 0;
    g->flag_lanes = fp64 ? kLanes64 : 2;
    g->flag_ctas = fp64 ? flag_shape<double, kLanes64>(*g, &g->flag_threads, &passes)
                        : flag_shape<float, 2>(*g, &g->flag_threads, &passes);
    if (!fp64 && passes > 1) {
      g->flag_lanes = 1;
      g->flag_ctas = flag_shape<float, 1>(*g, &g->flag_threads, &passes);
    }
  }
  cudaGetLastError();  // a query that failed leaves the other forms in use
}

// The sums of the CTAs with cells (up to four components), the iterates of both parities and the hook's.
size_t couple_flag_bytes(int ctas) { return 2 * (size_t)(ctas - 1) * 4 * sizeof(Words) + 3 * kPoseWords * 8; }

template <typename T>
void launch_couple_flag(const Geo& g, const Slots<T>& S, Ctrl* ctrl, Dof* it, const T* kref, const Moments* mom,
                        void* words, T* boxstore, int nbox, int di, cudaStream_t st) {
  if (g.dim == 3) return launch_couple_axis3d<T>(g, S, ctrl, it, kref, mom, words, boxstore, nbox, di, st);
  auto run = [&](auto kernel) {
    launch_coop(kernel, dim3((unsigned)g.flag_ctas), dim3((unsigned)g.flag_threads), 0, st, g, S, ctrl, it, kref, mom,
                words, boxstore, nbox, di);
  };
  if constexpr (sizeof(T) == 8)
    run(k_couple_flag<double, kLanes64>);
  else if (g.flag_lanes == 1)
    run(k_couple_flag<float, 1>);
  else
    run(k_couple_flag<float, 2>);
}

namespace {
unsigned apply_ctas(const Geo& g, int lanes) {
  return (unsigned)((g.box_cells * lanes + kApplyThreads - 1) / kApplyThreads);
}
}  // namespace

template <typename T>
void launch_apply_flag2d(const Geo& g, const Slots<T>& S, const Ctrl* ctrl, const Dof* it, const T* kref, T* boxstore,
                         int nbox, int di, cudaStream_t st) {
  auto run = [&](auto kernel, int lanes) {
    launch(kernel, dim3(apply_ctas(g, lanes)), kApplyThreads, 0, st, g, S, ctrl, it, kref, boxstore, nbox, di);
  };
  if constexpr (sizeof(T) == 8)
    run(k_apply_flag<double, kLanes64>, kLanes64);
  else if (g.fwd_form == 1)
    run(k_apply_flag<float, 1>, 1);
  else
    run(k_apply_flag<float, 2>, 2);
}

template <typename T>
void launch_support_flag2d(const Geo& g, const Dof& s, const T* kref, long long* out, cudaStream_t st) {
  auto run = [&](auto kernel, int lanes) { launch(kernel, dim3(apply_ctas(g, lanes)), kApplyThreads, 0, st, g, s, kref, out); };
  if constexpr (sizeof(T) == 8)
    run(k_support_flag<double, kLanes64>, kLanes64);
  else if (g.flag_lanes == 1)
    run(k_support_flag<float, 1>, 1);
  else
    run(k_support_flag<float, 2>, 2);
}

template void launch_support_flag2d<float>(const Geo&, const Dof&, const float*, long long*, cudaStream_t);
template void launch_support_flag2d<double>(const Geo&, const Dof&, const double*, long long*, cudaStream_t);
template void launch_apply_flag2d<float>(const Geo&, const Slots<float>&, const Ctrl*, const Dof*, const float*, float*,
                                         int, int, cudaStream_t);
template void launch_apply_flag2d<double>(const Geo&, const Slots<double>&, const Ctrl*, const Dof*, const double*,
                                          double*, int, int, cudaStream_t);
template void launch_couple_flag<float>(const Geo&, const Slots<float>&, Ctrl*, Dof*, const float*, const Moments*,
                                        void*, float*, int, int, cudaStream_t);
template void launch_couple_flag<double>(const Geo&, const Slots<double>&, Ctrl*, Dof*, const double*, const Moments*,
                                         void*, double*, int, int, cudaStream_t);

}  // namespace lks
