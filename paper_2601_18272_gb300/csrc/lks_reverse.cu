// Reverse of one step's N_itr coupling iterations about one rotation axis, without the chain of
// kernels per iteration (lks_body.cu holds the per-iteration form, kept for free rotation).
//
// The reverse of iteration k takes dJ/dF, dJ/dT (D + 1 numbers, lam^k) and gives dJ/ds^(k-1), from
// which the EOM reverse makes lam^(k-1). Everything else it needs (the pose s^(k-1), kappa_n, u^S_n,
// u^(k)_n) is known from the forward, and the map is linear, so
//   dJ/ds^(k-1) = M_k lam^k (+ c for k = N_itr, where the adjoint state lam_n(t) enters),
// with an 8 x (D + 1) matrix M_k that depends on the forward only. The sums over the design points
// are taken on the cell side: with Phi = sum W, kap = sum W kappa, P = sum W l, L = sum W kappa l
// (l = R r_m, in the plane of rotation) and the same sums with dW/dx, the derivatives of a cell's
// kappa_n, u^S_n and L_n with respect to x^G and theta are closed forms, so no pass over the design
// points' windows is needed for them.
//
//   k_rev_coef    box cells x iterations x steps of a chunk: the sums above, the per-cell planes the
//                 step needs later, per-CTA partials of M_k (independent of the reverse sweep, so
//                 all iterations of several steps run in one launch)
//   k_rev_mat     one CTA per (step, iteration): M_k in FP64 with the closed design-side terms, and
//                 the map lam^k -> lam^(k-1)
//   k_rev_const   box cells: c = sum_n lam_n(t) . du_n/ds^(N_itr-1), per-CTA partials
//   k_rev_apply   every CTA: the sum of c and the chain lam^N_itr -> .. -> lam^1 (FP64, a few fused
//                 multiply-adds); box cells: dJ/du* and dJ/dkappa_n of every iteration; one more CTA
//                 carries the direct EOM part dJ/ds(t-1)
//   k_rev_design  design points x steps of a chunk: dJ/dkappa^ref, from the support windows of
//                 u^(k)_n and dJ/dkappa_n (D + 1 values per window cell)
//   k_rev_dksum   dJ/dkappa^ref summed over the splits of k_rev_design, in a fixed order
//
// What it replaces: 3 N_itr dependent launches a step (cell, design and one-CTA finish kernel per
// iteration), bound by their latency on 2D boxes (about 5 us each for 35 k cells) and in FP64 by the
// few warps a small box gives each launch. Only k_rev_const, k_rev_apply and the transposed stencil
// are left in a step's chain; the rest runs over whole chunks of steps, on a branch of its own beside the
// chain (lks_api.cu: that took the gradients below by another 2 % (2D, small body) to 8 % (3D)). Gradients measured on GB300,
// before -> after: 512x256 / 128^2, 200 steps 30.2 -> 21.1 ms; 1024x512 / 256^2, 100 steps 30.2 -> 22.3
// ms; 80x40 / 16^2 FP64, 400 steps 256 -> 135 ms; 128x64x64 / 48^3, 40 steps 26.3 -> 21.9 ms.
#include <algorithm>
#include <climits>

#include "lks_reverse.cuh"

namespace lks {

namespace {

template <typename T, int D, int AX>
__device__ __forceinline__ void gather_moments(const Geo& g, const T* __restrict__ kref, const T (&d)[3], T cs, T sn,
                                               Moments1<T>& o) {
  constexpr int b = Axes<AX>::B, c = Axes<AX>::C, ax = Axes<AX>::A;
  const T S = (T)g.s;
#pragma unroll
  for (int e = 0; e < 4; ++e) o.phi[e] = o.kap[e] = o.Pb[e] = o.Pc[e] = o.Lb[e] = o.Lc[e] = T(0);
  o.qPb = o.qPc = o.qLb = o.qLc = T(0);
  const T xib = cs * d[b] + sn * d[c] + pivot<T>(g, b);
  const T xic = -sn * d[b] + cs * d[c] + pivot<T>(g, c);
  // candidate rows and, per row, the interval of candidates: bounds in FP32 with the support widened
  // by more than their rounding, so that no design point is lost; the exact test is in T
  const float csf = (float)cs, snf = (float)sn, pad = 2e-3f, Sp = (float)g.s + pad;
  const float xibf = (float)xib, xicf = (float)xic;
  const float h = Sp * (fabsf(csf) + fabsf(snf)) + pad;
  const int ib0 = max(0, (int)ceilf(xibf - h)), ib1 = min(g.nd[b] - 1, (int)floorf(xibf + h));
  const int ic0 = max(0, (int)ceilf(xicf - h)), ic1 = min(g.nd[c] - 1, (int)floorf(xicf + h));
  if (ib1 < ib0 || ic1 < ic0) return;
  T wa[4], dwa[4];
  int qa[4], ia0 = 0;
  if (D == 3) {
    const T xia = d[ax] + pivot<T>(g, ax);
    const int fa = (int)floor(xia);
    ia0 = max(0, fa - g.s + 1);
    const int ia1 = min(g.nd[ax] - 1, fa + g.s);
    bool any = false;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int ia = ia0 + q;
      const T oa = xia - (T)ia;
      wa[q] = dwa[q] = T(0);
      qa[q] = INT_MAX;
      if (ia <= ia1 && fabs(oa) < S) {
        w_dw(g.wk, oa, &wa[q], &dwa[q]);
        qa[q] = dsq(ia, g.nd[ax]);
        any = true;
      }
    }
    if (!any) return;
  }
  const int sx = 1, sy = g.nd[0], sz = g.nd[0] * g.nd[1];
  const int sb = (b == 0) ? sx : (b == 1 ? sy : sz);
  const int sc = (c == 0) ? sx : (c == 1 ? sy : sz);
  const int sa = (ax == 0) ? sx : (ax == 1 ? sy : sz);
  const float tiny = 1e-6f;
  const float ics = fabsf(csf) > tiny ? 1.0f / csf : 0.0f, isn = fabsf(snf) > tiny ? 1.0f / snf : 0.0f;
  for (int ib = ib0; ib <= ib1; ++ib) {
    const float ebf = (float)ib - xibf;
    float elo = -1e6f, ehi = 1e6f;
    if (isn != 0.0f) {
      const float e1 = (csf * ebf - Sp) * isn, e2 = (csf * ebf + Sp) * isn;
      elo = fmaxf(elo, fminf(e1, e2));
      ehi = fminf(ehi, fmaxf(e1, e2));
    } else if (fabsf(csf * ebf) >= Sp) {
      continue;
    }
    if (ics != 0.0f) {
      const float e1 = (-Sp - snf * ebf) * ics, e2 = (Sp - snf * ebf) * ics;
      elo = fmaxf(elo, fminf(e1, e2));
      ehi = fminf(ehi, fmaxf(e1, e2));
    } else if (fabsf(snf * ebf) >= Sp) {
      continue;
    }
    const int jc0 = max(ic0, (int)ceilf(xicf + elo - pad)), jc1 = min(ic1, (int)floorf(xicf + ehi + pad));
    const T eb = (T)ib - xib;
    const int qb = dsq(ib, g.nd[b]);
    for (int ic = jc0; ic <= jc1; ++ic) {
      const T ec = (T)ic - xic;
      const T lb0 = cs * eb - sn * ec, lc0 = sn * eb + cs * ec;  // x^ref - x_n in the plane
      if (fabs(lb0) >= S || fabs(lc0) >= S) continue;
      const int qbc = qb + dsq(ic, g.nd[c]);
      if (qbc > g.rad4) continue;
      T wb, dwb, wc, dwc;
      w_dw(g.wk, -lb0, &wb, &dwb);
      w_dw(g.wk, -lc0, &wc, &dwc);
      const T lb = lb0 + d[b], lc = lc0 + d[c];  // R r_m
      const int m2 = ib * sb + ic * sc;
      T s0 = T(1), s1 = T(0), k0, k1 = T(0);
      if (D == 2) {
        k0 = kref[m2];
      } else {
        s0 = k0 = T(0);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (qa[q] > g.rad4 - qbc) continue;
          const T kq = kref[m2 + (ia0 + q) * sa];
          s0 += wa[q];
          s1 += dwa[q];
          k0 += wa[q] * kq;
          k1 += dwa[q] * kq;
        }
      }
      const T w2 = wb * wc, wB = dwb * wc, wC = wb * dwc;
      auto add = [&](int e, T A, T Ak) {
        o.phi[e] += A;
        o.kap[e] += Ak;
        o.Pb[e] += A * lb;
        o.Pc[e] += A * lc;
        o.Lb[e] += Ak * lb;
        o.Lc[e] += Ak * lc;
      };
      add(0, w2 * s0, w2 * k0);
      add(1 + b, wB * s0, wB * k0);
      add(1 + c, wC * s0, wC * k0);
      if (D == 3) add(1 + ax, w2 * s1, w2 * k1);
      const T rt = wB * lc - wC * lb, rs = rt * s0, rk = rt * k0;
      o.qPb += rs * lb;
      o.qPc += rs * lc;
      o.qLb += rk * lb;
      o.qLc += rk * lc;
    }
  }
}

template <typename T, int D, int AX>
__global__ void __launch_bounds__(kRevThreads) k_rev_coef(Geo g, const Ctrl* ctrl, const Dof* it,
                                                          const T* __restrict__ kref, const T* __restrict__ boxstore,
                                                          int nbox, T* __restrict__ slabs, long long slab,
                                                          typename Partial<T>::type* __restrict__ mpart, int di) {
  using RP = RevPlanes<D>;
  using RS = RevSums<D>;
  extern __shared__ __align__(16) unsigned char rev_smem[];
  const int K = g.K, k = (int)blockIdx.y + 1, i = blockIdx.z;
  const int t = rev_step(ctrl, di, i), base = ctrl->base;
  const Dof* row = it + (long long)(t - 1) * (K + 1);
  const Dof& sk = row[k - 1];
  const long long BC = g.box_cells;
  const long long bl = blockIdx.x * (long long)kRevThreads + threadIdx.x;
  T v[RS::N];
#pragma unroll
  for (int q = 0; q < RS::N; ++q) v[q] = T(0);
  if (bl < BC) {
    int lo[3];
    box_origin<D>(g, row[0], lo[0], lo[1], lo[2]);
    const unsigned ub = (unsigned)bl, r = ub / (unsigned)g.B[0];
    const int j0 = (int)(ub - r * (unsigned)g.B[0]);
    const int j1 = (int)(D == 3 ? r % (unsigned)g.B[1] : r), j2 = (int)(D == 3 ? r / (unsigned)g.B[1] : 0);
    const int px = lo[0] + j0, py = lo[1] + j1, pz = lo[2] + j2;
    long long n;
    const bool ing = cell_index<D>(g, px, py, pz, n);
    const DofView<T> V(sk);
    const T d[3] = {V.rel(0, px), V.rel(1, py), D == 3 ? V.rel(2, pz) : T(0)};
    Moments1<T> A;
    if (ing) {
      gather_moments<T, D, AX>(g, kref, d, V.cs, V.sn, A);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) A.phi[e] = A.kap[e] = A.Pb[e] = A.Pc[e] = A.Lb[e] = A.Lc[e] = T(0);
      A.qPb = A.qPc = A.qLb = A.qLc = T(0);
    }
    const T* bs = boxstore + (long long)((t - base - 1) % nbox) * BC * D;
    rev_cell<T, D, AX>(g, V, A, ing, bs, bl, slabs + (long long)i * slab + bl, k, v);
  }
  row_sums<RS::N>(v, reinterpret_cast<T*>(rev_smem),
                  mpart + (((long long)i * K + (k - 1)) * gridDim.x + blockIdx.x) * RS::N);
}

// M_k (rows the 8 DOFs, columns lam_F[3], lam_T) with the design-side closed forms of F and T
// (F -= K0 u^G + omega R'K1, T -= RK1 x u^G + omega K2p), and G = the EOM reverse of iteration k - 1
// applied to it: lam^(k-1) = G lam^k.
struct RevMat {
  double M[8][4], G[4][4];
};

template <typename T, int D, int AX>
__global__ void __launch_bounds__(kRevThreads) k_rev_mat(Geo g, const Ctrl* ctrl, const Dof* it,
                                                         const Moments* __restrict__ mom,
                                                         const typename Partial<T>::type* __restrict__ mpart,
                                                         int nparts, RevMat* __restrict__ mats, int di) {
  using RS = RevSums<D>;
  constexpr int b = Axes<AX>::B, c = Axes<AX>::C;
  __shared__ double s[RS::N], M[8][4];
  const int K = g.K, k = (int)blockIdx.x + 1, i = blockIdx.y, tid = threadIdx.x;
  if ((tid & ~31) < RS::N * 8) {
    const int rw = min(tid >> 3, RS::N - 1);
    const double a = part_sum(mpart + ((long long)i * K + (k - 1)) * nparts * RS::N, nparts, RS::N, rw, tid & 7);
    if ((tid >> 3) < RS::N && (tid & 7) == 0) s[tid >> 3] = a;
  }
  if (tid < 32) (&M[0][0])[tid] = 0.0;
  __syncthreads();
  if (tid == 0) {
    const Dof& sk = it[(long long)(rev_step(ctrl, di, i) - 1) * (K + 1) + (k - 1)];
    const double cs = sk.cs, sn = sk.sn, om = sk.s[7];
    const double K1[3] = {mom->K1[0], mom->K1[1], mom->K1[2]};
    double r[3], dr[3];
    rot<AX>(cs, sn, K1, r);
    drot<AX>(cs, sn, K1, dr);
    const double K0 = mom->K0;
    const double ug[3] = {sk.s[3], sk.s[4], sk.s[5]};
    for (int e = 0; e <= D; ++e) {
      const int j = e < D ? e : 6;
      for (int a = 0; a < D; ++a) M[j][a] = s[e * (D + 1) + a];
      M[j][3] = s[e * (D + 1) + D];
    }
    M[6][b] += om * r[b];
    M[6][c] += om * r[c];
    M[6][3] -= dr[b] * ug[c] - dr[c] * ug[b];
    for (int a = 0; a < D; ++a) M[3 + a][a] = s[RS::uF] - K0;
    M[3 + b][3] = s[RS::uT] + r[c];
    M[3 + c][3] = s[RS::uT + 1] - r[b];
    M[7][b] = s[RS::oF] - dr[b];
    M[7][c] = s[RS::oF + 1] - dr[c];
    M[7][3] = s[RS::oT] - mom->K2p;
  }
  __syncthreads();
  RevMat& o = mats[(long long)i * K + (k - 1)];
  if (tid < 32) (&o.M[0][0])[tid] = (&M[0][0])[tid];
  if (tid < 16) {
    const int a = tid >> 2, q = tid & 3;
    double v = 0.0;
    if (a < 3) {
      if (a < D && (g.dof_mask & (1 << a))) v = (M[3 + a][q] + M[a][q]) * g.inv_mass;
    } else if (g.dof_mask & DOF_ROT) {
      v = (M[7][q] + M[6][q]) * g.inv_inertia;
    }
    o.G[a][q] = v;
  }
}

// Box cell bl of the box at lo: its grid index; false outside a non-periodic axis.
template <int D>
__device__ __forceinline__ bool box_cell(const Geo& g, const int (&lo)[3], long long bl, long long& n) {
  const unsigned ub = (unsigned)bl, r = ub / (unsigned)g.B[0];
  const int j0 = (int)(ub - r * (unsigned)g.B[0]);
  const int j1 = (int)(D == 3 ? r % (unsigned)g.B[1] : r), j2 = (int)(D == 3 ? r / (unsigned)g.B[1] : 0);
  return cell_index<D>(g, lo[0] + j0, lo[1] + j1, lo[2] + j2, n);
}

// MANY: boxes of more cells than the launch has threads. A thread's cells are then summed as pairs in FP32, whose
// loads go out several cells at a time (one after the other took 25 % longer for the step's two kernels on
// 5 million cells); FP64 adds every term to the sums directly (forming a cell's terms first: 31 -> 38 us a
// step for the two kernels on 93,000 cells).
template <typename T, int D, int AX, bool MANY>
__global__ void __launch_bounds__(kRevThreads) k_rev_const(Geo g, const Ctrl* ctrl, const Dof* it,
                                                           const T* __restrict__ slabs, long long slab, const T* Lb,
                                                           long long lstride,
                                                           typename Partial<T>::type* __restrict__ cpart, int di,
                                                           int i) {
  using RP = RevPlanes<D>;
  constexpr int b = Axes<AX>::B, c = Axes<AX>::C, NC = rev_nconst<D>();
  extern __shared__ __align__(16) unsigned char rev_smem[];
  const int K = g.K, t = rev_step(ctrl, di, i);
  const T* __restrict__ Lcur = Lb + (long long)(t & 1) * lstride;
  const long long BC = g.box_cells, N = g.N;
  int lo[3];
  box_origin<D>(g, it[(long long)(t - 1) * (K + 1)], lo[0], lo[1], lo[2]);
  const T* P0 = slabs + (long long)i * slab + (long long)K * RP::per_itr * BC;
  // adds the cell's terms (zero off the box and the grid)
  auto cell = [&](long long bl, T (&v)[NC]) {
    long long n = 0;
    const bool in = bl < BC && box_cell<D>(g, lo, bl, n);
    const T* P = P0 + (in ? bl : 0);
    if (!in) n = 0;
    T lam[3];
    const T bphi = P[RP::bphi * BC];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const T l = Lcur[(a + 1) * N + n];
      lam[a] = in ? l : T(0);
      v[D + 1 + a] += lam[a] * bphi;
    }
#pragma unroll
    for (int e = 0; e <= D; ++e)
#pragma unroll
      for (int a = 0; a < D; ++a) v[e] += lam[a] * P[(RP::Q + e * D + a) * BC];
    v[2 * D + 1] += lam[c] * P[RP::bP * BC] - lam[b] * P[(RP::bP + 1) * BC];
  };
  const long long stride = (long long)gridDim.x * kRevThreads;
  long long bl = blockIdx.x * (long long)kRevThreads + threadIdx.x;
  auto* out = cpart + blockIdx.x * NC;
  if constexpr (!MANY || sizeof(T) == 8) {
    T v[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) v[q] = T(0);
    if constexpr (!MANY) {
      cell(bl, v);
    } else {
#pragma unroll 4
      for (; bl < BC; bl += stride) cell(bl, v);
    }
    row_sums<NC>(v, reinterpret_cast<T*>(rev_smem), out);
  } else {
    constexpr int U = D == 2 ? 4 : 2;
    typename SumOf<T>::type v[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) v[q].zero();
    for (; bl < BC; bl += U * stride) {
      T x[U][NC];
#pragma unroll
      for (int u = 0; u < U; ++u) {
#pragma unroll
        for (int q = 0; q < NC; ++q) x[u][q] = T(0);
        cell(bl + u * stride, x[u]);
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int q = 0; q < NC; q += 2) run_add2(v[q], v[q + 1], x[u][q], x[u][q + 1]);
    }
    row_sums<NC>(v, reinterpret_cast<T*>(rev_smem), out);
  }
}

template <typename T, int D, int AX>
__global__ void __launch_bounds__(kRevThreads) k_rev_apply(Geo g, Ctrl* ctrl, const Dof* it, T* __restrict__ slabs,
                                                           long long slab, T* Lb, long long lstride,
                                                           const typename Partial<T>::type* __restrict__ cpart,
                                                           int nparts, const RevMat* __restrict__ mats,
                                                           T* __restrict__ lamh, int di, int i) {
  using RP = RevPlanes<D>;
  constexpr int b = Axes<AX>::B, c = Axes<AX>::C, NC = rev_nconst<D>();
  extern __shared__ __align__(16) unsigned char rev_smem[];
  __shared__ double cc[8];  // c by DOF
  const int K = g.K, t = rev_step(ctrl, di, i), tid = threadIdx.x;
  RevMat* mat = reinterpret_cast<RevMat*>(rev_smem);   // the step's matrices [K]
  double* lamd = reinterpret_cast<double*>(mat + K);   // lam^k [K][4]
  T* lamt = reinterpret_cast<T*>(lamd + 4 * K);        // the same in the field type
  for (int q = tid; q < K * (int)(sizeof(RevMat) / sizeof(double)); q += kRevThreads)
    reinterpret_cast<double*>(mat)[q] = reinterpret_cast<const double*>(mats + (long long)i * K)[q];
  const double* lin = ctrl->rev_lam[t & 1];  // dJ/ds(t) direct part [8], lam^K [4]
  if (tid < 8) cc[tid] = 0.0;
  __syncthreads();
  if ((tid & ~31) < NC * 8) {
    const int rw = min(tid >> 3, NC - 1);
    const double a = part_sum(cpart, nparts, NC, rw, tid & 7);
    if ((tid >> 3) < NC && (tid & 7) == 0) {
      const int q = tid >> 3;
      cc[q < D ? q : (q == D ? 6 : (q < 2 * D + 1 ? 3 + q - (D + 1) : 7))] = a;
    }
  }
  __syncthreads();
  if (tid < 32) {  // the chain, one lane per component
    const int a = tid & 3;
    double x = lin[8 + a], gc = 0.0;
    if (a < 3) {
      if (a < D && (g.dof_mask & (1 << a))) gc = (cc[3 + a] + cc[a]) * g.inv_mass;
    } else if (g.dof_mask & DOF_ROT) {
      gc = (cc[7] + cc[6]) * g.inv_inertia;
    }
    for (int k = K; k >= 1; --k) {
      if (tid < 4) {
        lamd[(k - 1) * 4 + a] = x;
        lamt[(k - 1) * 4 + a] = (T)x;
      }
      if (k == 1) break;
      const double* G = mat[k - 1].G[a];
      double y = k == K ? gc : 0.0;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const double xq = __shfl_sync(0xffffffffu, x, q);
        if (q < D || q == 3) y += G[q] * xq;
      }
      x = y;
    }
  }
  __syncthreads();
  if (blockIdx.x == gridDim.x - 1) {  // the direct EOM part: one lane per DOF
    for (int q = tid; q < 4 * K; q += kRevThreads) lamh[(long long)i * 4 * K + q] = lamt[q];
    if (tid < 32) {
      const int j = tid & 7, a = j % 3;
      const bool tr = j < 6;
      const bool fr = tr ? (a < D && (g.dof_mask & (1 << a))) : (g.dof_mask & DOF_ROT) != 0;
      double lp = lin[j], ls = 0.0;
      for (int k = K; k >= 1; --k) {
        ls = k == K ? cc[j] : 0.0;
        const double* Mj = mat[k - 1].M[j];
#pragma unroll
        for (int q = 0; q < 4; ++q) ls += Mj[q] * lamd[(k - 1) * 4 + q];
        if (k == 1) break;
        // position rows add their own, velocity rows also the position's if the DOF is free
        const double lx = __shfl_sync(0xffffffffu, ls, j == 7 ? 6 : (tr && j >= 3 ? j - 3 : j));
        lp += ls;
        if (fr && (j == 7 || (tr && j >= 3))) lp += lx;
      }
      const double full = lp + ls;  // dJ/ds(t-1)
      if (tid < 8) ctrl->lam_s0[j] = full;
      const double lx = __shfl_sync(0xffffffffu, full, j == 7 ? 6 : (tr && j >= 3 ? j - 3 : j));
      double* lout = ctrl->rev_lam[(t - 1) & 1];
      if (tid < 8) {
        const bool vel = j == 7 || (tr && j >= 3);
        lout[j] = full + (vel && fr ? lx : 0.0);
        if (vel) lout[8 + (j == 7 ? 3 : a)] = fr ? (full + lx) * (j == 7 ? g.inv_inertia : g.inv_mass) : 0.0;
      }
    }
    return;
  }
  T* __restrict__ Lcur = Lb + (long long)(t & 1) * lstride;
  const long long BC = g.box_cells, N = g.N;
  int lo[3];
  box_origin<D>(g, it[(long long)(t - 1) * (K + 1)], lo[0], lo[1], lo[2]);
  for (long long bl = blockIdx.x * (long long)kRevThreads + tid; bl < BC;
       bl += (long long)(gridDim.x - 1) * kRevThreads) {
    long long n;
    if (!box_cell<D>(g, lo, bl, n)) continue;
    T* P = slabs + (long long)i * slab + bl;
    const T* Pc = P + (long long)K * RP::per_itr * BC;
    T acc[3] = {T(0), T(0), T(0)}, lk = T(0);
    const T inv = Pc[RP::inv * BC];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const T lam = Lcur[(a + 1) * N + n];
      acc[a] = lam * inv;
      lk += lam * Pc[(RP::del + a) * BC];
    }
    for (int k = K; k >= 1; --k) {
      T* Pk = P + (long long)(k - 1) * RP::per_itr * BC;
      const T* l = lamt + (k - 1) * 4;
      const T beta = Pk[RP::beta * BC], lT = l[3];
      lk += lT * Pk[RP::eps * BC];
#pragma unroll
      for (int a = 0; a < D; ++a) {
        acc[a] += beta * l[a];
        lk += l[a] * Pk[(RP::kd + a) * BC];
      }
      acc[b] -= lT * Pk[(RP::iL + 1) * BC];
      acc[c] += lT * Pk[RP::iL * BC];
      Pk[RP::eps * BC] = lk;
      lk = T(0);
    }
#pragma unroll
    for (int a = 0; a < D; ++a) Lcur[(a + 1) * N + n] = acc[a];
  }
}

// 2D: LN lanes per design point, one row of the window each; split blockIdx.y takes the chunk's steps
// blockIdx.y, blockIdx.y + gridDim.y, ... and keeps its own dJ/dkappa^ref. (3D: k_design_axis3d.)
template <typename T>
__global__ void __launch_bounds__(kRevThreads) k_rev_design(Geo g, Ctrl* ctrl, const Dof* it,
                                                            const T* __restrict__ slabs, long long slab,
                                                            const T* __restrict__ lamh, double* __restrict__ dkp,
                                                            int nsteps, int di) {
  using RP = RevPlanes<2>;
  const int K = g.K, lane = threadIdx.x % LN;
  const int m = (int)((blockIdx.x * (unsigned)kRevThreads + threadIdx.x) / LN);
  const int mm = m < g.ND ? m : 0;
  const int ix = mm % g.nd[0], iy = mm / g.nd[0];
  const bool valid = m < g.ND && dsq(ix, g.nd[0]) + dsq(iy, g.nd[1]) <= g.rad4;
  const T r[3] = {(T)ix - pivot<T>(g, 0), (T)iy - pivot<T>(g, 1), T(0)};
  const int S2 = 2 * g.s, B0 = g.B[0], B1 = g.B[1];
  const long long BC = g.box_cells;
  bool inside = true;
  double acc = 0.0;
  for (int i = blockIdx.y; i < nsteps; i += gridDim.y) {
    const Dof* row = it + (long long)(rev_step(ctrl, di, i) - 1) * (K + 1);
    int lo[3];
    box_origin<2>(g, row[0], lo[0], lo[1], lo[2]);
    for (int k = K; k >= 1; --k) {
      const DofView<T> V(row[k - 1]);
      T l[3], dl[3], usr[2], fr[2], w[2][4];
      int f[2] = {0, 0};
      rot<2>(V.cs, V.sn, r, l);
      drot<2>(V.cs, V.sn, r, dl);
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        usr[a] = V.ug[a] + V.om * dl[a];
        V.split(a, l[a], &f[a], &fr[a]);
        window_weights(g, fr[a], w[a]);
        f[a] += 1 - g.s - lo[a];
      }
      // the window's cells with weight 0 (fr = 0 puts the last one on the support's edge) need not
      // lie in the box
      T we = T(0);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q == lane) we = w[1][q];
      const bool here = valid && lane < S2 && we != T(0);
      const int pe = f[1] + lane;
      if (here && (f[0] < 0 || f[0] + S2 - 1 - (fr[0] == T(0)) >= B0 || pe < 0 || pe >= B1)) inside = false;
      T uref[2] = {T(0), T(0)}, slk = T(0);
      if (here && inside) {
        const T* P = slabs + (long long)i * slab + (long long)(k - 1) * RP::per_itr * BC + f[0] + B0 * pe;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (q >= S2 || w[0][q] == T(0)) continue;
          const T W = w[0][q] * we;
          slk += W * __ldg(P + RP::eps * BC + q);
#pragma unroll
          for (int a = 0; a < 2; ++a) uref[a] += W * __ldg(P + (RP::u + a) * BC + q);
        }
      }
#pragma unroll
      for (int off = 1; off < LN; off <<= 1) {
        slk += __shfl_xor_sync(0xffffffffu, slk, off);
#pragma unroll
        for (int a = 0; a < 2; ++a) uref[a] += __shfl_xor_sync(0xffffffffu, uref[a], off);
      }
      if (valid && lane == 0) {
        const T* lam = lamh + ((long long)i * K + (k - 1)) * 4;
        T dk = slk;
#pragma unroll
        for (int a = 0; a < 2; ++a) {
          uref[a] -= usr[a];
          dk += lam[a] * uref[a];
        }
        dk += lam[3] * (l[0] * uref[1] - l[1] * uref[0]);
        acc += (double)dk;
      }
    }
  }
  if (!inside) atomicOr(&ctrl->status, ST_BOX_OVERFLOW);
  if (valid && lane == 0) dkp[(long long)blockIdx.y * g.ND + m] += acc;
}

__global__ void __launch_bounds__(kRevThreads) k_rev_dksum(int nd, int splits, const double* __restrict__ dkp,
                                                           double* __restrict__ dkref) {
  const int m = blockIdx.x * kRevThreads + threadIdx.x;
  if (m >= nd) return;
  double s = 0.0;
  for (int q = 0; q < splits; ++q) s += dkp[(long long)q * nd + m];
  dkref[m] = s;
}

// Seed of the sweep in the double-buffered carried adjoint (k_adj_init has filled lam_prev, lam_F, lam_T).
__global__ void k_rev_init(Ctrl* ctrl, int nt) {
  double* o = ctrl->rev_lam[nt & 1];
  for (int a = 0; a < 8; ++a) o[a] = ctrl->lam_prev[a];
  for (int a = 0; a < 3; ++a) o[8 + a] = ctrl->lam_F[a];
  o[11] = ctrl->lam_T[0];
}

unsigned rev_ctas(const Geo& g) {
  const long long n = (g.box_cells + kRevThreads - 1) / kRevThreads;
  return (unsigned)(n < kRevMaxCtas ? n : kRevMaxCtas);
}

template <typename T, int D, int AX>
void coef_ax(const Geo& g, const RevBuffers& R, Ctrl* ctrl, const Dof* it, const T* kref, const Moments* mom,
             const T* boxstore, int nbox, int nsteps, int di, cudaStream_t st) {
  using PT = typename Partial<T>::type;
  unsigned nc = (unsigned)((g.box_cells + kRevThreads - 1) / kRevThreads);
  if (D == 3 && coef_axis3d_fits(g)) {
    nc = (unsigned)coef_axis3d_ctas(g, sizeof(T) == 8);
    launch_coef_axis3d<T>(g, R, ctrl, it, kref, boxstore, nbox, nsteps, di, st);
  } else {
    launch(k_rev_coef<T, D, AX>, dim3(nc, g.K, nsteps), kRevThreads, row_bytes<T>(RevSums<D>::N, false), st, g,
           (const Ctrl*)ctrl, it, kref, boxstore, nbox, (T*)R.slabs, R.slab, (PT*)R.mpart, di);
  }
  launch(k_rev_mat<T, D, AX>, dim3(g.K, nsteps), kRevThreads, 0, st, g, (const Ctrl*)ctrl, it, mom, (const PT*)R.mpart,
         (int)nc, (RevMat*)R.mats, di);
}
template <typename T, int D, int AX>
void step_ax(const Geo& g, const RevBuffers& R, Ctrl* ctrl, const Dof* it, T* Lb, long long lstride, int i, int di,
             cudaStream_t st) {
  using PT = typename Partial<T>::type;
  const unsigned nc = rev_ctas(g);
  const bool many = g.box_cells > (long long)nc * kRevThreads;
  launch(many ? k_rev_const<T, D, AX, true> : k_rev_const<T, D, AX, false>, nc, kRevThreads,
         row_bytes<T>(rev_nconst<D>(), many), st, g, (const Ctrl*)ctrl, it, (const T*)R.slabs, R.slab, (const T*)Lb, lstride,
         (PT*)R.cpart, di, i);
  launch(k_rev_apply<T, D, AX>, nc + 1, kRevThreads, (size_t)g.K * (sizeof(RevMat) + 4 * (sizeof(double) + sizeof(T))), st, g, ctrl, it,
         (T*)R.slabs, R.slab, Lb, lstride, (const PT*)R.cpart, (int)nc, (const RevMat*)R.mats, (T*)R.lamh, di, i);
}
#define LKS_REV_DISPATCH(F, ...)                  \
  do {                                            \
    if (g.dim == 2) F<T, 2, 2>(__VA_ARGS__);      \
    else if (g.ax == 0) F<T, 3, 0>(__VA_ARGS__);  \
    else if (g.ax == 1) F<T, 3, 1>(__VA_ARGS__);  \
    else F<T, 3, 2>(__VA_ARGS__);                 \
  } while (0)

}  // namespace

bool reverse_affine_fits(const Geo& g) {
  return (g.dim == 2 || axis3d_fits(g)) && g.box_cells < (1LL << 29) && g.K <= kRevMaxItr;
}

size_t reverse_layout(const Geo& g, bool fp64, int max_steps, RevBuffers* R) {
  const long long esz = fp64 ? 8 : 4, K = g.K;
  const int D = g.dim;
  const long long planes = D == 2 ? K * RevPlanes<2>::per_itr + RevPlanes<2>::consts
                                  : K * RevPlanes<3>::per_itr + RevPlanes<3>::consts;
  const long long nm = D == 2 ? RevSums<2>::N : RevSums<3>::N;
  long long nc = (g.box_cells + kRevThreads - 1) / kRevThreads;
  if (D == 3 && coef_axis3d_fits(g)) nc = std::max(nc, (long long)coef_axis3d_ctas(g, fp64));
  R->slab = planes * g.box_cells;
  // steps per chunk: two chunks' slabs in about half of the L2, so that the planes written by one kernel
  // are read from L2 by the next; at least one, and several chunks a segment to overlap them
  const long long want = (32LL << 20) / (R->slab * esz), part = (max_steps + 3) / 4;
  R->steps = (int)std::max(1LL, std::min({want, part, 64LL}));
  // splits of the design kernel over the chunk's steps (3D: steps and iterations): about 2^17 threads in
  // 2D, 2^17 of the 3D form's, each of which takes eight points
  long long sp = D == 2 ? (1LL << 17) / ((long long)g.ND * LN) : (1LL << 20) / g.ND;
  sp = sp < 1 ? 1 : (sp > 16 ? 16 : sp);
  const long long items = D == 2 ? R->steps : R->steps * K;
  R->splits = (int)(sp < items ? sp : items);
  size_t off = 0;
  auto take = [&](long long bytes) {
    const size_t at = off;
    off += (size_t)((bytes + 255) & ~255LL);
    return at;
  };
  const size_t slabs = take(R->steps * R->slab * esz);
  const size_t mpart = take(R->steps * K * nc * nm * 8);
  const size_t mats = take(R->steps * K * (long long)sizeof(RevMat));
  const size_t lamh = take(R->steps * K * 4 * esz);
  // a second set only where a chunk follows another in a segment, and while the two stay within the limit
  const bool two = max_steps > R->steps && 2 * off <= kRevMaxBytes;
  R->other = two ? off : 0;
  if (two) off *= 2;
  const size_t cpart = take((long long)kRevMaxCtas * 8 * 8);
  const size_t dkp = take((long long)R->splits * g.ND * 8);
  if (R->block) {
    char* p = (char*)R->block;
    R->slabs = p + slabs;
    R->mpart = p + mpart;
    R->mats = p + mats;
    R->cpart = p + cpart;
    R->lamh = p + lamh;
    R->dkp = (double*)(p + dkp);
  }
  return off;
}

void launch_rev_init(const Geo& g, const RevBuffers& R, Ctrl* ctrl, int nt, cudaStream_t st) {
  cudaMemsetAsync(R.dkp, 0, sizeof(double) * (size_t)R.splits * g.ND, st);
  launch(k_rev_init, 1, 1, 0, st, ctrl, nt);
}
void launch_rev_dksum(const Geo& g, const RevBuffers& R, double* dkref, cudaStream_t st) {
  launch(k_rev_dksum, (g.ND + kRevThreads - 1) / kRevThreads, kRevThreads, 0, st, g.ND, R.splits,
         (const double*)R.dkp, dkref);
}

template <typename T>
void launch_rev_coef(const Geo& g, const RevBuffers& R, Ctrl* ctrl, const Dof* it, const T* kref, const Moments* mom,
                     const T* boxstore, int nbox, int nsteps, int di, cudaStream_t st) {
  LKS_REV_DISPATCH(coef_ax, g, R, ctrl, it, kref, mom, boxstore, nbox, nsteps, di, st);
}
template <typename T>
void launch_rev_step(const Geo& g, const RevBuffers& R, Ctrl* ctrl, const Dof* it, T* Lb, long long lstride, int i,
                     int di, cudaStream_t st) {
  LKS_REV_DISPATCH(step_ax, g, R, ctrl, it, Lb, lstride, i, di, st);
}
template <typename T>
void launch_rev_design(const Geo& g, const RevBuffers& R, Ctrl* ctrl, const Dof* it, int nsteps, int di,
                       cudaStream_t st) {
  if (g.dim == 3) return launch_design_axis3d<T>(g, R, ctrl, it, nsteps, di, st);
  const unsigned nb = (unsigned)(((long long)g.ND * LN + kRevThreads - 1) / kRevThreads);
  launch(k_rev_design<T>, dim3(nb, R.splits), kRevThreads, 0, st, g, ctrl, it, (const T*)R.slabs, R.slab,
         (const T*)R.lamh, R.dkp, nsteps, di);
}

#define LKS_REV_INST(T)                                                                                             \
  template void launch_rev_coef<T>(const Geo&, const RevBuffers&, Ctrl*, const Dof*, const T*, const Moments*,      \
                                   const T*, int, int, int, cudaStream_t);                                          \
  template void launch_rev_step<T>(const Geo&, const RevBuffers&, Ctrl*, const Dof*, T*, long long, int, int,       \
                                   cudaStream_t);                                                                   \
  template void launch_rev_design<T>(const Geo&, const RevBuffers&, Ctrl*, const Dof*, int, int, cudaStream_t);
LKS_REV_INST(float)
LKS_REV_INST(double)

}  // namespace lks
