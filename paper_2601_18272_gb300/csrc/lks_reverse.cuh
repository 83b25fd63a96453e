// Layouts and helpers shared by the kernels of the reverse by linear maps (lks_reverse.cu) and their
// 3D forms (lks_axis3d.cu).
#pragma once

#include <climits>

#include "lks_flag.cuh"

namespace lks {

namespace {

constexpr int kRevThreads = 256;
constexpr int kRevMaxItr = 64;     // iterations k_rev_apply's shared memory holds (432 bytes each)
constexpr int kRevMaxCtas = 304;  // k_rev_const, k_rev_apply: every CTA of the latter sums the former's partials

// Planes of a step's slab (box cells each). Per iteration: kappa/(1+kappa), L/(1+kappa) in the plane,
// u, kappa du/dkappa, and the dJ/dT coefficient of dJ/dkappa (k_rev_apply puts dJ/dkappa there).
// Then for iteration N_itr: 1/(1+kappa), du/dkappa, du/d(x^G, theta), du/du^G and du/domega parts.
template <int D>
struct RevPlanes {
  static constexpr int beta = 0, iL = 1, u = 3, kd = 3 + D, eps = 3 + 2 * D, per_itr = 4 + 2 * D;
  static constexpr int inv = 0, del = 1, Q = 1 + D, bphi = Q + (D + 1) * D, bP = bphi + 1, consts = bP + 2;
};
// Sums of k_rev_coef: rows x^G and theta by columns lam_F and lam_T, then the u^G and omega rows.
template <int D>
struct RevSums {
  static constexpr int uF = (D + 1) * (D + 1), uT = uF + 1, oF = uT + 2, oT = oF + 2, N = oT + 1;
};
template <int D>
__host__ __device__ constexpr int rev_nconst() { return 2 * D + 2; }  // c: x^G[D], theta, u^G[D], omega

// Block sums of NV per-thread values with few instructions: the values go through shared memory
// (rows of kRevThreads), 8 threads sum each row's eighths in order and combine them with shuffles.
// A shuffle tree over all threads costs NV * 5 levels in every warp: with 15 to 22 values that was
// as much as the gather itself. FP32 values are summed as double-float pairs.
template <int NV>
struct RowBuf {
  static constexpr int pitch = kRevThreads + 1;
};
template <int NV>
__device__ __forceinline__ void row_sums(const float (&v)[NV], float* buf, float2* out) {
  constexpr int pitch = RowBuf<NV>::pitch;
  const int tid = threadIdx.x;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < NV; ++i) buf[i * pitch + tid] = v[i];
  __syncthreads();
  const int row = tid >> 3, seg = tid & 7;
  static_assert(NV * 8 <= kRevThreads, "eight threads per value");
  if ((tid & ~31) < NV * 8) {  // whole warps (shuffles below)
    float hi = 0.0f, lo = 0.0f;
    if (row < NV) {
      const float* p = buf + row * pitch + seg;
#pragma unroll 8
      for (int j = 0; j < kRevThreads / 8; ++j) {
        const float b = p[8 * j], s = hi + b, bb = s - hi;
        lo += (hi - (s - bb)) + (b - bb);
        hi = s;
      }
    }
#pragma unroll
    for (int off = 4; off > 0; off >>= 1)
      df_add(hi, lo, __shfl_down_sync(0xffffffffu, hi, off, 8), __shfl_down_sync(0xffffffffu, lo, off, 8));
    if (row < NV && seg == 0) out[row] = make_float2(hi, lo);
  }
}
template <int NV>
__device__ __forceinline__ void row_sums(const double (&v)[NV], double* buf, double* out) {
  constexpr int pitch = RowBuf<NV>::pitch;
  const int tid = threadIdx.x;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < NV; ++i) buf[i * pitch + tid] = v[i];
  __syncthreads();
  const int row = tid >> 3, seg = tid & 7;
  static_assert(NV * 8 <= kRevThreads, "eight threads per value");
  if ((tid & ~31) < NV * 8) {
    double s = 0.0;
    if (row < NV) {
      const double* p = buf + row * pitch + seg;
#pragma unroll 8
      for (int j = 0; j < kRevThreads / 8; ++j) s += p[8 * j];
    }
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off, 8);
    if (row < NV && seg == 0) out[row] = s;
  }
}
// Sum of each of N (a power of two) values over the warp's lanes by halving (each level exchanges half of the
// values); lane l ends with that of value l mod N.
template <int N>
__device__ __forceinline__ float halve_sums(float (&x)[N], int lane) {
#pragma unroll
  for (int h = N / 2; h > 0; h >>= 1)
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const float send = (lane & h) ? x[i] : x[h + i], keep = (lane & h) ? x[h + i] : x[i];
      x[i] = keep + __shfl_xor_sync(0xffffffffu, send, h);
    }
#pragma unroll
  for (int off = N; off < 32; off <<= 1) x[0] += __shfl_xor_sync(0xffffffffu, x[0], off);
  return x[0];
}
// The same for threads that have summed several cells, as pairs: the high parts through the rows, the low ones
// by shuffles within each warp, whose sums the row's eight threads add. (Rows for both, twice the buffer, gave
// the kernels another split of L1 and shared memory, and with it no place beside the other branch's CTAs:
// gradients 2 % (128x64x64) to 6 % (157x67x70 duct) longer.)
__host__ __device__ constexpr int pow2_from(int n) { return n <= 8 ? 8 : (n <= 16 ? 16 : 32); }
template <int NV>
__device__ __forceinline__ void row_sums(const Df (&v)[NV], float* buf, float2* out) {
  constexpr int pitch = RowBuf<NV>::pitch, N = pow2_from(NV);
  static_assert(NV * 8 <= kRevThreads && kRevThreads == 256, "eight threads per value, one per warp");
  const int tid = threadIdx.x, lane = tid & 31, row = tid >> 3, seg = tid & 7;
  float* low = buf + NV * pitch;  // [warp][N]
  __syncthreads();
  float x[N];
#pragma unroll
  for (int i = 0; i < N; ++i) x[i] = i < NV ? v[i < NV ? i : 0].lo : 0.0f;
#pragma unroll
  for (int i = 0; i < NV; ++i) buf[i * pitch + tid] = v[i].hi;
  const float l = halve_sums<N>(x, lane);
  if (lane < N) low[(tid >> 5) * N + lane] = l;
  __syncthreads();
  if ((tid & ~31) < NV * 8) {  // whole warps (shuffles below)
    float hi = 0.0f, lo = 0.0f;
    if (row < NV) {
      const float* p = buf + row * pitch + seg;
#pragma unroll 8
      for (int j = 0; j < kRevThreads / 8; ++j) {
        const float b = p[8 * j], s = hi + b, bb = s - hi;
        lo += (hi - (s - bb)) + (b - bb);
        hi = s;
      }
      lo += low[seg * N + row];
    }
#pragma unroll
    for (int off = 4; off > 0; off >>= 1)
      df_add(hi, lo, __shfl_down_sync(0xffffffffu, hi, off, 8), __shfl_down_sync(0xffffffffu, lo, off, 8));
    if (row < NV && seg == 0) out[row] = make_float2(hi, lo);
  }
}
template <int NV>
__device__ __forceinline__ void row_sums(const Dd (&v)[NV], double* buf, double* out) {
  double x[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) x[i] = v[i].v;
  row_sums<NV>(x, buf, out);
}
// Shared memory of row_sums for nv values or pairs.
template <typename T>
size_t row_bytes(int nv, bool pairs) {
  return ((size_t)nv * RowBuf<1>::pitch + (sizeof(T) == 4 && pairs ? 8 * pow2_from(nv) : 0)) * sizeof(T);
}
// Row `row` of partials [n][nv] summed by 8 threads in a fixed order (result in seg 0's thread).
__device__ __forceinline__ double part_sum(const float2* p, int n, int nv, int row, int seg) {
  float hi = 0.0f, lo = 0.0f;
#pragma unroll 4
  for (int q = seg; q < n; q += 8) {
    const float2 b = __ldcg(p + (long long)q * nv + row);
    df_add(hi, lo, b.x, b.y);
  }
#pragma unroll
  for (int off = 4; off > 0; off >>= 1)
    df_add(hi, lo, __shfl_down_sync(0xffffffffu, hi, off, 8), __shfl_down_sync(0xffffffffu, lo, off, 8));
  return (double)hi + (double)lo;
}
__device__ __forceinline__ double part_sum(const double* p, int n, int nv, int row, int seg) {
  double s = 0.0;
#pragma unroll 4
  for (int q = seg; q < n; q += 8) s += __ldcg(p + (long long)q * nv + row);
#pragma unroll
  for (int off = 4; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off, 8);
  return s;
}

// w(r) and w'(r) inside the support.
__device__ __forceinline__ void w_dw(int wk, float r, float* w, float* dw) {
  *w = wfun(wk, r);
  *dw = dwfun(wk, r);
}
__device__ __forceinline__ void w_dw(int wk, double r, double* w, double* dw) {
  if (wk == W_BILINEAR) {
    *w = wfun(wk, r);
    *dw = dwfun(wk, r);
    return;
  }
  double s, c;
  sincospi(0.5 * r, &s, &c);
  *w = 0.25 * (1.0 + c);
  *dw = -0.125 * 3.141592653589793 * s;
}

// Sums over the design points within the support of one cell: index 0 with W, 1 + e with dW/dx_e
// (e the world axis); q: sums with the rotation derivative W_b l_c - W_c l_b times l_b, l_c.
template <typename T>
struct Moments1 {
  T phi[4], kap[4], Pb[4], Pc[4], Lb[4], Lc[4];
  T qPb, qPc, qLb, qLc;
};

// Step of slab i of the chunk that starts di steps below ctrl->t0.
__device__ __forceinline__ int rev_step(const Ctrl* ctrl, int di, int i) { return ctrl->t0 - di - i; }

// One box cell of iteration k from its sums A: its planes (at P, the cell's place in its slab) and
// its share v of the sums of M_k. bs: the step's stored u*; off the grid (ing false) A is zero.
template <typename T, int D, int AX>
__device__ __forceinline__ void rev_cell(const Geo& g, const DofView<T>& V, const Moments1<T>& A, bool ing,
                                         const T* __restrict__ bs, long long bl, T* __restrict__ P, int k,
                                         T (&v)[RevSums<D>::N]) {
  using RP = RevPlanes<D>;
  using RS = RevSums<D>;
  constexpr int b = Axes<AX>::B, c = Axes<AX>::C;
  const int K = g.K;
  const long long BC = g.box_cells;
  const T kap = A.kap[0], inv = T(1) / (T(1) + kap), beta = kap * inv, om = V.om;
  T us[3], u[3], del[3];
#pragma unroll
  for (int a = 0; a < D; ++a) {
    us[a] = V.ug[a] * A.phi[0];
    if (a == b) us[a] -= om * A.Pc[0];
    if (a == c) us[a] += om * A.Pb[0];
    u[a] = ing ? (bs[a * BC + bl] + kap * us[a]) * inv : T(0);  // no stored u* off the grid
    del[a] = (us[a] - u[a]) * inv;
  }
  T* Pk = P + (long long)(k - 1) * RP::per_itr * BC;
  Pk[RP::beta * BC] = beta;
  Pk[RP::iL * BC] = inv * A.Lb[0];
  Pk[(RP::iL + 1) * BC] = inv * A.Lc[0];
#pragma unroll
  for (int a = 0; a < D; ++a) {
    Pk[(RP::u + a) * BC] = u[a];
    Pk[(RP::kd + a) * BC] = kap * del[a];
  }
  Pk[RP::eps * BC] = A.Lb[0] * del[c] - A.Lc[0] * del[b];
  const T bphi = beta * A.phi[0], bPb = beta * A.Pb[0], bPc = beta * A.Pc[0];
  T* Pc = P + (long long)K * RP::per_itr * BC;
  if (k == K) {
    Pc[RP::inv * BC] = inv;
#pragma unroll
    for (int a = 0; a < D; ++a) Pc[(RP::del + a) * BC] = del[a];
    Pc[RP::bphi * BC] = bphi;
    Pc[RP::bP * BC] = bPb;
    Pc[(RP::bP + 1) * BC] = bPc;
  }
  // rows x^G_e (derivative -dW/dx_e) and theta (W_b l_c - W_c l_b, and l turning with the body)
#pragma unroll
  for (int e = 0; e <= D; ++e) {
    T dphi, dk, dPb, dPc, dLb, dLc;
    if (e < D) {
      dphi = -A.phi[1 + e];
      dk = -A.kap[1 + e];
      dPb = -A.Pb[1 + e];
      dPc = -A.Pc[1 + e];
      dLb = -A.Lb[1 + e];
      dLc = -A.Lc[1 + e];
    } else {
      dphi = A.Pc[1 + b] - A.Pb[1 + c];
      dk = A.Lc[1 + b] - A.Lb[1 + c];
      dPb = A.qPb - A.Pc[0];
      dPc = A.qPc + A.Pb[0];
      dLb = A.qLb - A.Lc[0];
      dLc = A.qLc + A.Lb[0];
    }
    T du[3];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      T dus = V.ug[a] * dphi;
      if (a == b) dus -= om * dPc;
      if (a == c) dus += om * dPb;
      du[a] = del[a] * dk + beta * dus;
      if (k == K) Pc[(RP::Q + e * D + a) * BC] = du[a];
      v[e * (D + 1) + a] = kap * du[a] + u[a] * dk;
    }
    v[e * (D + 1) + D] = A.Lb[0] * du[c] - A.Lc[0] * du[b] + dLb * u[c] - dLc * u[b];
  }
  v[RS::uF] = kap * bphi;
  v[RS::uT] = -A.Lc[0] * bphi;
  v[RS::uT + 1] = A.Lb[0] * bphi;
  v[RS::oF] = -kap * bPc;
  v[RS::oF + 1] = kap * bPb;
  v[RS::oT] = A.Lb[0] * bPb + A.Lc[0] * bPc;
}

// Kernel weights of the 2s window cells from floor(x) - s + 1, at the fraction fr of x.
__device__ __forceinline__ void window_weights(const Geo& g, float fr, float (&w)[4]) {
  if (g.wk == W_BILINEAR) {
    w[0] = 1.0f - fr;
    w[1] = fr;
    w[2] = w[3] = 0.0f;
    return;
  }
  const float c = __cosf(1.57079632679f * fr), s = __sinf(1.57079632679f * fr);
  w[0] = 0.25f * (1.0f - s);
  w[1] = 0.25f * (1.0f + c);
  w[2] = 0.25f * (1.0f + s);
  w[3] = 0.25f * (1.0f - c);
}
__device__ __forceinline__ void window_weights(const Geo& g, double fr, double (&w)[4]) {
  if (g.wk == W_BILINEAR) {
    w[0] = 1.0 - fr;
    w[1] = fr;
    w[2] = w[3] = 0.0;
    return;
  }
  double s, c;
  sincospi(0.5 * fr, &s, &c);
  w[0] = 0.25 * (1.0 - s);
  w[1] = 0.25 * (1.0 + c);
  w[2] = 0.25 * (1.0 + s);
  w[3] = 0.25 * (1.0 - c);
}

}  // namespace

}  // namespace lks
