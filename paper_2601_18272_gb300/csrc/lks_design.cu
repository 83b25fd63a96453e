// Design chain (Sec. 3.2, Eqs. filter and projection; Sec. 4.2, cyclic periodic mapping) and its
// transpose, on the design grid in FP64.
//
//   gamma --(cyclic expansion)--> g1 --(density filter)--> gtil --(Heaviside projection)--> gbar
//
// Cyclic expansion (order 2 or 4): every design point takes the value of its orbit's
// representative, the smallest index among its images under rotations by 360/order degrees about
// the design-grid centre in the plane normal to the rotation axis. Filter: gtil_i = sum_j w_ij g1_j
// / W_i with w_ij = (R - |x_i - x_j|) / R for |x_i - x_j| <= R and W_i = sum_j w_ij, both points in
// the design domain. Projection: gbar = (tanh(beta eta) + tanh(beta (gtil - eta))) /
// (tanh(beta eta) + tanh(beta (1 - eta))). gbar feeds the Brinkman coefficient and the volume
// constraint G = sum_dom gbar / (V_min N_dom) - 1 (Eq. constraint).
//
// Transpose: v3 = dJ/dgbar -> v2 = v3 dgbar/dgtil -> v1_j = sum_i w_ij v2_i / W_i (the weights are
// symmetric, so this is the same gather as the filter applied to v2 / W) -> out_m = sum of v1 over
// m's orbit when m is its own representative, else 0. Every output is one thread's fixed-order sum.
#include <climits>
#include <cmath>

#include "lks_kernels.h"

namespace lks {

namespace {

constexpr int kDB = 256;

__device__ __forceinline__ void design_ijk(const Geo& g, int m, int* i) {
  i[0] = m % g.nd[0];
  i[1] = (m / g.nd[0]) % g.nd[1];
  i[2] = m / (g.nd[0] * g.nd[1]);
}
__device__ __forceinline__ int design_index(const Geo& g, const int* i) { return i[0] + g.nd[0] * (i[1] + g.nd[1] * i[2]); }

__device__ __forceinline__ bool in_domain(const Geo& g, const int* i) {
  return dsq(i[0], g.nd[0]) + dsq(i[1], g.nd[1]) + dsq(i[2], g.nd[2]) <= g.rad4;
}

// The images of design point m under the cyclic rotations (img[0] = m); returns their number.
__device__ __forceinline__ int orbit(const Geo& g, int m, int* img) {
  img[0] = m;
  if (g.cyc <= 1) return 1;
  const int b = g.axb, c = g.axc;
  int i[3];
  design_ijk(g, m, i);
  for (int k = 1; k < g.cyc; ++k) {
    int j[3] = {i[0], i[1], i[2]};
    if (g.cyc == 4) {
      j[b] = g.nd[c] - 1 - i[c];
      j[c] = i[b];
    } else {
      j[b] = g.nd[b] - 1 - i[b];
      j[c] = g.nd[c] - 1 - i[c];
    }
    i[0] = j[0];
    i[1] = j[1];
    i[2] = j[2];
    img[k] = design_index(g, i);
  }
  return g.cyc;
}

__global__ void __launch_bounds__(kDB) k_expand(Geo g, const double* __restrict__ gamma, double* __restrict__ g1) {
  const int m = blockIdx.x * kDB + threadIdx.x;
  if (m >= g.ND) return;
  int img[4];
  const int n = orbit(g, m, img);
  int rep = img[0];
  for (int k = 1; k < n; ++k) rep = min(rep, img[k]);
  g1[m] = gamma[rep];
}

// Filter weights by squared distance, (R - sqrt(d2)) / R up to R (beyond: -1), and the weights' sum
// over a whole disc in the order of filter_sum. The square root and the division took most of the
// filter's FP64 instructions (each costs a warp 64 cycles) when every pair of points computed its own;
// the host makes the table (the same IEEE operations) and passes it as an argument, whose uniform index
// costs no shared load (lks_constraint with its gradient on a 256^2 design, R = 3, with projection and
// cyclic order 4: 350 us per pair, 111 with a table per block, which each block waited for, 96 so). Radii whose
// table does not fit compute each pair's.
constexpr int kTab = 128;
struct FilterTab {
  int n;  // entries (0: no table)
  double full, w[kTab];
};
__host__ __device__ inline double filter_weight(double R, int d2) {
  const double dist = sqrt((double)d2);
  return dist > R ? -1.0 : (R - dist) / R;
}
FilterTab make_table(const Geo& g) {
  FilterTab t;
  t.n = 0;
  t.full = 0.0;
  const double R = g.frad;
  if (!(R > 0.0) || R * R + 2.0 > (double)kTab) return t;
  const int rr = (int)std::floor(R), ez = g.dim == 3 ? rr : 0;
  t.n = (int)std::floor(R * R) + 2;  // every squared distance up to R^2, one more for its rounding
  for (int d2 = 0; d2 < t.n; ++d2) t.w[d2] = filter_weight(R, d2);
  for (int dz = -ez; dz <= ez; ++dz)
    for (int dy = -rr; dy <= rr; ++dy)
      for (int dx = -rr; dx <= rr; ++dx) {
        const int d2 = dx * dx + dy * dy + dz * dz;
        if (d2 < t.n && t.w[d2] >= 0.0) t.full += t.w[d2];
      }
  return t;
}

// Sum of w_ij src_j over the filter disc of i (points of the design domain). All lanes of the warp call it, for
// its vote; those without a point of their own (in false) get 0.
template <bool NEED_W>
__device__ __forceinline__ double filter_sum(const Geo& g, const FilterTab& tab, const double* __restrict__ src,
                                             const int* i, bool in, double* W) {
  const double R = g.frad;
  const int rr = (int)floor(R);
  const int ez = (g.dim == 3) ? rr : 0;
  const bool ball = g.rad4 != INT_MAX, table = tab.n > 0;
  double a = 0.0, w = 0.0;
  const int x0 = max(-rr, -i[0]), x1 = min(rr, g.nd[0] - 1 - i[0]);
  const int y0 = max(-rr, -i[1]), y1 = min(rr, g.nd[1] - 1 - i[1]);
  const int z0 = max(-ez, -i[2]), z1 = min(ez, g.nd[2] - 1 - i[2]);
  const bool whole = !ball && table && x0 == -rr && x1 == rr && y0 == -rr && y1 == rr && z0 == -ez && z1 == ez;
  const bool even = __all_sync(0xffffffffu, whole || !in);
  if (!in) return 0.0;
  for (int dz = even ? -ez : z0; dz <= (even ? ez : z1); ++dz)
    for (int dy = even ? -rr : y0; dy <= (even ? rr : y1); ++dy) {
      const int r2 = dy * dy + dz * dz;
      const double* row = src + i[0] + (long long)g.nd[0] * (i[1] + dy + (long long)g.nd[1] * (i[2] + dz));
      if (even) {  // the warp's discs are whole: the same weights for every lane
#pragma unroll 4
        for (int dx = -rr; dx <= rr; ++dx) {
          const int d2 = dx * dx + r2;
          const double wij = d2 < tab.n ? tab.w[d2] : -1.0;
          if (wij >= 0.0) a += wij * row[dx];
        }
        continue;
      }
      for (int dx = x0; dx <= x1; ++dx) {
        const int d2 = dx * dx + r2;
        const double wij = table ? (d2 < tab.n ? tab.w[d2] : -1.0) : filter_weight(R, d2);
        if (wij < 0.0) continue;
        if (ball) {
          const int j[3] = {i[0] + dx, i[1] + dy, i[2] + dz};
          if (!in_domain(g, j)) continue;
        }
        a += wij * row[dx];
        if (NEED_W && !whole) w += wij;
      }
    }
  if (NEED_W) *W = whole ? tab.full : w;
  return a;
}

// tanh(beta eta) and the projection's denominator, the same for every point: once per block.
__device__ __forceinline__ void make_projection(const Geo& g, double (&pr)[2]) {
  if (g.pbeta > 0.0) {
    if (threadIdx.x == 32) pr[0] = tanh(g.pbeta * g.peta);
    if (threadIdx.x == 64) pr[1] = tanh(g.pbeta * (1.0 - g.peta));
  }
}

__global__ void __launch_bounds__(kDB) k_filter_project(Geo g, const __grid_constant__ FilterTab tab,
                                                        const double* __restrict__ g1, double* __restrict__ gtil,
                                                        double* __restrict__ gbar, double* __restrict__ W) {
  __shared__ double pr[2];
  make_projection(g, pr);
  __syncthreads();
  const int m = blockIdx.x * kDB + threadIdx.x;
  int i[3];
  design_ijk(g, min(m, g.ND - 1), i);
  const bool in = m < g.ND && in_domain(g, i);
  double gt = 0.0, w = 1.0;
  if (g.frad > 0.0) gt = filter_sum<true>(g, tab, g1, i, in, &w) / w;
  if (m >= g.ND) return;
  if (!in) {
    gtil[m] = gbar[m] = 0.0;
    W[m] = 1.0;
    return;
  }
  if (!(g.frad > 0.0)) gt = g1[m];
  gtil[m] = gt;
  W[m] = w;
  if (g.pbeta > 0.0)
    gbar[m] = (pr[0] + tanh(g.pbeta * (gt - g.peta))) / (pr[0] + pr[1]);
  else
    gbar[m] = gt;
}

// out = dJ/dgbar dgbar/dgtil / W, zero outside the domain, with dJ/dgbar = dJ/dkappa^ref times
// dkappa^ref/dgbar (Eq. brinkman_coefficient), or a constant over the domain (the volume's gradient,
// 1 / (v_min * vol[1])).
struct GradIn {
  const double *gbar, *dkref;
  double kmax, q;
  const double* vol;  // dkref null
  double v_min;
};
__global__ void __launch_bounds__(kDB) k_project_T(Geo g, GradIn in, const double* __restrict__ gtil,
                                                   const double* __restrict__ W, double* __restrict__ out) {
  __shared__ double pr[2];
  make_projection(g, pr);
  __syncthreads();
  const int m = blockIdx.x * kDB + threadIdx.x;
  if (m >= g.ND) return;
  int i[3];
  design_ijk(g, m, i);
  if (!in_domain(g, i)) {
    out[m] = 0.0;
    return;
  }
  double v;
  if (in.dkref) {
    const double den = (1.0 - in.gbar[m]) + in.q;
    v = in.dkref[m] * in.kmax * in.q * (1.0 + in.q) / (den * den);
  } else {
    v = 1.0 / (in.v_min * in.vol[1]);
  }
  double d = 1.0;
  if (g.pbeta > 0.0) {
    const double th = tanh(g.pbeta * (gtil[m] - g.peta));
    d = g.pbeta * (1.0 - th * th) / (pr[0] + pr[1]);
  }
  out[m] = g.frad > 0.0 ? v * d / W[m] : v * d;
}

__global__ void __launch_bounds__(kDB) k_filter_T(Geo g, const __grid_constant__ FilterTab tab,
                                                  const double* __restrict__ v, double* __restrict__ out) {
  const int m = blockIdx.x * kDB + threadIdx.x;
  int i[3];
  design_ijk(g, min(m, g.ND - 1), i);
  const double s = filter_sum<false>(g, tab, v, i, m < g.ND && in_domain(g, i), nullptr);
  if (m < g.ND) out[m] = s;
}

__global__ void __launch_bounds__(kDB) k_orbit_sum(Geo g, const double* __restrict__ v, double* __restrict__ out) {
  const int m = blockIdx.x * kDB + threadIdx.x;
  if (m >= g.ND) return;
  int img[4];
  const int n = orbit(g, m, img);
  bool rep = true;
  double s = 0.0;
  for (int k = 0; k < n; ++k) {
    rep = rep && img[k] >= m;
    bool seen = false;  // a point the rotation fixes appears more than once among the images
    for (int q = 0; q < k; ++q) seen = seen || img[q] == img[k];
    if (!seen) s += v[img[k]];
  }
  out[m] = rep ? s : 0.0;
}

// Sum of gbar over the design domain in a fixed order, and the domain's point count: one cluster of
// eight CTAs, whose sums the first one reads from the others' shared memory (one CTA alone was bound
// by the latency of its loads).
constexpr int kVolCtas = 8;
__global__ void __cluster_dims__(kVolCtas, 1, 1) __launch_bounds__(1024) k_volume(Geo g, const double* __restrict__ gbar,
                                                                                  double* __restrict__ out) {
  __shared__ double red[32 * 2], mine[2];
  const bool ball = g.rad4 != INT_MAX;
  double v[2] = {0.0, 0.0};
  const int stride = 1024 * kVolCtas;
  for (int m = blockIdx.x * 1024 + threadIdx.x; m < g.ND; m += 4 * stride) {
    double x[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) x[j] = m + j * stride < g.ND ? gbar[m + j * stride] : 0.0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (m + j * stride >= g.ND) continue;
      if (ball) {
        int i[3];
        design_ijk(g, m + j * stride, i);
        if (!in_domain(g, i)) continue;
      }
      v[0] += x[j];
      if (ball) v[1] += 1.0;
    }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int h = 0; h < 2; ++h) {  // a tree over the lanes, then over the warps
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
      if (ball) v[1] += __shfl_xor_sync(0xffffffffu, v[1], off);
    }
    if (h == 0) {
      if (lane == 0) {
        red[warp] = v[0];
        red[32 + warp] = v[1];
      }
      __syncthreads();
      if (warp != 0) break;
      v[0] = red[lane];
      v[1] = red[32 + lane];
    }
  }
  if (threadIdx.x == 0) {
    mine[0] = v[0];
    mine[1] = v[1];
  }
  auto cluster_sync = [] {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  };
  cluster_sync();
  if (blockIdx.x == 0 && threadIdx.x < 2) {
    const unsigned at = (unsigned)__cvta_generic_to_shared(&mine[threadIdx.x]);
    double s = 0.0;
    for (int c = 0; c < kVolCtas; ++c) {
      unsigned ra;
      double x;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(at), "r"(c));
      asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(x) : "r"(ra) : "memory");
      s += x;
    }
    out[threadIdx.x] = threadIdx.x == 1 && !ball ? (double)g.ND : s;
  }
  cluster_sync();  // no CTA leaves before its sums are read
}

inline unsigned nblk(const Geo& g) { return (unsigned)((g.ND + kDB - 1) / kDB); }

}  // namespace

// The expansion is a copy without cyclic order: the filter then reads gamma itself.
int launch_design_chain(const Geo& g, const double* gamma, double* g1, double* gtil, double* gbar, double* W,
                        cudaStream_t st) {
  const double* src = gamma;
  if (g.cyc > 1) {
    launch(k_expand, nblk(g), kDB, 0, st, g, gamma, g1);
    src = g1;
  }
  launch(k_filter_project, nblk(g), kDB, 0, st, g, make_table(g), src, gtil, gbar, W);
  return g.cyc > 1 ? 2 : 1;
}

namespace {
// Transpose of the chain: projection, filter and orbit sum, without the steps that are off.
int chain_T(const Geo& g, const GradIn& in, const double* gtil, const double* W, double* v, double* tmp, double* out,
            cudaStream_t st) {
  const bool filter = g.frad > 0.0, cyclic = g.cyc > 1;
  double* o1 = filter || cyclic ? v : out;
  launch(k_project_T, nblk(g), kDB, 0, st, g, in, gtil, W, o1);
  double* o2 = cyclic ? tmp : out;
  if (filter) launch(k_filter_T, nblk(g), kDB, 0, st, g, make_table(g), (const double*)o1, o2);
  if (cyclic) launch(k_orbit_sum, nblk(g), kDB, 0, st, g, (const double*)(filter ? o2 : o1), out);
  return 1 + (filter ? 1 : 0) + (cyclic ? 1 : 0);
}
}  // namespace

int launch_sensitivity(const Geo& g, const double* gbar, const double* dkref, double kappa_max, double q,
                       const double* gtil, const double* W, double* v, double* tmp, double* out, cudaStream_t st) {
  return chain_T(g, GradIn{gbar, dkref, kappa_max, q, nullptr, 0.0}, gtil, W, v, tmp, out, st);
}

void launch_volume(const Geo& g, const double* gbar, double* out2, cudaStream_t st) {
  launch(k_volume, kVolCtas, 1024, 0, st, g, gbar, out2);
}

int launch_volume_gradient(const Geo& g, const double* vol, double v_min, const double* gtil, const double* W, double* v,
                           double* tmp, double* out, cudaStream_t st) {
  return chain_T(g, GradIn{nullptr, nullptr, 0.0, 0.0, vol, v_min}, gtil, W, v, tmp, out, st);
}

}  // namespace lks
