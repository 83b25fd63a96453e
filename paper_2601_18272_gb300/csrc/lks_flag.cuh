// Exchange of the coupling sums and the iterate through flagged words, and the EOM of an iteration,
// shared by the one-launch coupling kernels (lks_couple2d.cu, lks_axis3d.cu).
//
// CTA 0 has no cells: the others publish their D + 1 sums (force, torque) to it, it adds them up, runs
// the EOM and publishes the iterate. Values travel as 64-bit words that carry the iteration's number
// beside 32 bits of payload, so the arrival of the data is the synchronisation: one trip through L2
// each way, and every waiting CTA polls one or two lines. (A form in which every CTA polled the words
// of all others and ran the EOM itself needed one trip only, but took 4.3 us an iteration without
// gather and EOM with 152 CTAs: 57 lines polled by all of them.) A word's number tells it from the one
// two iterations earlier in the same place (two places by the iteration's parity): sums of iteration
// e + 2 are published after the iterate of e + 1 was read, which CTA 0 publishes after it has read
// the sums of e; and likewise the other way. All sums are taken in a fixed order (warps, CTA, then 32
// lanes over the CTAs), so results do not vary between runs. Waits are bounded by one second.
#pragma once

#include "lks_body_common.cuh"
#include "lks_wait.cuh"

namespace lks {

namespace {

// Roundings spelled out where a forward kernel and its recompute must agree to the bit: how the compiler
// joins the products and sums of an expression into multiply-adds is its own choice in each kernel.
__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float mul_(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_(double a, double b) { return __dmul_rn(a, b); }
// a b + c d
template <typename T>
__device__ __forceinline__ T dot2(T a, T b, T c, T d) { return fma_(a, b, mul_(c, d)); }
// The Brinkman update of a cell: (u* + kappa u^S) / (1 + kappa), inv the reciprocal.
template <typename T>
__device__ __forceinline__ T brinkman(T ustar, T kap, T us, T inv) { return mul_(fma_(kap, us, ustar), inv); }

// One value as two 64-bit words (number << 32 | payload) and back.
struct Words {
  unsigned long long a, b;
};
__device__ __forceinline__ void st_words(Words* p, Words w) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(w.a), "l"(w.b) : "memory");
}
__device__ __forceinline__ Words ld_words(const Words* p) {
  Words w;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w.a), "=l"(w.b) : "l"(p) : "memory");
  return w;
}
__device__ __forceinline__ Words pack(unsigned e, unsigned x, unsigned y) {
  return Words{((unsigned long long)e << 32) | x, ((unsigned long long)e << 32) | y};
}

// The value of a whole warp's lanes (fixed order), and a CTA's or the grid's sum of one component.
struct Df {
  float hi, lo;
  __device__ __forceinline__ void zero() { hi = lo = 0.0f; }
  __device__ __forceinline__ void set(float v) { hi = v, lo = 0.0f; }
  __device__ __forceinline__ void add(const Df& o) { df_add(hi, lo, o.hi, o.lo); }
  __device__ __forceinline__ Df from_xor(int off) const {
    return Df{__shfl_xor_sync(0xffffffffu, hi, off), __shfl_xor_sync(0xffffffffu, lo, off)};
  }
  __device__ __forceinline__ Words words(unsigned e) const { return pack(e, __float_as_uint(hi), __float_as_uint(lo)); }
  __device__ __forceinline__ void read(const Words& w) {
    hi = __uint_as_float((unsigned)w.a);
    lo = __uint_as_float((unsigned)w.b);
  }
  __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};
struct Dd {
  double v;
  __device__ __forceinline__ void zero() { v = 0.0; }
  __device__ __forceinline__ void set(double x) { v = x; }
  __device__ __forceinline__ void add(const Dd& o) { v += o.v; }
  __device__ __forceinline__ Dd from_xor(int off) const { return Dd{__shfl_xor_sync(0xffffffffu, v, off)}; }
  __device__ __forceinline__ Words words(unsigned e) const {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return pack(e, (unsigned)b, (unsigned)(b >> 32));
  }
  __device__ __forceinline__ void read(const Words& w) {
    v = __longlong_as_double((long long)((w.a & 0xffffffffull) | (w.b << 32)));
  }
  __device__ __forceinline__ double value() const { return v; }
};
template <typename T>
struct SumOf;
template <>
struct SumOf<float> {
  using type = Df;
};
template <>
struct SumOf<double> {
  using type = Dd;
};
// A running sum of FP32 values as a double-float pair, or of doubles.
__device__ __forceinline__ void run_add(Df& s, float b) {
  const float t = s.hi + b, bb = t - s.hi;
  s.lo += (s.hi - (t - bb)) + (b - bb);
  s.hi = t;
}
__device__ __forceinline__ void run_add(Dd& s, double b) { s.v += b; }
// Two sums at once (FP32 in packed instructions).
__device__ __forceinline__ void run_add2(Df& s, Df& t, float b, float c) {
  const float2 h = make_float2(s.hi, t.hi), x = make_float2(b, c), one = make_float2(-1.0f, -1.0f);
  const float2 sum = __fadd2_rn(h, x), bb = __ffma2_rn(one, h, sum);
  const float2 e = __fadd2_rn(__ffma2_rn(one, __ffma2_rn(one, bb, sum), h), __ffma2_rn(one, bb, x));
  const float2 lo = __fadd2_rn(make_float2(s.lo, t.lo), e);
  s = Df{sum.x, lo.x};
  t = Df{sum.y, lo.y};
}
__device__ __forceinline__ void run_add2(Dd& s, Dd& t, double b, double c) {
  s.v += b;
  t.v += c;
}
template <int STRIDE, typename V>
__device__ __forceinline__ void warp_total(V& v) {
#pragma unroll
  for (int off = 16; off >= STRIDE; off >>= 1) v.add(v.from_xor(off));
}

// EOM of an iteration, one component per warp (below D: an axis; D: the rotation), in FP64. Every FP64
// instruction of a warp costs 64 cycles, dependent or not, so prepare (while the other warps gather)
// does what does not need the sums, and finish spends about a dozen. The cosine of the step's rotation
// is taken on the even lanes and its sine on the odd ones by the same instructions with their own
// coefficients. Range tests are made on the exponent in integers. All lanes of the warp call both.
struct EomPart {
  double c0, im, q0, f0, x0, y0;  // v = s im + c0; q = q0 + v; f0 = frac(q0); cos/sin(t-1) by lane
  int xi0;
  bool fr;
  template <int D, int AX>
  __device__ __forceinline__ void prepare(const Geo& g, const Moments& mom, const Dof& s0, const Dof& sk, int comp,
                                          int lane) {
    constexpr int B = Axes<AX>::B, C = Axes<AX>::C;
    const double cs = sk.cs, sn = sk.sn, om = sk.s[7];
    const double kb = cs * mom.K1[B] - sn * mom.K1[C], kc = sn * mom.K1[B] + cs * mom.K1[C];  // R K1
    double pre, v0;
    if (comp < D) {
      pre = mom.K0 * sk.s[3 + comp] + om * (comp == B ? -kc : (comp == C ? kb : 0.0));
      fr = (g.dof_mask & (1 << comp)) != 0;
      v0 = s0.s[3 + comp];
      im = g.inv_mass;
      q0 = s0.s[comp];
      const double fl = floor(q0);
      xi0 = (int)fl;
      f0 = q0 - fl;
    } else {
      pre = (kb * sk.s[3 + C] - kc * sk.s[3 + B]) + om * mom.K2p;
      fr = (g.dof_mask & DOF_ROT) != 0;
      v0 = s0.s[7];
      im = g.inv_inertia;
      q0 = s0.s[6];
      x0 = (lane & 1) ? s0.sn : s0.cs;  // cos' = cs c - sn s, sin' = sn c + cs s
      y0 = (lane & 1) ? s0.cs : -s0.sn;
    }
    c0 = fr ? v0 - pre * im : v0;
    if (!fr) im = 0.0;
  }
  // s: the component's sum. Writes the iterate's entries to nx and publishes those the gather reads
  // (see Pose); returns the status bits.
  template <typename T, int D>
  __device__ __forceinline__ int finish(const Geo& g, double s, Dof* nx, unsigned long long* pose, unsigned e, int comp,
                                        int lane) const;
};

// What the cells need of an iterate, and its words: FP32 per axis u^G, fraction and floor of x^G, then
// cos, sin, omega (3 D + 3 words); FP64 per axis u^G and x^G, then cos, sin, omega (4 D + 6 words).
template <typename T, int D>
struct Pose;
template <int D>
struct Pose<float, D> {
  static constexpr int words = 3 * D + 3;
  float cs, sn, om, ug[D], xf[D];
  int xi[D];
  __device__ __forceinline__ void set(const Dof& d) {
    cs = d.csf, sn = d.snf, om = d.om;
    for (int a = 0; a < D; ++a) ug[a] = d.ug[a], xf[a] = d.xf[a], xi[a] = d.xi[a];
  }
  // word w of the iterate
  __device__ __forceinline__ void put(int w, unsigned p, unsigned) {
    const float f = __uint_as_float(p);
    const int a = w / 3, i = w % 3;
    if (a < D) {
      if (i == 0) ug[a] = f;
      if (i == 1) xf[a] = f;
      if (i == 2) xi[a] = (int)p;
    } else {
      (i == 0 ? cs : i == 1 ? sn : om) = f;
    }
  }
  __device__ __forceinline__ float rel(int a, int p) const { return (float)(p - xi[a]) - xf[a]; }
};
template <int D>
struct Pose<double, D> {
  static constexpr int words = 4 * D + 6;
  double cs, sn, om, ug[D], x[D];
  __device__ __forceinline__ void set(const Dof& d) {
    cs = d.cs, sn = d.sn, om = d.s[7];
    for (int a = 0; a < D; ++a) ug[a] = d.s[3 + a], x[a] = d.s[a];
  }
  // the low word w (even) of the iterate, hi the next one
  __device__ __forceinline__ void put(int w, unsigned p, unsigned hi) {
    if (w & 1) return;
    const double f = __hiloint2double((int)hi, (int)p);
    if (w < 4 * D) {
      (w & 2 ? x[w / 4] : ug[w / 4]) = f;
    } else {
      (w == 4 * D ? cs : w == 4 * D + 2 ? sn : om) = f;
    }
  }
  __device__ __forceinline__ double rel(int a, int p) const { return (double)p - x[a]; }
};

__device__ __forceinline__ void st_word(unsigned long long* p, unsigned e, unsigned payload) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(((unsigned long long)e << 32) | payload) : "memory");
}
__device__ __forceinline__ unsigned long long ld_word(const unsigned long long* p) {
  unsigned long long w;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
  return w;
}

template <typename T, int D>
__device__ __forceinline__ int EomPart::finish(const Geo& g, double s, Dof* nx, unsigned long long* pose, unsigned e,
                                               int comp, int lane) const {
  constexpr bool D64 = sizeof(T) == 8;
  const double v = fma(s, im, c0);
  const int hi = __double2hiint(v) & 0x7fffffff;
  int st = 0;
  if (hi >= 0x7ff00000 || (__double2hiint(s) & 0x7fffffff) >= 0x7ff00000) st = ST_NONFINITE;
  if (comp < D) {
    const double q = fr ? q0 + v : q0;
    if constexpr (D64) {
      const double w = lane < 2 ? v : q;
      if (lane < 4) st_word(pose + 4 * comp + lane, e, (unsigned)((lane & 1) ? __double2hiint(w) : __double2loint(w)));
    }
    if (hi >= 0x3ff00000 && fr && fabs(v) > (double)g.margin) st |= ST_BOX_OVERFLOW;
    // floor and fraction of the position from those of t-1 (a crossing renews them)
    double f = fr ? f0 + v : f0;
    int xi = xi0;
    const int hf = __double2hiint(f);
    if (hf < 0 || hf >= 0x3ff00000) {
      const double fl = floor(f);
      xi += (int)fl;
      f -= fl;
    }
    const float vf = (float)v, ff = (float)f;
    if constexpr (!D64) {
      const unsigned w = lane == 0 ? __float_as_uint(vf) : (lane == 1 ? __float_as_uint(ff) : (unsigned)xi);
      if (lane < 3) st_word(pose + 3 * comp + lane, e, w);
    }
    if (lane == 0) {
      nx->s[comp] = q;
      nx->s[3 + comp] = v;
      nx->xi[comp] = xi;
      nx->xf[comp] = ff;
      nx->ug[comp] = vf;
    }
    return st;
  }
  const bool sine = lane & 1;
  const double x = fr ? v : 0.0;  // the step's rotation
  const int hx = fr ? hi : 0;
  double p;
  if (hx > 0x3fd00000) {  // above 1/4
    double sd, cd;
    sincos(x, &sd, &cd);
    p = sine ? sd : cd;
  } else {
    // sums of (-1)^k x^2k / (2k)! and x (-1)^k x^2k / (2k+1)!: up to |x| = 2^-10 three terms leave
    // less than 2e-21, up to 1/64 five (1e-25), up to 1/4 nine (1e-27)
    const double x2 = x * x;
    p = 0.0;
    if (hx > 0x3f500000) {
      if (hx > 0x3f900000) {
        p = sine ? 1.0 / 355687428096000.0 : 1.0 / 20922789888000.0;
        p = fma(p, x2, sine ? -1.0 / 1307674368000.0 : -1.0 / 87178291200.0);
        p = fma(p, x2, sine ? 1.0 / 6227020800.0 : 1.0 / 479001600.0);
        p = fma(p, x2, sine ? -1.0 / 39916800.0 : -1.0 / 3628800.0);
      }
      p = fma(p, x2, sine ? 1.0 / 362880.0 : 1.0 / 40320.0);
      p = fma(p, x2, sine ? -1.0 / 5040.0 : -1.0 / 720.0);
    }
    p = fma(p, x2, sine ? 1.0 / 120.0 : 1.0 / 24.0);
    p = fma(p, x2, sine ? -1.0 / 6.0 : -1.0 / 2.0);
    p = fma(p, x2, 1.0);
    const double ps = p * x;
    if (sine) p = ps;
  }
  const double other = __shfl_xor_sync(0xffffffffu, p, 1);
  const double trig = fma(x0, sine ? other : p, y0 * (sine ? p : other));  // cos, sin by lane parity
  const float tf = (float)trig, vf = (float)v;
  if constexpr (D64) {
    const double c = __shfl_sync(0xffffffffu, trig, 0), sn = __shfl_sync(0xffffffffu, trig, 1);
    const double w = lane < 2 ? c : (lane < 4 ? sn : v);
    if (lane < 6) st_word(pose + 4 * D + lane, e, (unsigned)((lane & 1) ? __double2hiint(w) : __double2loint(w)));
  } else {
    if (lane < 3) st_word(pose + 3 * D + lane, e, __float_as_uint(lane < 2 ? tf : vf));
  }
  if (lane == 0) {
    nx->s[6] = fr ? q0 + v : q0;
    nx->s[7] = v;
    nx->om = vf;
    nx->cs = trig;
    nx->csf = tf;
  } else if (lane == 1) {
    nx->sn = trig;
    nx->snf = tf;
  }
  return st;
}

// The exchange's words: sums [parity][component][CTA], then iterates [parity][kPoseWords] and as many
// that the test hook writes to.
constexpr int kPoseWords = 24;
template <int D>
__device__ __forceinline__ Words* sum_words(void* w, unsigned e, int comp, int cells) {
  return static_cast<Words*>(w) + ((long long)(e & 1u) * (D + 1) + comp) * cells;
}
template <int D>
__device__ __forceinline__ unsigned long long* pose_words(void* w, int cells, int place) {
  return reinterpret_cast<unsigned long long*>(static_cast<Words*>(w) + 2LL * (D + 1) * cells) + place * kPoseWords;
}

// CTA 0: warp `comp` adds the CTAs' sums of its component and runs its part of the EOM.
template <typename T, int D, int AX>
__device__ __forceinline__ void flag_root(const Geo& g, Ctrl* ctrl, Dof* row, const Moments* __restrict__ mom,
                                          void* words, int cells, unsigned e0, bool skip, Dof (&sd)[2], int& gave_up) {
  using V = typename SumOf<T>::type;
  constexpr int NVC = D + 1, DW = (int)(sizeof(Dof) / sizeof(double));
  const int tid = threadIdx.x, comp = tid >> 5, lane = tid & 31, K = g.K;
  if (comp >= NVC) return;
  auto sync = [] { asm volatile("bar.sync 1, %0;" ::"n"(NVC * 32) : "memory"); };
  double* sdw = reinterpret_cast<double*>(sd);
  for (int k = 1; k <= K; ++k) {
    const unsigned e = e0 + (unsigned)k;
    EomPart eom;
    eom.prepare<D, AX>(g, *mom, sd[0], sd[1], comp, lane);
    const Words* place = sum_words<D>(words, e, comp, cells);
    V s;
    s.zero();
    WaitLimit limit;
    bool ok = true;
    for (int q0 = lane; q0 < cells && ok; q0 += 32 * 4) {
      Words w[4];
      bool have;
      do {  // up to four words at a time in flight
        have = true;
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (q0 + 32 * j < cells) w[j] = ld_words(place + q0 + 32 * j);
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (q0 + 32 * j < cells) have = have && (unsigned)(w[j].a >> 32) == e && (unsigned)(w[j].b >> 32) == e;
        if (!have && limit.over(&ctrl->status)) ok = false;
      } while (!have && ok);
      if (ok)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (q0 + 32 * j < cells) {
            V x;
            x.read(w[j]);
            s.add(x);
          }
    }
    __syncwarp();
    ok = __all_sync(0xffffffffu, ok);
    if (!ok && lane == 0) gave_up = 1;
    sync();  // every warp has read sd[1]
    if (gave_up) return;
    warp_total<1>(s);
    unsigned long long* pose = pose_words<D>(words, cells, skip ? 2 : (int)(e & 1u));
    const int st = eom.finish<T, D>(g, s.value(), &sd[1], pose, e, comp, lane);
    if (st && lane == 0) atomicOr(&ctrl->status, st);
    sync();
    if (tid < DW) {
      reinterpret_cast<double*>(row + k)[tid] = sdw[DW + tid];
      if (k == K) reinterpret_cast<double*>(row + K + 1)[tid] = sdw[DW + tid];  // s(t): the next step's row 0
    }
  }
}

// The end of an iteration in a CTA with cells, after the block barrier that follows its warps' sums
// part[warp][component]: the first warps publish the CTA's sums, the last one waits for the iterate.
// All threads of the block call it; a block barrier must follow.
template <typename T, int D>
__device__ __forceinline__ void flag_exchange(void* words, unsigned e, int cta, int cells, bool last, int* status,
                                              const typename SumOf<T>::type* part, Pose<T, D>& pose, int& gave_up) {
  using V = typename SumOf<T>::type;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = (int)(blockDim.x >> 5);
  if (warp <= D) {
    V s;
    s.zero();
    if (lane < nw) s = part[lane * (D + 1) + warp];
    warp_total<1>(s);
    if (lane == 0) st_words(sum_words<D>(words, e, warp, cells) + cta, s.words(e));
  }
  if (!last && warp == nw - 1) {
    const unsigned long long* p = pose_words<D>(words, cells, (int)(e & 1u));
    unsigned long long w = 0;
    WaitLimit limit;
    bool ok = true;
    if (lane < Pose<T, D>::words)
      while ((unsigned)((w = ld_word(p + lane)) >> 32) != e)
        if (limit.over(status)) {
          ok = false;
          break;
        }
    __syncwarp();
    const unsigned hi = __shfl_down_sync(0xffffffffu, (unsigned)w, 1);
    if (lane < Pose<T, D>::words) {
      if (ok)
        pose.put(lane, (unsigned)w, hi);
      else
        gave_up = 1;
    }
  }
}

}  // namespace

}  // namespace lks
