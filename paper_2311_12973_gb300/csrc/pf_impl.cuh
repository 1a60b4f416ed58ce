// pf_impl.cuh -- bootstrap particle filter kernel (Sec. II of the paper).
//
// One group of threads runs one filter over all T steps: each thread holds
// PPT consecutive particles in registers.  Per step:
//   1. propagate with the state equation (Eq. 1) using counter-based normals;
//   2. log-weight with the observation density (Eq. 2; bootstrap form of Eq. 5);
//   3. group max of the log-weights (warp shuffles, one barrier);
//   4. quantise q_j = floor(exp(l_j - max) 2^B), warp-local inclusive scan of q
//      in registers + shuffles, warp totals to shared memory (second barrier);
//   5. log-likelihood increment log((1/M) sum_j w_j) = max + log(S 2^-B) - log M
//      from the exact integer total S (Eq. 8, with the mean-weight reset of
//      Eq. 13 every step);
//   6. systematic resampling (Eqs. 26-27): slot j takes the first particle whose
//      cumulative weight exceeds tau_j = floor((j + u) S / M).  Equivalently
//      particle i fills the slots F(C_{i-1}) .. F(C_i) - 1, F(C) being the
//      number of thresholds below C; each thread computes F at its particles'
//      cumulative weights (a float estimate, settled by an exact 128-bit
//      comparison near integers).  A warp's particles fill one contiguous run
//      of slots, which the warp copies 32 slots at a time (each lane finds its
//      slot's particle by a shuffle search over the lanes' ranges), and after
//      a third barrier every thread reads the states of its own slots.
//      (Staged variants keep the prefix in shared memory and search it instead.)
// A work unit is `count` filters of one job (dataset); units are taken from an
// atomic queue so that jobs of uneven length balance over the SMs.
// With 8 or more particles per thread ("staged"), the log-weights and the
// thread-local prefixes pass through shared memory instead of registers, which
// lets a 512-particle filter run in a single warp: the group reductions become
// warp shuffles and the per-thread costs are shared by 16 particles.
#pragma once
#include <cfloat>
#include <cmath>
#include <type_traits>

#include "binomial.cuh"
#include "common.cuh"
#include "internal.h"
#include "soft64.cuh"

namespace smc2 {

template <typename R>
struct R4Of;
template <>
struct R4Of<float> {
  using type = float4;
};
struct __align__(32) Double4 {
  double x, y, z, w;
};
template <>
struct R4Of<double> {
  using type = Double4;
};

template <int MODEL>
struct ModelDims;
template <>
struct ModelDims<MODEL_LG> {
  static constexpr int D = 3, NS = 1;
};
template <>
struct ModelDims<MODEL_SEIR> {
  static constexpr int D = 4, NS = 4;
};
template <>
struct ModelDims<MODEL_SIR> {
  static constexpr int D = 2, NS = 2;
};

__host__ __device__ inline int group_threads_for(int ppt, int M) {
  const int t = (M + ppt - 1) / ppt;
  return (t + 31) & ~31;
}

// Shared memory of one filter group (Mp = particles incl. padding, nw warps):
//   P  u64 [Mp]      inclusive prefix of the quantised weights (staged: warp-local; variants:
//                    global, for multinomial slots; absent otherwise)
//   X  R   [Mp][ns]  particle states, one vector per particle (per slot after resampling)
//   Xo R   [Mp][ns]  states before resampling, by particle (register-resident variants)
//   Z  R   [4][Mp]   the four normals of the current Philox counter of every particle
//   L  R   [Mp]      log-weights (staged path only)
//   wsum u64 [nw], wmax 8 B [nw], wq2 u128 [nw] (variants: sums of q^2 for the ESS),
//   sU u32 [8] (resampling words of two groups of four steps)
__host__ __device__ constexpr bool is_staged(int ppt) { return ppt >= 8; }
__host__ __device__ inline size_t region_bytes(int Mp, int nw, int ns, int rsize, bool staged,
                                               bool general) {
  size_t b = (size_t)(staged ? 1 : 2) * ns * Mp * rsize + (size_t)4 * Mp * rsize + (size_t)nw * 16 + 32;
  if (staged || general) b += (size_t)Mp * 8;
  if (general) b += (size_t)nw * 16;
  if (staged) b += (size_t)Mp * rsize;
  return (b + 15) & ~(size_t)15;
}

// Register budget per variant (threads x registers must fit the SM at the
// shapes the tuner tries); beyond it the compiler spills to local memory.  The FP64 caps were chosen
// on the SEIR-type model (see run_filter64); under them the SIR model's filter spills 540 to 1580 bytes
// at ppt 2 and 4, which has not been weighed against fewer resident warps.
template <typename R, int PPT>
struct RegCap {
  static constexpr int value =
      sizeof(R) == 4 ? (PPT <= 2 ? 64 : (PPT == 4 ? 96 : (PPT == 8 ? 128 : 168)))
                     : (PPT == 1 ? 128 : PPT <= 4 ? 80 : (PPT == 8 ? 128 : 168));
  static_assert(PPT == 1 || PPT == 2 || PPT == 4 || PPT == 8 || PPT == 16, "particles per thread");
};

template <typename R, int NS>
struct StateVec;
template <typename R>
struct StateVec<R, 1> {
  __device__ __forceinline__ static void store(R* X, int j, const R* x) { X[j] = x[0]; }
  __device__ __forceinline__ static void load(const R* X, int j, R* x) { x[0] = X[j]; }
};
template <>
struct StateVec<float, 2> {
  __device__ __forceinline__ static void store(float* X, int j, const float* x) {
    reinterpret_cast<float2*>(X)[j] = make_float2(x[0], x[1]);
  }
  __device__ __forceinline__ static void load(const float* X, int j, float* x) {
    const float2 v = reinterpret_cast<const float2*>(X)[j];
    x[0] = v.x;
    x[1] = v.y;
  }
};
template <>
struct StateVec<float, 4> {
  __device__ __forceinline__ static void store(float* X, int j, const float* x) {
    reinterpret_cast<float4*>(X)[j] = make_float4(x[0], x[1], x[2], x[3]);
  }
  __device__ __forceinline__ static void load(const float* X, int j, float* x) {
    const float4 v = reinterpret_cast<const float4*>(X)[j];
    x[0] = v.x;
    x[1] = v.y;
    x[2] = v.z;
    x[3] = v.w;
  }
};
template <>
struct StateVec<double, 4> {
  __device__ __forceinline__ static void store(double* X, int j, const double* x) {
    reinterpret_cast<double2*>(X)[2 * j] = make_double2(x[0], x[1]);
    reinterpret_cast<double2*>(X)[2 * j + 1] = make_double2(x[2], x[3]);
  }
  __device__ __forceinline__ static void load(const double* X, int j, double* x) {
    const double2 a = reinterpret_cast<const double2*>(X)[2 * j];
    const double2 b = reinterpret_cast<const double2*>(X)[2 * j + 1];
    x[0] = a.x;
    x[1] = a.y;
    x[2] = b.x;
    x[3] = b.y;
  }
};

template <typename R>
__device__ __forceinline__ R neg_inf();
template <>
__device__ __forceinline__ float neg_inf<float>() {
  return -INFINITY;
}
template <>
__device__ __forceinline__ double neg_inf<double>() {
  return -HUGE_VAL;
}

// floor(v) for a float 0 <= v <= 2^52 as its two 32-bit halves: hi = floor(v 2^-32)
// and lo = floor(v - hi 2^32).  Both steps are exact in float (v 2^-32 is a power-of-
// two scaling; v - hi 2^32 = v mod 2^32 holds at most v's 24 significant bits), and
// the two 32-bit conversions avoid the float-to-u64 one, which runs on the FP64 pipe.
__device__ __forceinline__ uint64_t floor_to_u64(float v) {
  const uint32_t hi = __float2uint_rz(v * 0x1p-32f);
  const float lo = fmaf(-__uint2float_rn(hi), 0x1p32f, v);
  return ((uint64_t)hi << 32) | (uint64_t)__float2uint_rz(lo);
}

// u64 to float from its two 32-bit halves (relative error below 2^-23).
__device__ __forceinline__ float u64_to_float(uint64_t v) {
  return fmaf(__uint2float_rn((uint32_t)(v >> 32)), 0x1p32f, __uint2float_rn((uint32_t)v));
}

// Counting slot thresholds of systematic resampling (Eqs. 26-27) below a
// cumulative weight C: tau_j = floor((2^33 j + 2U + 1) S / (M 2^33)) < C holds
// exactly when (2^33 j + 2U + 1) S < C M 2^33 (both sides below 2^110).
struct SlotCount {
  uint64_t S, M33, U21;  // total, M 2^33, 2U + 1
  float scale, off;      // M / S and (2U + 1) 2^-33 for the float estimate
  float margin;          // bound on the error of the estimate
  int M;
};
__device__ __forceinline__ SlotCount slot_count_setup(uint32_t U, uint64_t S, int M) {
  SlotCount sc;
  sc.S = S;
  sc.M33 = (uint64_t)M << 33;
  sc.U21 = 2ull * U + 1ull;
  sc.scale = __fdividef((float)M, u64_to_float(S));
  sc.off = fmaf(2.f, (float)U, 1.f) * 0x1p-33f;
  sc.margin = fmaf((float)M, 0x1p-18f, 0x1p-16f);
  sc.M = M;
  return sc;
}
// F(C) = #{j in [0, M): tau_j < C} = ceil(C M / S - (2U+1) 2^-33) clamped to
// [0, M].  The crossing point is estimated in float: Cf approximates C to
// about 2^-22 relative, so the estimate is within M 2^-19 of it, inside
// `margin`.  Away from an integer the estimate's ceiling is F; within the
// margin of an integer n (clamped to [0, M - 1]), F is n or n + 1 and one exact
// comparison, tau_n < C, says which.
// Away from integers the estimate lies in (-1, M) (0 <= C <= S), so its ceiling is
// already in [0, M]; only the exact branch clamps.
__device__ __forceinline__ int slots_below(const SlotCount& sc, uint64_t C, float Cf) {
  const float est = fmaf(Cf, sc.scale, -sc.off);
  const float nf = rintf(est);
  if (fabsf(est - nf) > sc.margin) return (int)nf + (est > nf ? 1 : 0);
  int n = min(max((int)nf, 0), sc.M - 1);
  const uint64_t a = ((uint64_t)n << 33) + sc.U21;
  const uint64_t lh = __umul64hi(a, sc.S), ll = a * sc.S;
  const uint64_t rh = __umul64hi(C, sc.M33), rl = C * sc.M33;
  n += (lh < rh || (lh == rh && ll < rl)) ? 1 : 0;
  return n;
}

// slots_below split for a whole warp: the float estimate decides every crossing
// point away from an integer (slots_estimate, which flags the others), and the
// exact 128-bit comparison (slots_exact) settles the flagged ones.
__device__ __forceinline__ int slots_estimate(const SlotCount& sc, float Cf, bool& near) {
  const float est = fmaf(Cf, sc.scale, -sc.off);
  near = !(fabsf(est - rintf(est)) > sc.margin);
  return __float2int_ru(est);  // the ceiling, in one conversion
}
__device__ __forceinline__ int slots_exact(const SlotCount& sc, uint64_t C, float Cf) {
  const float est = fmaf(Cf, sc.scale, -sc.off);
  int n = min(max((int)rintf(est), 0), sc.M - 1);
  const uint64_t a = ((uint64_t)n << 33) + sc.U21;
  const uint64_t lh = __umul64hi(a, sc.S), ll = a * sc.S;
  const uint64_t rh = __umul64hi(C, sc.M33), rl = C * sc.M33;
  return n + ((lh < rh || (lh == rh && ll < rl)) ? 1 : 0);
}

// exp of the FP32 filters: the hardware exp2 approximation (relative error about 2^-22); the FP64
// filters' exponentials are soft64.cuh's.
__device__ __forceinline__ float fast_exp(float x) { return __expf(x); }

// Per-filter constants of the model in the working precision.
template <typename R, int MODEL>
struct FilterParams;

// e^a[0] .. e^a[N - 1], the same in every lane: one evaluation, lane k's argument a[k] (every warp of
// a filter forms them, and an exponential is about 17 FP64 instructions of 19 clocks each).
template <int N>
__device__ __forceinline__ void warp_exps(const double* a, double* out) {
  const int lane = threadIdx.x & 31;
  double v = a[0];
#pragma unroll
  for (int n = 1; n < N; ++n) v = lane == n ? a[n] : v;
  v = exp(v);
#pragma unroll
  for (int n = 0; n < N; ++n) out[n] = __shfl_sync(0xffffffffu, v, n);
}

template <typename R>
struct FilterParams<R, MODEL_LG> {
  R phi, sx, inv_sy, c_obs;
  __device__ void load(const double* th, const PFModel&) {
    double e[2];  // sigma_x, sigma_y
    warp_exps<2>(th + 1, e);
    phi = (R)th[0];
    sx = (R)e[0];
    inv_sy = (R)(1.0 / e[1]);
    c_obs = (R)(-0.5 * kLog2Pi - th[2]);
  }
  __device__ __forceinline__ void init(R* x, R z0, const double*) const { x[0] = z0; }
  __device__ __forceinline__ void propagate(R* x, R z) const { x[0] = phi * x[0] + sx * z; }
  template <typename R4>
  __device__ __forceinline__ R log_obs(const R* x, const R4& ob) const {
    const R r = (ob.x - x[0]) * inv_sy;
    return c_obs - (R)0.5 * r * r;
  }
};

template <typename R>
struct FilterParams<R, MODEL_SEIR> {
  R srw, kappa, gamma, inv_npop, dt, lam_floor, S0, E0, I0, lb0;
  int n_sub;
  __device__ void load(const double* th, const PFModel& m) {
    double e[3];
    warp_exps<3>(th + 1, e);
    lb0 = (R)th[0];
    srw = (R)e[0];
    kappa = (R)e[1];
    gamma = (R)e[2];
    inv_npop = m.inv_npop_f32;
    dt = m.dt_f32;
    n_sub = m.n_sub;
    lam_floor = (R)m.lambda_floor;
    S0 = (R)(m.npop - m.e0 - m.i0);
    E0 = (R)m.e0;
    I0 = (R)m.i0;
  }
  __device__ __forceinline__ void init(R* x, R, const double*) const {
    x[0] = S0;
    x[1] = E0;
    x[2] = I0;
    x[3] = lb0;
  }
  // x = (S, E, I, log beta); the day's incidence lambda is returned in x[4]'s place
  __device__ __forceinline__ void propagate(R* x, R z) const {
    x[3] = x[3] + srw * z;
  }
  __device__ __forceinline__ void substep(R beta, R& S, R& E, R& I, R& lam) const {
    const R infection = beta * S * I * inv_npop;
    const R onset = kappa * E;
    const R recovery = gamma * I;
    lam += dt * onset;
    S = fmax(S - dt * infection, (R)0);
    E = fmax(E + dt * (infection - onset), (R)0);
    I = fmax(I + dt * (onset - recovery), (R)0);
  }
  __device__ __forceinline__ R day(R* x) const {
    const R beta = fast_exp(x[3]);
    R S = x[0], E = x[1], I = x[2], lam = (R)0;
    if (n_sub == 2) {  // the common case, unrolled
      substep(beta, S, E, I, lam);
      substep(beta, S, E, I, lam);
    } else {
      for (int s = 0; s < n_sub; ++s) substep(beta, S, E, I, lam);
    }
    x[0] = S;
    x[1] = E;
    x[2] = I;
    return fmax(lam, lam_floor);
  }
  // Poisson log-pmf written as y (log1p(d) - d) + c_y with d = (lambda - y) / y and
  // c_y = y log y - y - log y! precomputed: no cancellation between y log lambda and lambda.
  template <typename R4>
  __device__ __forceinline__ R log_pois(R lam, const R4& ob) const {
    if (ob.x > (R)0) {
      const R d = (lam - ob.x) * ob.y;
      return ob.x * (log1p(d) - d) + ob.z;
    }
    return -lam;
  }
};

// One day of the SEIR-type dynamics in FP64 instructions, for states and parameters outside
// the range of the fixed-point form below (it recomputes the filter's constants).
struct SeirDay {
  double S, E, I, lam;
};
static __device__ __noinline__ SeirDay seir_day_fp64(SeirDay s, double log_beta, double th2, double th3,
                                                     const PFModel& m) {
  const double beta = exp(log_beta), kappa = exp(th2), gamma = exp(th3);
  const double inv_npop = m.inv_npop, dt = m.dt;
  s.lam = 0.0;
  for (int n = 0; n < m.n_sub; ++n) {
    const double infection = beta * s.S * s.I * inv_npop;
    const double onset = kappa * s.E;
    const double recovery = gamma * s.I;
    s.lam += dt * onset;
    s.S = fmax(s.S - dt * infection, 0.0);
    s.E = fmax(s.E + dt * (infection - onset), 0.0);
    s.I = fmax(s.I + dt * (onset - recovery), 0.0);
  }
  return s;
}

// The Poisson log-pmf y (log1p(d) - d) + c_y, d = (lambda - y) / y (no cancellation between
// y log lambda and lambda), from the observation terms (y, 1/y, c_y, 64-bit mantissa of 1/y).
__device__ __forceinline__ double log_pois64(double lam, const Double4& ob, const Soft64Tables& T) {
  if (!(ob.x > 0.0)) return -lam;
  const uint64_t inv_m = s64_bits(ob.w);
  if (inv_m != 0ull && (uint32_t)(s64_bits(lam) >> 52) - 1u < 2046u) {  // lambda > 0 normal
    bool ok;
    const double g = s64_log1p_minus(lam, inv_m, (int)(s64_bits(ob.y) >> 52) - 1023, T, ok);
    if (ok) return fma(ob.x, g, ob.z);
  }
  const double d = (lam - ob.x) * ob.y;
  return ob.x * (log1p(d) - d) + ob.z;
}

// max(x, 0) of a number
__device__ __forceinline__ double clamp0(double x) { return __double_as_longlong(x) < 0 ? 0.0 : x; }

// The SEIR-type model in FP64: exp(log beta), the products beta S I dt / npop and kappa dt E and
// the sum of E in integers with 64-bit mantissas; the sums of S, I (gamma dt I inside an FMA) and
// lambda on the FP64 pipe, 7 operations a day, so that the two pipes take about as long.  With
// n_sub substeps of dt:
//   S' = S - infection, E' = (E + infection) - kappa dt E, I' = (I + onset) - gamma dt I, all >= 0.
template <>
struct FilterParams<double, MODEL_SEIR> {
  double srw, nkdt, ngdt, lam_floor, S0, E0, I0, lb0, th2, th3;
  uint64_t c_m, k_m;  // mantissas of dt / npop and kappa dt
  int c_e, k_e;       // their exponents
  int n_sub;
  bool tame;          // parameters inside the range of the fixed-point form
  __device__ void load(const double* th, const PFModel& m) {
    lb0 = th[0];
    th2 = th[2];
    th3 = th[3];
    double e[3];
    warp_exps<3>(th + 1, e);
    srw = e[0];
    const double dt = m.dt, kdt = e[1] * dt, gdt = e[2] * dt;
    nkdt = -kdt;
    ngdt = -gdt;
    n_sub = m.n_sub;
    lam_floor = m.lambda_floor;
    S0 = m.npop - m.e0 - m.i0;
    E0 = m.e0;
    I0 = m.i0;
    c_m = s64_unpack(dt / m.npop, c_e);
    k_m = s64_unpack(kdt, k_e);
    // no product overflows or underflows within a day: npop, kappa dt and gamma dt are moderate, and S,
    // which stays non-negative and never grows, starts so (the allocation-free entry point takes
    // e0 + i0 > npop, and s64_unpack wants no sign)
    tame = m.npop > 0x1p-20 && m.npop < 0x1p60 && kdt > 0x1p-100 && kdt < 0x1p20 && gdt < 0x1p20 &&
           S0 >= 0.0 && S0 < 0x1p61;
  }
  __device__ __forceinline__ void init(double* x, double, const double*) const {
    x[0] = S0;
    x[1] = E0;
    x[2] = I0;
    x[3] = lb0;
  }
  __device__ __forceinline__ void propagate(double* x, double z) const { x[3] = fma(srw, z, x[3]); }
  // E as mantissa (leading one at bit 63, or 0) and exponent
  __device__ __forceinline__ void substep(uint64_t bc, int eb, double& S, uint64_t& mE, int& ee, double& I,
                                          double& lam, bool first) const {
    int es, ei;
    const uint64_t mS = s64_unpack(S, es), mI = s64_unpack(I, ei);
    uint64_t p = s64_mulhi(s64_mulhi(bc, mS), mI);  // beta dt / npop (Q61 in [1, 4]) S I: Q59
    int e = eb + es + ei + 3;
    if (!(p >> 61)) {
      p <<= 2;
      e -= 2;
    }
    if (!(p >> 62)) {
      p <<= 1;
      --e;
    }
    if (p == 0ull || e < -1000) {
      p = 0ull;
      e = -1000;
    }
    const double inf = p == 0ull ? 0.0 : s64_pack62(p, e);
    uint64_t o = s64_mulhi(k_m, mE);  // Q62 in [1, 4)
    int eo = k_e + ee;
    if (o >> 63) {
      o >>= 1;
      ++eo;
    }
    if (o == 0ull || eo < -1000) {
      o = 0ull;
      eo = -1000;
    }
    const double onset = o == 0ull ? 0.0 : s64_pack62(o, eo);
    lam = first ? onset : lam + onset;
    S = clamp0(S - inf);
    I = clamp0(fma(ngdt, I, I + onset));
    // E + infection - onset, aligned to the largest of the three (Q61 of it)
    const int em = max(max(e, eo), ee);
    const int64_t v = (int64_t)((mE >> 2) >> min(em - ee, 63)) + (int64_t)((p >> 1) >> min(em - e, 63)) -
                      (int64_t)((o >> 1) >> min(em - eo, 63));
    if (v >= (1ll << 32)) {
      const int lz = s64_clz((uint64_t)v);
      mE = (uint64_t)v << lz;
      ee = em + 2 - lz;
    } else if (v > 0) {  // nearly all of it cancelled
      const int lz = s64_clz((uint64_t)v << 32) + 32;
      mE = (uint64_t)v << lz;
      ee = em + 2 - lz;
    } else {
      mE = 0ull;
      ee = -1000;
    }
  }
  __device__ __forceinline__ double day(double* x, const PFModel& m, const Soft64Tables& T) const {
    double lam;
    // |log beta| < 32, E and I below 2^257
    if (tame && (((uint32_t)(s64_bits(x[3]) >> 52)) & 0x7ffu) < 1023u + 5u &&
        max((uint32_t)(s64_bits(x[1]) >> 32), (uint32_t)(s64_bits(x[2]) >> 32)) < 0x50000000u) {
      int k;
      // e^(log beta) dt / npop: Q62 in [1, 2] times Q63 in [1, 2)
      const uint64_t bc = s64_mulhi(s64_exp_q57(s64_q57(x[3]), T, k) << 1, c_m);
      k += c_e;
      double S = x[0], I = x[2];
      int ee;
      uint64_t mE = s64_unpack(x[1], ee);
      substep(bc, k, S, mE, ee, I, lam, true);
      if (n_sub == 2)
        substep(bc, k, S, mE, ee, I, lam, false);
      else
        for (int s = 1; s < n_sub; ++s) substep(bc, k, S, mE, ee, I, lam, false);
      x[0] = S;
      x[1] = mE == 0ull || ee < -1000 ? 0.0 : s64_pack62(mE >> 1, ee);
      x[2] = I;
    } else {
      const SeirDay d = seir_day_fp64({x[0], x[1], x[2], 0.0}, x[3], th2, th3, m);
      x[0] = d.S;
      x[1] = d.E;
      x[2] = d.I;
      lam = d.lam;
    }
    // max(lambda, floor), both non-negative (a NaN gives the floor)
    return s64_bits(lam) > s64_bits(lam_floor) && s64_bits(lam) <= 0x7ff0000000000000ull ? lam : lam_floor;
  }
};

// The AR(1) model in FP64: three FMA-pipe operations for the log-weight (the halving of r is
// an exponent decrement).
template <>
struct FilterParams<double, MODEL_LG> {
  double phi, sx, inv_sy, c_obs;
  __device__ void load(const double* th, const PFModel&) {
    double e[2];  // sigma_x, sigma_y
    warp_exps<2>(th + 1, e);
    phi = th[0];
    sx = e[0];
    inv_sy = 1.0 / e[1];
    c_obs = -0.5 * kLog2Pi - th[2];
  }
  __device__ __forceinline__ void init(double* x, double z0, const double*) const { x[0] = z0; }
  __device__ __forceinline__ void propagate(double* x, double z) const { x[0] = phi * x[0] + sx * z; }
  __device__ __forceinline__ double log_obs(const double* x, const Double4& ob) const {
    const double r = (ob.x - x[0]) * inv_sy;
    // -r / 2 (0 for |r| < 2^-1021, whose square is 0 too)
    const uint64_t b = s64_bits(r);
    const double h = s64_double((b & 0x7fe0000000000000ull) ? (b ^ 0x8000000000000000ull) - 0x0010000000000000ull : 0ull);
    return fma(r, h, c_obs);
  }
};

// Binomial SIR model (Sec. V-A): theta = (beta, gamma), state (S, I) integers
// held in the working precision (exact below 2^24).  Each day, from the previous
// day's compartments, n(S->I) ~ Bin(S, 1 - exp(-beta I / Npop)) and
// n(I->R) ~ Bin(I, 1 - exp(-gamma)); y_t ~ Poisson(I_t).  (The printed S->I
// probability also carries S_{t-1} in the exponent; this is the per-susceptible
// hazard of the chain-binomial model the section cites.)  Both flows are drawn
// by the binomial sampler of the working precision from particle j's one word
// stream of step t, the I->R draw reading from where the S->I draw stopped.
template <typename R>
struct FilterParams<R, MODEL_SIR> {
  R beta, npop, S0, I0, p_ir;
  __device__ void load(const double* th, const PFModel& m) {
    beta = (R)th[0];
    npop = (R)m.npop;
    p_ir = (R)(-expm1(-th[1]));
    S0 = (R)(m.npop - m.i0);
    I0 = (R)m.i0;
  }
  __device__ __forceinline__ void init(R* x, R, const double*) const {
    x[0] = S0;
    x[1] = I0;
  }
  __device__ __forceinline__ void day(R* x, uint32_t j, uint32_t t, uint32_t c2, uint32_t c3,
                                      uint2 key) const {
    const R S = x[0], I = x[1];
    const R h = beta * I / npop;
    const R p_si = -expm1(-h);
    BinomWordsF b(make_uint4(j, t, c2, c3), key);
    const R n_si = binomial_draw(S, p_si, b);
    const R n_ir = binomial_draw(I, p_ir, b);
    x[0] = S - n_si;
    x[1] = (I + n_si) - n_ir;  // integers: exact in either precision
  }
  // Poisson(y; I) as for the SEIR-type model, with a point mass at 0 when I = 0
  template <typename R4>
  __device__ __forceinline__ R log_obs(const R* x, const R4& ob, const Soft64Tables&) const {
    const R I = x[1];
    if (!(I > (R)0)) return ob.x > (R)0 ? neg_inf<R>() : (R)0;
    if (ob.x > (R)0) {
      const R d = (I - ob.x) * ob.y;
      return ob.x * (log1p(d) - d) + ob.z;
    }
    return -I;
  }
};

// One flow drawn by the FP64 sampler, for the draws that binomial_filtered leaves open.
static __device__ __noinline__ double sir_flow_fp64(double n, double p, double hazard, BinomWords& b) {
  return binomial_draw(n, hazard != 0.0 ? -expm1(-hazard) : p, b);
}

// The same model in FP64.  The draws' decisions come from binomial_filtered, whose probability
// for the S->I flow is 1 - e^(-beta I / npop) in fixed point; draws that it leaves open (one in
// 8000 at npop = 1e4) run the FP64 sampler, whose results all draws have.
// N = 256, M = 500, T = 30: 13.8 ms with every draw by the FP64 sampler (FP64 pipe 85 % busy), 0.90 ms so.
template <>
struct FilterParams<double, MODEL_SIR> {
  double beta, npop, rate, S0, I0, p_ir;  // rate = beta / npop
  uint64_t pq_ir;                         // p_ir in Q63; 0: the flow needs the FP64 sampler
  __device__ void load(const double* th, const PFModel& m) {
    beta = th[0];
    npop = m.npop;
    rate = beta / npop;
    p_ir = -expm1(-th[1]);
    pq_ir = p_ir > 0x1p-30 && p_ir < 1.0 - 0x1p-30 ? (uint64_t)__double2ull_rz(p_ir * 0x1p63) : 0ull;
    S0 = m.npop - m.i0;
    I0 = m.i0;
  }
  __device__ __forceinline__ void init(double* x, double, const double*) const {
    x[0] = S0;
    x[1] = I0;
  }
  __device__ __forceinline__ void day(double* x, uint32_t j, uint32_t t, uint32_t c2, uint32_t c3, uint2 key,
                                      const Soft64Tables& T) const {
    // compartments are integers below 2^24: their low words after adding 2^52
    const uint32_t S = (uint32_t)s64_bits(x[0] + 0x1p52), I = (uint32_t)s64_bits(x[1] + 0x1p52);
    const double h = x[1] * rate;
    uint64_t pq_si = 0ull;
    if (h > 0x1p-40 && h < 20.0) {
      int k;
      const uint64_t e = s64_exp_q57(s64_q57(-h), T, k);  // Q61 2^k, k < 0 (0 next to h = 0)
      pq_si = (1ull << 63) - ((e << 2) >> min(-k, 63));
    }
    BinomWords b(make_uint4(j, t, c2, c3), key);
    uint32_t flow = 0, n_si = 0;
#pragma unroll 1
    for (int f = 0; f < 2; ++f) {
      const uint32_t n = f ? I : S;
      const uint64_t pq = f ? pq_ir : pq_si;
      n_si = flow;
      flow = 0;
      if (n != 0u && (f ? p_ir > 0.0 : h > 0.0)) {
        const BinomWords start = b;
        bool ok = false;
        if (pq != 0ull) flow = binomial_filtered(n, pq, b, ok);
        if (!ok) {
          BinomWords again = start;
          flow = (uint32_t)sir_flow_fp64((double)n, p_ir, f ? 0.0 : beta * x[1] / npop, again);
          b = again;
        }
      }
    }
    x[0] = s64_double(0x4330000000000000ull | (S - n_si)) - 0x1p52;
    x[1] = s64_double(0x4330000000000000ull | (I + n_si - flow)) - 0x1p52;
  }
  __device__ __forceinline__ double log_obs(const double* x, const Double4& ob, const Soft64Tables& T) const {
    const double I = x[1];
    if (!(I > 0.0)) return ob.x > 0.0 ? neg_inf<double>() : 0.0;
    return log_pois64(I, ob, T);
  }
};

// Order-preserving integer key of a number (-inf included), and its inverse: maxima of FP64
// values by integer comparisons, which keeps them off the FP64 pipe.
__device__ __forceinline__ long long order_key(double v) {
  const long long b = __double_as_longlong(v);
  return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ double max_num(double a, double b) { return order_key(a) > order_key(b) ? a : b; }
__device__ __forceinline__ float max_num(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ float warp_max_num(float v) { return warp_max(v); }
__device__ __forceinline__ double warp_max_num(double v) {  // high words, then low words among equal high ones
  const long long k = order_key(v);
  const int hi = (int)(k >> 32);
  const int mh = __reduce_max_sync(0xffffffffu, hi);
  const uint32_t ml = __reduce_max_sync(0xffffffffu, hi == mh ? (uint32_t)k : 0u);
  const long long m = ((long long)mh << 32) | (long long)ml;
  return __longlong_as_double(m ^ ((m >> 63) & 0x7fffffffffffffffll));
}
__device__ __forceinline__ bool is_nan(float v) { return isnan(v); }
__device__ __forceinline__ bool is_nan(double v) {
  return (s64_bits(v) & 0x7fffffffffffffffull) > 0x7ff0000000000000ull;
}

// floor(e^a 2^B) for a = l - max <= 0 (0 below e^-37, where the value is under one)
__device__ __forceinline__ uint64_t quantise64(double a, int B, const Soft64Tables& T) {
  const uint32_t hi = (uint32_t)(s64_bits(a) >> 32);
  int k;
  const uint64_t m = s64_exp_q57(s64_q57(a), T, k);
  // a = 0 or -37 < a < 0; a weight set whose maximum is infinite has no valid a
  return hi == 0u || (hi - 0x80000000u) < 0x40428000u ? m >> min(61 - B - min(k, 0), 63) : 0ull;
}

// A warp's sum of squared weights for the ESS test, c the thread's inclusive prefixes.  The test needs
// the exact 128-bit sum (40 shuffles and adds) only near a tie; a sum of floats, within 2^-20 of it
// (each weight reaches float to 2^-22, the squares and the sums over PPT, 5 and at most 16 terms
// add a rounding each), decides the others.
template <int PPT>
__device__ __forceinline__ void store_q2_float(const uint64_t (&c)[PPT], int lane, float* out) {
  float q2 = 0.f;
  uint64_t prev = 0;
#pragma unroll
  for (int r = 0; r < PPT; ++r) {
    const float q = u64_to_float(c[r] - prev);
    prev = c[r];
    q2 = fmaf(q, q, q2);
  }
  q2 = warp_sum(q2);
  if (lane == 0) *out = q2;
}
__device__ __forceinline__ float total_q2_float(const unsigned __int128* wq2, int nw, int lane) {
  return warp_sum(lane < nw ? *reinterpret_cast<const float*>(wq2 + lane) : 0.f);
}
template <int PPT>
__device__ __forceinline__ void store_q2(const uint64_t (&c)[PPT], int lane, unsigned __int128* out) {
  unsigned __int128 q2 = 0;
  uint64_t prev = 0;
#pragma unroll
  for (int r = 0; r < PPT; ++r) {
    const uint64_t q = c[r] - prev;
    prev = c[r];
    q2 += (unsigned __int128)q * q;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const uint64_t lo = __shfl_xor_sync(0xffffffffu, (uint64_t)q2, o);
    const uint64_t hi = __shfl_xor_sync(0xffffffffu, (uint64_t)(q2 >> 64), o);
    q2 += ((unsigned __int128)hi << 64) | lo;
  }
  if (lane == 0) *out = q2;
}

// NAMED: groups wider than a warp that share a CTA synchronise on named
// barriers 1..15 (ptxas then reserves all 16 barriers of the CTA, which limits
// residency to four CTAs per SM).  Otherwise a wide group is the whole CTA and
// uses __syncthreads, and a one-warp group uses __syncwarp.
template <typename R, int MODEL, int PPT, bool NAMED, bool GENERAL>
__device__ __forceinline__ void run_filter(const PFJob& J, const PFModel& mdl, int i, int g, int lt,
                                           int gt, unsigned char* region, uint2 key, uint32_t k,
                                           int t_cap, const Soft64Tables& tab) {
  constexpr int NS = ModelDims<MODEL>::NS;
  constexpr int D = ModelDims<MODEL>::D;
  constexpr bool F64 = sizeof(R) == 8;
  using R4 = typename R4Of<R>::type;
  const int M = J.M, T = t_cap > 0 ? min(J.T, t_cap) : J.T;
  const int Mp = gt * PPT;
  const int nw = gt >> 5;
  const int lane = lt & 31, warp = lt >> 5;
  const int seg = 32 * PPT;  // particles per warp

  constexpr bool STAGED = is_staged(PPT);
  static_assert(STAGED || !F64, "the FP64 filter of up to four particles per thread is run_filter64");
  constexpr bool GEN = GENERAL && !STAGED;
  uint64_t* P = reinterpret_cast<uint64_t*>(region);   // [Mp] inclusive prefix of q (staged, variants)
  R* X = reinterpret_cast<R*>(P + (STAGED || GEN ? Mp : 0));  // [Mp][NS] particle states
  R* Xo = X + (size_t)NS * Mp;                          // [Mp][NS] states by particle (not staged)
  R* Z = X + (size_t)NS * Mp * (STAGED ? 1 : 2);       // [4][Mp] cached normals
  uint64_t* wsum = reinterpret_cast<uint64_t*>(Z + (size_t)4 * Mp);  // [nw] warp totals
  R* wmax = reinterpret_cast<R*>(wsum + nw);            // [nw] warp maxima (8-byte slots)
  unsigned __int128* wq2 = reinterpret_cast<unsigned __int128*>(wsum + 2 * nw);  // [nw] sums of q^2 (variants)
  uint32_t* sU = reinterpret_cast<uint32_t*>(wsum + (GEN ? 4 : 2) * nw);  // [8] resampling words
  R* Lw = reinterpret_cast<R*>(reinterpret_cast<unsigned char*>(sU) + 32);  // [Mp] staged log-weights

  auto group_sync = [&]() {
    if (nw == 1)
      __syncwarp();
    else if constexpr (NAMED)
      named_barrier(1 + g, gt);
    else
      __syncthreads();
  };

  double th[D];
#pragma unroll
  for (int d = 0; d < D; ++d) th[d] = J.theta[(size_t)d * J.ld + i];
  FilterParams<R, MODEL> fp;
  fp.load(th, mdl);

  const uint32_t c2 = counter_c2((uint32_t)i, J.c2hi);
  const uint32_t c3prop = counter_c3(TAG_PF_PROP, k);
  const uint32_t c3res = counter_c3(TAG_PF_RES, k);
  const uint32_t c3multi = counter_c3(TAG_PF_MULTI, k);
  const uint32_t c3binom = counter_c3(TAG_PF_BINOM, k);
  const int B = fixed_point_bits(M);
  const uint64_t inv_M = STAGED ? slot_reciprocal(M) : 0ull;
  const R scaleB = (R)ldexp(1.0, B);
  const double log_norm = warp == 0 ? -(double)B * kLn2 - log((double)M) : 0.0;  // thread 0's
  const R4* obs = reinterpret_cast<const R4*>(J.obs);

  R x[PPT][NS];
#pragma unroll
  for (int r = 0; r < PPT; ++r) {
    R z0 = (R)0;
    if constexpr (MODEL == MODEL_LG) {
      const uint4 ctr = make_uint4((uint32_t)(lt * PPT + r), 0u, c2, counter_c3(TAG_PF_INIT, k));
      if constexpr (F64) {
        const uint4 w = philox4x32_10(ctr, key);
        double z1;
        s64_normal_pair(w.x, w.y, tab, z0, z1);
      } else {
        R z[4];
        normals4<R>(ctr, key, z);
        z0 = z[0];
      }
    }
    fp.init(x[r], z0, th);
  }

  // Weights (Eq. 5): exp(Lc + lwc_j), Lc the common log weight set by the last
  // resampling (Eq. 13), lwc_j the particle's log factor since (register-resident
  // variants; with resampling every step lwc stays zero).
  // (GENERAL instantiations only: the ESS schedule and multinomial slots; the default
  // instantiations resample systematically every step and keep no factors)
  const bool adaptive = GEN && mdl.pf_ess_frac > 0.0;
  const float ess_thr = (float)(mdl.pf_ess_frac * (double)M);  // mixed precision's ESS threshold
  const bool multinomial = GEN && mdl.pf_scheme == 1;
  R lwc[GEN ? PPT : 1];
#pragma unroll
  for (int r = 0; r < (GEN ? PPT : 1); ++r) lwc[r] = (R)0;
  double Lc = 0.0;
  double loglik = 0.0;  // log p^(y_{1:t}) (Eq. 8)
  for (int t = 1; t <= T; ++t) {
    const int tm = (t - 1) & 3;
    if (F64 && MODEL != MODEL_SIR && tm == 0) {
#pragma unroll 1
      for (int r = 0; r < PPT; ++r) {  // one copy of the long integer code
        const uint4 w = philox4x32_10(make_uint4((uint32_t)(lt * PPT + r), (uint32_t)((t - 1) >> 2), c2, c3prop), key);
        double z0, z1;
        s64_normal_pair(w.x, w.y, tab, z0, z1);
        Z[lt * PPT + r] = (R)z0;
        Z[Mp + lt * PPT + r] = (R)z1;
        s64_normal_pair(w.z, w.w, tab, z0, z1);
        Z[2 * Mp + lt * PPT + r] = (R)z0;
        Z[3 * Mp + lt * PPT + r] = (R)z1;
      }
    }
    if (!F64 && MODEL != MODEL_SIR && tm == 0) {  // one Philox call per particle every four steps; normals kept in shared memory
#pragma unroll
      for (int r = 0; r < PPT; ++r) {
        R z4[4];
        normals4<R>(make_uint4((uint32_t)(lt * PPT + r), (uint32_t)((t - 1) >> 2), c2, c3prop), key,
                    z4);
#pragma unroll
        for (int e = 0; e < 4; ++e) Z[e * Mp + lt * PPT + r] = z4[e];
      }
    }
    // resampling words of steps t..t+3, one lane each, double-buffered by step group
    uint32_t* sUg = sU + 4 * (((t - 1) >> 2) & 1);
    if (tm == 0 && lt < 4 && t + lt < T)
      sUg[lt] = philox4x32_10(make_uint4(0u, (uint32_t)(t + lt), c2, c3res), key).x;
    const R4 ob = obs[t - 1];
    R ell[STAGED ? 1 : PPT];
    R lmax = neg_inf<R>();
#pragma unroll
    for (int r = 0; r < PPT; ++r) {
      R l;
      if constexpr (MODEL == MODEL_SIR) {
        fp.day(x[r], (uint32_t)(lt * PPT + r), (uint32_t)t, c2, c3binom, key);
        l = fp.log_obs(x[r], ob, tab);
      } else if constexpr (MODEL == MODEL_LG) {
        fp.propagate(x[r], Z[tm * Mp + lt * PPT + r]);
        l = fp.log_obs(x[r], ob);
      } else {
        fp.propagate(x[r], Z[tm * Mp + lt * PPT + r]);
        if constexpr (F64)
          l = log_pois64(fp.day(x[r], mdl, tab), ob, tab);
        else
          l = fp.log_pois(fp.day(x[r]), ob);
      }
      if (is_nan(l) || lt * PPT + r >= M) l = neg_inf<R>();
      if constexpr (STAGED) {
        Lw[lt * PPT + r] = l;
      } else {
        if constexpr (GEN) l = lwc[GEN ? r : 0] + l;  // Eq. (5) in logs: the factor since the last resampling
        ell[r] = l;
        StateVec<R, NS>::store(Xo, lt * PPT + r, x[r]);
      }
      lmax = max_num(lmax, l);
    }
    // (3) group maximum
    lmax = warp_max_num(lmax);
    if (nw > 1 && lane == 0) wmax[warp] = lmax;
    group_sync();
    if (nw > 1) lmax = warp_max_num(lane < nw ? wmax[lane] : neg_inf<R>());
    const R m = lmax;
    if (m == neg_inf<R>()) {  // every weight vanished: the estimate is zero
      loglik = -HUGE_VAL;
      if (lt == 0 && J.delta)
        for (int s = t; s <= T; ++s) J.delta[(size_t)i * T + (s - 1)] = -HUGE_VAL;
      break;
    }
    // (4) quantise and scan (warp-local inclusive prefix in P, warp totals in wsum)
    uint64_t run = 0;
    if constexpr (STAGED) {
      // thread-local inclusive prefix into P, then the thread's offset added in place
#pragma unroll
      for (int r = 0; r < PPT; ++r) {
        const R l = Lw[lt * PPT + r];
        if constexpr (F64)
          run += quantise64(l - m, B, tab);
        else
          run += (l > neg_inf<R>()) ? floor_to_u64(fast_exp(l - m) * scaleB) : 0ull;
        P[lt * PPT + r] = run;
        StateVec<R, NS>::store(X, lt * PPT + r, x[r]);
      }
    }
    uint64_t c[STAGED ? 1 : PPT];  // thread-local inclusive prefix of q
    float cf[STAGED ? 1 : PPT];     // the same from the unfloored values, in float
    if constexpr (!STAGED) {
      float runf = 0.f;
#pragma unroll
      for (int r = 0; r < PPT; ++r) {
        const R v = (ell[r] > neg_inf<R>()) ? fast_exp(ell[r] - m) * scaleB : (R)0;
        run += floor_to_u64(v);
        runf += (float)v;
        cf[r] = runf;
        c[r] = run;
      }
    }
    const uint64_t incl = warp_incl_scan_u64(run, lane);
    const uint64_t excl = incl - run;
    if constexpr (STAGED) {
#pragma unroll
      for (int r = 0; r < PPT; ++r) P[lt * PPT + r] += excl;
    }
    if (lane == 31) wsum[warp] = incl;
    if constexpr (GEN) {
      if (adaptive) store_q2_float<PPT>(c, lane, reinterpret_cast<float*>(wq2 + warp));
    }
    group_sync();
    // total S, and the weight `base` of the warps before this one: an inclusive
    // scan of the warp totals across the lanes
    uint64_t wpre = lane < nw ? wsum[lane] : 0ull;
    for (int o = 1; o < nw; o <<= 1) {
      const uint64_t n = __shfl_up_sync(0xffffffffu, wpre, o);
      if (lane >= o) wpre += n;
    }
    const uint64_t S = __shfl_sync(0xffffffffu, wpre, nw - 1);
    const uint64_t base_incl = __shfl_sync(0xffffffffu, wpre, warp > 0 ? warp - 1 : 0);
    const uint64_t base = warp > 0 ? base_incl : 0ull;
    // (5) log-likelihood increment: log S from its binary exponent and mantissa
    // log p^(y_{1:t}) = Lc + log((1/M) sum_j exp(lwc_j + l_j)) from the exact integer total
    // (thread 0 of the group carries Lc and the estimate)
    if (lt == 0) {
      const int e = 63 - __clzll((long long)S);
      const R mant = (R)(e >= 52 ? (S >> (e - 52)) : (S << (52 - e))) * (R)0x1p-52;
      const double lmean = (double)m + ((double)e * kLn2 + (double)log(mant)) + log_norm;
      double delta = lmean;
      if constexpr (GEN) {
        const double logp_prev = loglik;
        loglik = Lc + lmean;
        delta = loglik - logp_prev;
      } else {
        loglik += lmean;
      }
      if (J.delta) J.delta[(size_t)i * T + (t - 1)] = delta;
    }
    // the schedule: every step, or when the ESS of the integer weights (Eq. 12) is below
    // pf_ess_frac M (by lane 0 of every warp, from the same totals, so the whole group decides alike)
    bool resample = t < T;
    if constexpr (GEN) {
      if (adaptive && resample) {
        // the test of Eq. (12) as S^2 < threshold sum q^2, from sums in float; near a tie from the exact sum
        const float Sf = u64_to_float(S), rhs = ess_thr * total_q2_float(wq2, nw, lane);
        resample = Sf * Sf < rhs;
        if (!(fabsf(Sf * Sf - rhs) > 0x1p-16f * rhs)) {
          group_sync();  // the float sums are read
          store_q2<PPT>(c, lane, wq2 + warp);
          group_sync();
          unsigned __int128 Q2 = 0;
          for (int w = 0; w < nw; ++w) Q2 += wq2[w];
          const float q2 = fmaf(__ull2float_rn((uint64_t)(Q2 >> 64)), 0x1p64f, __ull2float_rn((uint64_t)Q2));
          resample = Sf * Sf < ess_thr * q2;
        }
      }
    }
    if constexpr (GEN) {
      if (resample) Lc = loglik;  // Eq. (13): every particle will carry the mean weight (thread 0)
      if (t < T && !resample) {  // every particle keeps its state and its factor
#pragma unroll
        for (int r = 0; r < (GEN ? PPT : 1); ++r) {
          lwc[r] = ell[STAGED ? 0 : r];
          const int j = lt * PPT + r;
          if (J.anc && j < M) J.anc[((size_t)i * (T - 1) + (t - 1)) * M + j] = j;
        }
        continue;
      }
#pragma unroll
      for (int r = 0; r < (GEN ? PPT : 1); ++r) lwc[r] = (R)0;
    }
    if (GEN && resample && multinomial) {
      // slot j draws u_j = (2 U_j + 1) / 2^33 (word j & 3 of call j >> 2) and takes the
      // first particle with C_i > floor(u_j S)
#pragma unroll
      for (int r = 0; r < PPT; ++r) P[lt * PPT + r] = base + excl + c[r];
      group_sync();
      uint4 wj = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
      for (int r = 0; r < PPT; ++r) {
        const int j = lt * PPT + r;
        if (r == 0 || (j & 3) == 0)  // a thread's consecutive slots share their calls
          wj = philox4x32_10(make_uint4((uint32_t)j >> 2, (uint32_t)t, c2, c3multi), key);
        if (j >= M) continue;
        const uint32_t Uj = (j & 2) ? ((j & 1) ? wj.w : wj.z) : ((j & 1) ? wj.y : wj.x);
        const uint64_t tau = (uint64_t)(((unsigned __int128)(2ull * Uj + 1ull) * S) >> 33);
        int lo = 0, hi = M - 1;
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (P[mid] > tau)
            hi = mid;
          else
            lo = mid + 1;
        }
        StateVec<R, NS>::load(Xo, lo, x[r]);
        if (J.anc) J.anc[((size_t)i * (T - 1) + (t - 1)) * M + j] = lo;
      }
      group_sync();  // P and Xo free for the next step
      continue;
    }
    // (6) systematic resampling and ancestor gather.  The thread's slots are
    // consecutive and their ancestors non-decreasing: the first is found by a
    // search over the warp totals and a binary search inside one warp's prefix,
    // the others by galloping forward from the previous ancestor.
    if (!STAGED && t < T) {
      const SlotCount sc = slot_count_setup(sUg[tm], S, M);
      const uint64_t C0 = base + excl;  // cumulative weight before the thread's first particle
      const float C0f = u64_to_float(C0);
      int ends[PPT];
#pragma unroll
      for (int r = 0; r < PPT; ++r) ends[r] = slots_below(sc, C0 + c[r], C0f + cf[r]);
      // the warp's particles fill the slots [first, last), in particle order
      const int first = __shfl_sync(0xffffffffu, slots_below(sc, C0, C0f), 0);
      const int last = __shfl_sync(0xffffffffu, ends[PPT - 1], 31);
      const int pbase = warp * 32 * PPT;  // the warp's first particle
      __syncwarp();                       // the warp's states in Xo
      for (int j0 = first; j0 < last; j0 += 32) {
        const int j = j0 + lane;
        // the lane whose particles cover slot j: the lanes whose ranges end at or before j
        int src = 0;
#pragma unroll
        for (int step = 16; step >= 1; step >>= 1) {
          const int e = __shfl_sync(0xffffffffu, ends[PPT - 1], src + step - 1);
          if (e <= j) src += step;
        }
        src = min(src, 31);
        int rr = 0;
#pragma unroll
        for (int r = 0; r < PPT - 1; ++r) rr += __shfl_sync(0xffffffffu, ends[r], src) <= j ? 1 : 0;
        if (j < last) {
          const int a = pbase + src * PPT + rr;
          R v[NS];
          StateVec<R, NS>::load(Xo, a, v);
          StateVec<R, NS>::store(X, j, v);
          if (J.anc) J.anc[((size_t)i * (T - 1) + (t - 1)) * M + j] = a;
        }
      }
      group_sync();
#pragma unroll
      for (int r = 0; r < PPT; ++r)
        if (lt * PPT + r < M) StateVec<R, NS>::load(X, lt * PPT + r, x[r]);
    }
    if (STAGED && t < T) {
      const uint32_t U = sUg[tm];
      int w = 0, a = 0;
      uint64_t base = 0;
#pragma unroll
      for (int r = 0; r < PPT; ++r) {
        const int j = lt * PPT + r;
        if (j < M) {
          const uint64_t tau = slot_threshold((uint32_t)j, U, S, M, inv_M);
          while (w < nw - 1 && base + wsum[w] <= tau) {  // answer lies in a later warp
            base += wsum[w];
            ++w;
            a = w * seg;
          }
          const uint64_t tl = tau - base;
          const int seg_end = w * seg + seg - 1;  // P[seg_end] = wsum[w] > tl
          if (r == 0) {
            int lo = w * seg, hi = seg_end;
            while (lo < hi) {
              const int mid = (lo + hi) >> 1;
              if (P[mid] > tl)
                hi = mid;
              else
                lo = mid + 1;
            }
            a = lo;
          } else if (P[a] <= tl) {
            int lo = a + 1, step = 1;
            while (lo + step - 1 < seg_end && P[lo + step - 1] <= tl) {
              lo += step;
              step <<= 1;
            }
            int hi = min(lo + step - 1, seg_end);
            while (lo < hi) {
              const int mid = (lo + hi) >> 1;
              if (P[mid] > tl)
                hi = mid;
              else
                lo = mid + 1;
            }
            a = lo;
          }
          StateVec<R, NS>::load(X, a, x[r]);
          if (J.anc) J.anc[((size_t)i * (T - 1) + (t - 1)) * M + j] = a;
        }
      }
    }
  }
  if (lt == 0) J.loglik[i] = loglik;
}

// The FP64 filter with up to four particles per thread (M <= 2048): pf_kernel's filter with its
// long integer functions (soft64.cuh) in loops over the thread's particles that are not
// unrolled, and every per-particle value in shared memory.  The loop bodies are 100 to 1000
// instructions, so a shared load and store cost them nothing, one copy of each keeps the
// instruction cache, and a thread holds few registers whatever its particle count: the kernel is
// bound by latency (the FP64 pipe's and its own dependent integer chains'), which more resident
// warps hide.  SEIR, N = 1024, M = 512, T = 100: 15.4 ms with the math library's functions and
// states in registers (FP64 pipe 85 % busy), 3.35 ms with soft64.cuh in that form, 2.80 ms in
// this form, 2.54 ms with E's sum and the far log-weights in integers too (issue 60 %, ALU pipe
// 61 %, FP64 pipe 48 %); 80 registers (64: 2.61 ms, 96: 3.05 ms).
// Per-particle arrays keep particle (or slot) s at row s % PPT, column s / PPT, so that a warp
// reading one entry per thread touches consecutive words:
//   X    2 x [NS][Mp] double  states: step t reads buffer (t - 1) & 1 through the ancestors and
//                             writes the other, so no copy and no barrier lies between
//   Z    [4][Mp] double       the normals of four steps; a step's row then holds its log-weights
//                             and quantised weights (LG and SEIR)
//   L    [Mp] double          log-weights where they outlive the step (variants) or Z is absent (SIR)
//   P    [Mp] u64             quantised weights of the SIR variants
//   mark [Mp] u16, carry [T] u16   ancestors: see below
//   wsum u64, wmax double, wq2 u128 (variants) per warp; sU u32 [8]
// Resampling marks ancestors (Algorithm 1's order) as the FP32 filter does: particle i fills the
// slots F(C_{i-1}) .. F(C_i) - 1; it writes its index at its first slot and as the carry of every
// thread whose first slot it covers, and the ancestor of a slot is the largest index at or before
// it among the thread's slots (empty marks are 0, and the reader clears them).
template <int MODEL, bool GENERAL>
struct Region64 {
  static constexpr int NS = ModelDims<MODEL>::NS;
  static constexpr bool kZ = MODEL != MODEL_SIR;
  static constexpr bool kL = GENERAL || !kZ, kP = GENERAL && !kZ;
};
__host__ __device__ inline size_t region64_bytes(int Mp, int T, int ns, bool sir, bool general) {
  size_t b = (size_t)2 * ns * Mp * 8 + (sir ? 0 : (size_t)4 * Mp * 8);
  if (general || sir) b += (size_t)Mp * 8;
  if (general && sir) b += (size_t)Mp * 8;
  b += (size_t)(T >> 5) * (general ? 32 : 16) + 32;
  b += (size_t)Mp * 2 + (size_t)T * 2;
  return (b + 15) & ~(size_t)15;
}

template <int MODEL, int PPT, bool NAMED, bool GENERAL>
__device__ __forceinline__ void run_filter64(const PFJob& J, const PFModel& mdl, int i, int g, int lt, int T,
                                             unsigned char* region, uint2 key, uint32_t k, int t_cap,
                                             const Soft64Tables& tab) {
  using Rg = Region64<MODEL, GENERAL>;
  constexpr int NS = Rg::NS, D = ModelDims<MODEL>::D;
  constexpr int LOG2P = PPT == 1 ? 0 : (PPT == 2 ? 1 : 2);
  const int M = J.M, TT = t_cap > 0 ? min(J.T, t_cap) : J.T;
  const int Mp = T * PPT, nw = T >> 5, lane = lt & 31, warp = lt >> 5;
  double* X = reinterpret_cast<double*>(region);
  double* Z = X + (size_t)2 * NS * Mp;
  double* La = Z + (Rg::kZ ? (size_t)4 * Mp : 0);
  uint64_t* Pa = reinterpret_cast<uint64_t*>(La + (Rg::kL ? Mp : 0));
  unsigned __int128* wq2 = reinterpret_cast<unsigned __int128*>(Pa + (Rg::kP ? Mp : 0));  // [nw] sums of q^2
  uint64_t* wsum = reinterpret_cast<uint64_t*>(wq2 + (GENERAL ? nw : 0));                  // [nw]
  double* wmax = reinterpret_cast<double*>(wsum + nw);                                     // [nw]
  uint32_t* sU = reinterpret_cast<uint32_t*>(wmax + nw);                                   // [8]
  uint16_t* mark = reinterpret_cast<uint16_t*>(sU + 8);                                    // [Mp]
  uint16_t* carry = mark + Mp;                                                             // [T]

  auto group_sync = [&]() {
    if (nw == 1)
      __syncwarp();
    else if constexpr (NAMED)
      named_barrier(1 + g, T);
    else
      __syncthreads();
  };

  double th[D];
#pragma unroll
  for (int d = 0; d < D; ++d) th[d] = J.theta[(size_t)d * J.ld + i];
  FilterParams<double, MODEL> fp;
  fp.load(th, mdl);
  const uint32_t c2 = counter_c2((uint32_t)i, J.c2hi);
  const uint32_t c3prop = counter_c3(TAG_PF_PROP, k);
  const uint32_t c3res = counter_c3(TAG_PF_RES, k);
  const uint32_t c3multi = counter_c3(TAG_PF_MULTI, k);
  const uint32_t c3binom = counter_c3(TAG_PF_BINOM, k);
  const int B = fixed_point_bits(M);
  const Double4* obs = reinterpret_cast<const Double4*>(J.obs);
#pragma unroll 1
  for (int r = 0; r < PPT; ++r) {
    const int pos = r * T + lt;
    double x[NS], z0 = 0.0, z1;
    if constexpr (MODEL == MODEL_LG) {
      const uint4 w = philox4x32_10(
          make_uint4((uint32_t)(lt * PPT + r), 0u, c2, counter_c3(TAG_PF_INIT, k)), key);
      s64_normal_pair(w.x, w.y, tab, z0, z1);
    }
    fp.init(x, z0, th);
#pragma unroll
    for (int e = 0; e < NS; ++e) X[(size_t)e * Mp + pos] = x[e];
    mark[pos] = 0;
  }
  carry[lt] = 0;  // threads whose slots are all padding keep this valid ancestor (particle 0)

  // Weights (Eq. 5): exp(Lc + l_j), Lc the common log weight set by the last resampling (Eq. 13)
  const bool adaptive = GENERAL && mdl.pf_ess_frac > 0.0;
  const float ess_thr = (float)(mdl.pf_ess_frac * (double)M);
  const bool multinomial = GENERAL && mdl.pf_scheme == 1;
  double Lc = 0.0, loglik = 0.0;  // log p^(y_{1:t}) (Eq. 8)
  bool dead = false;
  int from = 0;  // where the next step's states come from: 0 their own slot, 1 the marks, 2 mark[] as it stands
  // Likelihood increments: lane (t - 1) % 32 of the group's first warp keeps step t's maximum and
  // total, and every 32 steps the lanes take their logarithms side by side and are summed (a
  // logarithm by one lane each step would cost that warp its full time).
  double inc_m = 0.0;
  uint64_t inc_S = 1;
  bool inc_res = false;
  auto add_increments = [&](int t_last) {  // the n = (t_last - 1) % 32 + 1 steps up to t_last
    if (warp != 0 || t_last < 1) return;
    const int n = ((t_last - 1) & 31) + 1, t0 = t_last - n;
    // max + log(S 2^-B) - log M, log S from its binary exponent and mantissa
    const int e = 63 - __clzll((long long)inc_S);
    const double mant = (double)(e >= 52 ? (inc_S >> (e - 52)) : (inc_S << (52 - e))) * 0x1p-52;
    const double lmean = lane < n ? inc_m + ((double)e * kLn2 + log(mant)) + (-(double)B * kLn2 - log((double)M)) : 0.0;
    if constexpr (GENERAL) {
      // Eq. (13): a resampling step's estimate is the common weight from there on, so the steps since
      // the last one are replaced by the latest
      const uint32_t res = __ballot_sync(0xffffffffu, inc_res && lane < n);
      if (J.delta) {  // estimates after each step: the increments of the resampling steps before it
        double before = Lc, prev = loglik;
        for (int s = 0; s < n; ++s) {
          const double v = before + __shfl_sync(0xffffffffu, lmean, s);
          if (lane == 0) J.delta[(size_t)i * TT + t0 + s] = v - prev;
          prev = v;
          if (res & (1u << s)) before = v;
        }
      }
      const double last = __shfl_sync(0xffffffffu, lmean, n - 1);
      Lc += warp_sum((res >> lane) & 1u ? lmean : 0.0);
      loglik = (res >> (n - 1)) & 1u ? Lc : Lc + last;
    } else {
      if (J.delta && lane < n) J.delta[(size_t)i * TT + t0 + lane] = lmean;
      loglik += warp_sum(lmean);
    }
  };
  Double4 ob_next = obs[0];

  for (int t = 1; t <= TT; ++t) {
    if (((t - 1) & 31) == 0) add_increments(t - 1);
    const int tm = (t - 1) & 3;
    const double* Xin = X + (size_t)((t - 1) & 1) * NS * Mp;
    double* Xout = X + (size_t)(t & 1) * NS * Mp;
    double* Lr = Rg::kL ? La : Z + (size_t)tm * Mp;
    uint64_t* Q = Rg::kP ? Pa : (Rg::kL && !Rg::kZ ? reinterpret_cast<uint64_t*>(La)
                                                   : reinterpret_cast<uint64_t*>(Z + (size_t)tm * Mp));
    // (1), (2) propagate (Eq. 1) and log-weight (Eq. 2) the particles
    uint32_t* sUg = sU + 4 * (((t - 1) >> 2) & 1);  // resampling words of four steps
    if (tm == 0 && lt < 4 && t + lt < TT)
      sUg[lt] = philox4x32_10(make_uint4(0u, (uint32_t)(t + lt), c2, c3res), key).x;
    const Double4 ob = PPT == 1 ? ob_next : obs[t - 1];
    if (PPT == 1) ob_next = obs[min(t, TT - 1)];  // in flight during the step
    double lmax = neg_inf<double>();
    uint32_t a = carry[lt];
#pragma unroll 1
    for (int r = 0; r < PPT; ++r) {
      const int j = lt * PPT + r, pos = r * T + lt;
      if (Rg::kZ && tm == 0) {  // one Philox call every four steps
        const uint4 w = philox4x32_10(make_uint4((uint32_t)j, (uint32_t)((t - 1) >> 2), c2, c3prop), key);
#pragma unroll (PPT == 1 ? 2 : 1)
        for (int h = 0; h < 2; ++h) {  // the two pairs side by side where few warps are resident
          double z0, z1;
          s64_normal_pair(h ? w.z : w.x, h ? w.w : w.y, tab, z0, z1);
          Z[(size_t)(2 * h) * Mp + pos] = z0;
          Z[(size_t)(2 * h + 1) * Mp + pos] = z1;
        }
      }
      int src = j;
      if (!GENERAL ? t > 1 : from != 0) {
        const uint32_t mk = mark[pos];
        if (!GENERAL || from == 1) {
          a = max(a, mk);
          src = (int)a;
          mark[pos] = 0;
        } else {
          src = (int)mk;
        }
      }
      if (J.anc && t > 1 && j < M) J.anc[((size_t)i * (TT - 1) + (t - 2)) * M + j] = src;
      const int spos = (src & (PPT - 1)) * T + (src >> LOG2P);
      double x[NS], l;
#pragma unroll
      for (int e = 0; e < NS; ++e) x[e] = Xin[(size_t)e * Mp + spos];
      if constexpr (MODEL == MODEL_SIR) {
        fp.day(x, (uint32_t)j, (uint32_t)t, c2, c3binom, key, tab);
        l = fp.log_obs(x, ob, tab);
      } else {
        fp.propagate(x, Z[(size_t)tm * Mp + pos]);
        if constexpr (MODEL == MODEL_LG)
          l = fp.log_obs(x, ob);
        else
          l = log_pois64(fp.day(x, mdl, tab), ob, tab);
      }
#pragma unroll
      for (int e = 0; e < NS; ++e) Xout[(size_t)e * Mp + pos] = x[e];
      if (is_nan(l) || j >= M) l = neg_inf<double>();
      if (adaptive && from == 0 && t > 1) l = Lr[pos] + l;  // Eq. (5) in logs: the factor since the last resampling
      Lr[pos] = l;
      lmax = max_num(lmax, l);
    }
    // (3) group maximum
    lmax = warp_max_num(lmax);
    if (nw > 1 && lane == 0) wmax[warp] = lmax;
    group_sync();
    // Up to four warps' maxima and totals are combined by every thread from the same words, which is
    // shorter than the reduction and the scan over the lanes that more warps take: where one particle per
    // thread leaves each step to latency (LG run, N=64/M=128/T=50/K=10: 1.397 -> 1.369 ms; with more
    // particles per thread no difference)
    const bool few = PPT == 1 && nw <= 4;
    if (few)
      lmax = nw > 1 ? max_num(max_num(wmax[0], wmax[1]), max_num(wmax[nw > 2 ? 2 : 0], wmax[nw > 3 ? 3 : 0])) : lmax;
    else if (nw > 1)
      lmax = warp_max_num(lane < nw ? wmax[lane] : neg_inf<double>());
    const double m = lmax;
    if (m == neg_inf<double>()) {  // every weight vanished: the estimate is zero
      if (((t - 1) & 31) != 0) add_increments(t - 1);
      loglik = -HUGE_VAL;
      dead = true;
      if (lt == 0 && J.delta)
        for (int s = t; s <= TT; ++s) J.delta[(size_t)i * TT + (s - 1)] = -HUGE_VAL;
      break;
    }
    // (4) quantise and scan
#pragma unroll 1
    for (int r = 0; r < PPT; ++r) Q[r * T + lt] = quantise64(Lr[r * T + lt] - m, B, tab);
    uint64_t c[PPT];  // thread-local inclusive prefix
    uint64_t run = 0;
#pragma unroll
    for (int r = 0; r < PPT; ++r) {
      run += Q[r * T + lt];
      c[r] = run;
    }
    const uint64_t incl = warp_incl_scan_u64(run, lane);
    const uint64_t excl = incl - run;
    if (lane == 31) wsum[warp] = incl;
    if (adaptive) store_q2_float<PPT>(c, lane, reinterpret_cast<float*>(wq2 + warp));
    group_sync();
    // total S, and the weight `base` of the warps before this one
    uint64_t S, C0 = excl;  // C0: weight before the thread's first particle
    if (few) {
      const uint64_t w0 = wsum[0], p2 = w0 + (nw > 1 ? wsum[1] : 0ull), p3 = p2 + (nw > 2 ? wsum[2] : 0ull);
      S = p3 + (nw > 3 ? wsum[3] : 0ull);
      C0 += warp == 0 ? 0ull : (warp == 1 ? w0 : (warp == 2 ? p2 : p3));
    } else {
      uint64_t wpre = lane < nw ? wsum[lane] : 0ull;
      for (int o = 1; o < nw; o <<= 1) {
        const uint64_t n = __shfl_up_sync(0xffffffffu, wpre, o);
        if (lane >= o) wpre += n;
      }
      S = __shfl_sync(0xffffffffu, wpre, nw - 1);
      const uint64_t base_incl = __shfl_sync(0xffffffffu, wpre, warp > 0 ? warp - 1 : 0);
      C0 += warp > 0 ? base_incl : 0ull;
    }
    // (5) likelihood increment (Eq. 8): see add_increments
    const bool mine = lane == ((t - 1) & 31);
    inc_m = mine ? m : inc_m;
    inc_S = mine ? S : inc_S;
    // the schedule: every step, or when the ESS of the integer weights (Eq. 12) is below
    // pf_ess_frac M: from sums in float, and near a tie from the exact sum of q^2 with the same
    // correctly rounded operations as the oracle (the whole group sees the same totals)
    bool resample = t < TT;
    if (adaptive && resample) {
      const float Sf = u64_to_float(S), rhs = ess_thr * total_q2_float(wq2, nw, lane);
      resample = Sf * Sf < rhs;
      if (!(fabsf(Sf * Sf - rhs) > 0x1p-16f * rhs)) {
        group_sync();  // the float sums are read
        store_q2<PPT>(c, lane, wq2 + warp);
        group_sync();
        unsigned __int128 Q2 = 0;
        for (int w = 0; w < nw; ++w) Q2 += wq2[w];
        const double q2 = (double)(uint64_t)(Q2 >> 64) * 0x1p64 + (double)(uint64_t)Q2;
        const double ess = __ddiv_rn((double)S * (double)S, q2);
        resample = ess < mdl.pf_ess_frac * (double)M;
      }
    }
    inc_res = mine ? resample : inc_res;
    from = resample ? (multinomial ? 2 : 1) : 0;
    if (!resample) continue;
    if (multinomial) {
      // slot j draws u_j = (2 U_j + 1) / 2^33 (word j & 3 of call j >> 2) and takes the
      // first particle with C_i > floor(u_j S)
#pragma unroll
      for (int r = 0; r < PPT; ++r) Q[r * T + lt] = C0 + c[r];
      group_sync();
      uint4 wj = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
      for (int r = 0; r < PPT; ++r) {
        const int j = lt * PPT + r;
        if (r == 0 || (j & 3) == 0)  // a thread's consecutive slots share their calls
          wj = philox4x32_10(make_uint4((uint32_t)j >> 2, (uint32_t)t, c2, c3multi), key);
        if (j >= M) continue;  // padding slots keep an earlier ancestor
        const uint32_t Uj = (j & 2) ? ((j & 1) ? wj.w : wj.z) : ((j & 1) ? wj.y : wj.x);
        const uint64_t tau = (uint64_t)(((unsigned __int128)(2ull * Uj + 1ull) * S) >> 33);
        int lo = 0, hi = M - 1;
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (Q[(mid & (PPT - 1)) * T + (mid >> LOG2P)] > tau)
            hi = mid;
          else
            lo = mid + 1;
        }
        mark[r * T + lt] = (uint16_t)lo;
      }
      group_sync();  // Q is free: the next step may write new normals over it
      continue;
    }
    // (6) systematic resampling by marks: every crossing from the float estimate, whose error is
    // under 17 M u + 2 u (u = 2^-24: S, C0 and the thread's share reach float through two
    // roundings each, M / S adds 4 u, the sum and the fma 1 u each, the offset 2 u absolute),
    // covered by M 2^-19 + 2^-20; those near an integer by the exact comparison
    SlotCount sc = slot_count_setup(sUg[tm], S, M);
    sc.margin = fmaf((float)M, 0x1p-19f, 0x1p-20f);
    const float C0f = u64_to_float(C0);
    int ends[PPT + 1];
    uint32_t near_mask = 0;
#pragma unroll
    for (int r = 0; r <= PPT; ++r) {
      bool nr;
      ends[r] = slots_estimate(sc, r == 0 ? C0f : C0f + u64_to_float(c[r - 1]), nr);
      near_mask |= nr ? (1u << r) : 0u;
    }
    if (__any_sync(0xffffffffu, near_mask != 0)) {
#pragma unroll
      for (int r = 0; r <= PPT; ++r)
        if (near_mask & (1u << r))
          ends[r] = slots_exact(sc, r == 0 ? C0 : C0 + c[r - 1], r == 0 ? C0f : C0f + u64_to_float(c[r - 1]));
    }
#pragma unroll
    for (int r = 0; r < PPT; ++r) {
      const int start = ends[r], end = ends[r + 1];
      const uint16_t id = (uint16_t)(lt * PPT + r);
      if (end > start) mark[(start & (PPT - 1)) * T + (start >> LOG2P)] = id;
      // the first slot of every thread inside [start, end)
      for (int b = (start + PPT - 1) & ~(PPT - 1); b < end; b += PPT) carry[b >> LOG2P] = id;
    }
    group_sync();
  }
  if (!dead) add_increments(TT);
  if (lt == 0) J.loglik[i] = loglik;
  group_sync();  // the region is free for the next filter
}

// The tables of soft64.cuh as a kernel reads them: a copy in shared memory, or in the staged
// FP64 variants, whose particles may need all of it, the device arrays.
template <bool SHARED>
__device__ __forceinline__ const Soft64Tables& soft64_tables() {
  if constexpr (SHARED) {
    __shared__ __align__(16) Soft64Tables s;
    static_assert(sizeof(Soft64Tables) % 16 == 0, "copied by 16-byte words");
    const uint4* from = reinterpret_cast<const uint4*>(&g_soft64);
    uint4* to = reinterpret_cast<uint4*>(&s);
    for (int w = threadIdx.x; w < (int)(sizeof(Soft64Tables) / 16); w += blockDim.x) to[w] = from[w];
    __syncthreads();
    return s;
  } else {
    return g_soft64;
  }
}

template <typename R, int MODEL, int PPT, bool NAMED, bool GENERAL>
__global__ void __maxnreg__((RegCap<R, PPT>::value)) pf_kernel(PFLaunch L) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_wu;
  const Soft64Tables& tab = soft64_tables<sizeof(R) == 8 && !is_staged(PPT)>();
  constexpr int NS = ModelDims<MODEL>::NS;
  const uint32_t k = L.k_done ? (uint32_t)(*L.k_done + 1) : (uint32_t)L.k_imm;
  const uint2 key = seed_key(L.seed);
  for (int it = 0;; ++it) {
    int w;
    if (L.wu_counter) {
      __syncthreads();
      if (threadIdx.x == 0) s_wu = atomicAdd(L.wu_counter, 1);
      __syncthreads();
      w = s_wu;
    } else {
      w = blockIdx.x + it * gridDim.x;
    }
    if (w >= L.n_wu) break;
    int job, first, count;
    if (L.wus) {
      const int4 u = L.wus[w];
      job = u.x;
      first = u.y;
      count = u.z;
    } else {
      job = 0;
      first = w * L.fpc_single;
      count = min(L.fpc_single, L.job0.n - first);
    }
    const PFJob J = L.jobs ? L.jobs[job] : L.job0;
    const int gt = group_threads_for(PPT, J.M);
    const int g = threadIdx.x / gt, lt = threadIdx.x - g * gt;
    if constexpr (sizeof(R) == 8 && !is_staged(PPT)) {
      const size_t rb = region64_bytes(gt * PPT, gt, NS, MODEL == MODEL_SIR, GENERAL);
      if (g < count && (g + 1) * gt <= (int)blockDim.x)
        run_filter64<MODEL, PPT, NAMED, GENERAL>(J, L.mdl, first + g, g, lt, gt, smem + g * rb, key, k, L.t_cap, tab);
    } else {
      const size_t rb = region_bytes(gt * PPT, gt >> 5, NS, (int)sizeof(R), is_staged(PPT), GENERAL);
      if (g < count && (g + 1) * gt <= (int)blockDim.x)
        run_filter<R, MODEL, PPT, NAMED, GENERAL>(J, L.mdl, first + g, g, lt, gt, smem + g * rb, key, k, L.t_cap, tab);
    }
    if (!L.wu_counter) __syncthreads();
  }
  release_queue(L.wu_counter);
}


template <typename R, int MODEL, int PPT, bool NAMED, bool GENERAL>
const void* pf_kernel_ptr() {
  return reinterpret_cast<const void*>(&pf_kernel<R, MODEL, PPT, NAMED, GENERAL>);
}

// The GENERAL instantiations exist for the register-resident shapes only.
template <typename R, int MODEL, bool NAMED, bool GENERAL>
const void* pf_select_ppt(int ppt) {
  switch (ppt) {
    case 1: return pf_kernel_ptr<R, MODEL, 1, NAMED, GENERAL>();
    case 2: return pf_kernel_ptr<R, MODEL, 2, NAMED, GENERAL>();
    case 4: return pf_kernel_ptr<R, MODEL, 4, NAMED, GENERAL>();
    case 8:  // the variants and the SIR model run in the register-resident shapes only
      if constexpr (GENERAL || MODEL == MODEL_SIR) return nullptr;
      else return pf_kernel_ptr<R, MODEL, 8, NAMED, false>();
    case 16:
      if constexpr (GENERAL || MODEL == MODEL_SIR) return nullptr;
      else return pf_kernel_ptr<R, MODEL, 16, NAMED, false>();
    default: return nullptr;
  }
}

template <typename R, bool GENERAL>
const void* pf_select_precision(int model, int ppt, bool named) {
  if (model == MODEL_LG)
    return named ? pf_select_ppt<R, MODEL_LG, true, GENERAL>(ppt) : pf_select_ppt<R, MODEL_LG, false, GENERAL>(ppt);
  return named ? pf_select_ppt<R, MODEL_SEIR, true, GENERAL>(ppt) : pf_select_ppt<R, MODEL_SEIR, false, GENERAL>(ppt);
}

template <typename R, bool GENERAL>
const void* pf_select_sir(int ppt, bool named) {
  return named ? pf_select_ppt<R, MODEL_SIR, true, GENERAL>(ppt) : pf_select_ppt<R, MODEL_SIR, false, GENERAL>(ppt);
}

const void* pf_select_f32(int model, int ppt, bool named);
const void* pf_select_f64(int model, int ppt, bool named);
const void* pf_select_general_f32(int model, int ppt, bool named);
const void* pf_select_general_f64(int model, int ppt, bool named);
// the SIR model's instantiations (pf_sir_f32.cu, pf_sir_f64.cu)
const void* pf_select_sir_f32(int ppt, bool named, bool general);
const void* pf_select_sir_f64(int ppt, bool named, bool general);

}  // namespace smc2
