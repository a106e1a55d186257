// Persistent radial-step kernel of the bulb model (arXiv:1912.10596, Sec. 2 and Sec. 3.4).
//
// One cooperative launch advances every active instance by up to n_steps radial steps.  A step is a
// sequence of passes over all beams separated by device-wide barriers, because every stage of the
// integrator needs the angular moments of *all* beams (Eq. Hnu / Eq. F):
//
//   pass p (p = 0 .. S-2): form the stage state Y_{p+2} of every beam from the step's initial
//       state y and the stage derivatives k_1..k_{p+1}, and reduce the moments of Y_{p+2}.  FP32
//       kernels recompute k_1..k_{p+1} in registers from y and the earlier stages' constants (the
//       stage vectors are not stored); FP64 RK4 / DP45 kernels read k_1..k_p and Y_{p+1} back from
//       HBM planes and evaluate only k_{p+1} (stored_stages);
//   final pass: form the new state (and, for DP45, the embedded error), write it to the second
//       state buffer and reduce either the moments of the new state (fixed step) or the error norm
//       (DP45).
//
// So every pass reads each beam's state once (vector loads of the SoA planes, or the per-thread
// cp.async ring of the FP32 two-flavour bulb kernels) and a step writes it once; the FP64 kernels
// also move their stage planes.  The exponential integrators (commutator-free Lie RK4, the
// exponential midpoint rule, the adaptive Lie RK4 with Richardson control) build every stage state
// from y by exact propagators exp(-i Om) y exp(i Om) of Eq. U instead: a rotation of the Bloch
// vector for two flavours, a closed form of the 3 x 3 exponential for three (propagate3).
//
// Moments without cancellation.  With the measure of Eq. Hnu in u-bins, the nu-nu term of beam b is
// mu(r) (J0 - cos(th_b) J1), J0 = sum w s / cos(th), J1 = sum w s.  Far from the neutrino sphere
// J0 and J1 agree to O(R^2/r^2) and the difference cancels catastrophically in FP32.  The kernel
// therefore reduces J1 and D = J0 - J1 = sum w s (1/cos(th) - 1), and assembles
// J0 - cos(th_b) J1 = D + (1 - cos(th_b)) J1, with 1 - cos = u x / (1 + cos), x = R^2/r^2, and
// 1/cos - 1 = (1 - cos)/cos: every term is computed without cancellation.
//
// Reduction.  FP64 path: each thread accumulates its beams' contributions in double, each block
// reduces them with a fixed shuffle/shared-memory tree in double and adds its partial to the
// instance accumulator as integers in units of 2^-34 and 2^-64 (exact to 2^-64, no carry; a third word for
// partials of 8 and more, up to 2^63).  Mixed path: each beam's
// contribution (an FP32 weight times an FP32 state) is summed per thread without rounding loss as an
// unevaluated (hi, lo) pair (MomAcc<float>); at the end of the pass the pair goes to integers in units
// of the instance's 2^-S (the FP32 weights carry that power-of-two scale), and the sums over lanes,
// warps and the grid are integer additions.  So the moments are FP64-accurate sums, with no FP64
// instruction per beam (GB300's FP64 pipe is ~1/68 of its FP32 rate).  Integer addition is associative, so either grid-level sum is
// identical whatever order the blocks arrive in.  Every block derives a stage's constants
// mu(r_s) D, mu(r_s) J1, lambda(r_s) from the integer sums; the last block to arrive at a step's
// final barrier runs the step-size controller in double.
#pragma once

#include "xflat_internal.cuh"

namespace xflat {

// --------------------------------------------------------------------------------------------
// Butcher tableaus (1-based stage indices).
// Traits of every tableau: S stages (stage radii r + c_s h), kPasses passes per step,
// kAdaptive (embedded error control), kErrPow (the controller's exponent is -1/kErrPow),
// kFinalMoments (the final pass reduces the moments of the new state: stage 1 of the next step),
// kEvalsPerStep (new stage evaluations per step), kEM2 (exponential midpoint rule).
struct TabRK4 {
  static constexpr bool kRichardson = false;
  static constexpr int S = 4;
  static constexpr int kPasses = 4;
  static constexpr bool kAdaptive = false;
  static constexpr int kErrPow = 5;
  static constexpr bool kFinalMoments = true;
  static constexpr int kEvalsPerStep = 4;
  static constexpr bool kEM2 = false;
  __host__ __device__ static constexpr double a(int i, int j) {
    return (i == 2 && j == 1) ? 0.5 : (i == 3 && j == 2) ? 0.5 : (i == 4 && j == 3) ? 1.0 : 0.0;
  }
  __host__ __device__ static constexpr double c(int i) {
    return i == 1 ? 0.0 : (i == 4 ? 1.0 : 0.5);
  }
  __host__ __device__ static constexpr double b(int i) {
    return (i == 1 || i == 4) ? 1.0 / 6.0 : 1.0 / 3.0;
  }
  __host__ __device__ static constexpr double e(int) { return 0.0; }
};

// Dormand & Prince (1980) 5(4) pair; b = row 7 of A (first same as last), e = b - bhat.
struct TabDP45 {
  static constexpr bool kRichardson = false;
  static constexpr int S = 7;
  static constexpr int kPasses = 7;
  static constexpr bool kAdaptive = true;
  static constexpr int kErrPow = 5;
  static constexpr bool kFinalMoments = false;   // first same as last: stage 7 is the new state
  static constexpr int kEvalsPerStep = 6;
  static constexpr bool kEM2 = false;
  __host__ __device__ static constexpr double a(int i, int j) {
    return i == 2 ? (j == 1 ? 1.0 / 5 : 0.0)
         : i == 3 ? (j == 1 ? 3.0 / 40 : j == 2 ? 9.0 / 40 : 0.0)
         : i == 4 ? (j == 1 ? 44.0 / 45 : j == 2 ? -56.0 / 15 : j == 3 ? 32.0 / 9 : 0.0)
         : i == 5 ? (j == 1 ? 19372.0 / 6561 : j == 2 ? -25360.0 / 2187 : j == 3 ? 64448.0 / 6561
                                             : j == 4 ? -212.0 / 729 : 0.0)
         : i == 6 ? (j == 1 ? 9017.0 / 3168 : j == 2 ? -355.0 / 33 : j == 3 ? 46732.0 / 5247
                     : j == 4 ? 49.0 / 176 : j == 5 ? -5103.0 / 18656 : 0.0)
         : i == 7 ? b(j) : 0.0;
  }
  __host__ __device__ static constexpr double c(int i) {
    return i == 1 ? 0.0 : i == 2 ? 0.2 : i == 3 ? 0.3 : i == 4 ? 0.8 : i == 5 ? 8.0 / 9 : 1.0;
  }
  __host__ __device__ static constexpr double b(int j) {
    return j == 1 ? 35.0 / 384 : j == 3 ? 500.0 / 1113 : j == 4 ? 125.0 / 192
         : j == 5 ? -2187.0 / 6784 : j == 6 ? 11.0 / 84 : 0.0;
  }
  // b - bhat, bhat = (5179/57600, 0, 7571/16695, 393/640, -92097/339200, 187/2100, 1/40)
  __host__ __device__ static constexpr double e(int j) {
    return j == 1 ? 71.0 / 57600 : j == 3 ? -71.0 / 16695 : j == 4 ? 71.0 / 1920
         : j == 5 ? -17253.0 / 339200 : j == 6 ? 22.0 / 525 : j == 7 ? -1.0 / 40 : 0.0;
  }
};

// Commutator-free Lie RK4 (Celledoni, Marthinsen & Owren 2003): stage radii as classical RK4.
struct TabCF4 {
  static constexpr bool kRichardson = false;
  static constexpr int S = 4;
  static constexpr int kPasses = 4;
  static constexpr bool kAdaptive = false;
  static constexpr int kErrPow = 5;
  static constexpr bool kFinalMoments = true;
  static constexpr int kEvalsPerStep = 4;
  static constexpr bool kEM2 = false;
  __host__ __device__ static constexpr double a(int, int) { return 0.0; }
  __host__ __device__ static constexpr double b(int) { return 0.0; }
  __host__ __device__ static constexpr double e(int) { return 0.0; }
  __host__ __device__ static constexpr double c(int i) { return TabRK4::c(i); }
};

// Exponential midpoint rule (Lie-group Runge-Kutta-Munthe-Kaas method with Runge's midpoint
// tableau) with its exponential-Euler partner as the embedded first-order estimate: stage 1 at r
// (generator K1), stage 2 at r + h/2 from the half step Y_half = exp(h/2 K1) y, the new state
// exp(h K2) y, the estimate exp(h K1) y; stage 3 is the new state at r + h (the next step's stage 1).
struct TabEM2 {
  static constexpr bool kRichardson = false;
  static constexpr int S = 3;
  static constexpr int kPasses = 2;
  static constexpr bool kAdaptive = true;
  static constexpr int kErrPow = 2;
  static constexpr bool kFinalMoments = true;
  static constexpr int kEvalsPerStep = 2;
  static constexpr bool kEM2 = true;
  __host__ __device__ static constexpr double a(int, int) { return 0.0; }
  __host__ __device__ static constexpr double b(int) { return 0.0; }
  __host__ __device__ static constexpr double e(int) { return 0.0; }
  __host__ __device__ static constexpr double c(int i) { return i == 1 ? 0.0 : (i == 2 ? 0.5 : 1.0); }
};

// Commutator-free Lie RK4 (as TabCF4) with Richardson step-size control: every attempt takes the
// full step of size h and two half steps from the same state, keeps the two half steps and
// estimates their local error as (y_two - y_full) / (2^4 - 1) (error norm, acceptance and
// controller as DP45, exponent 1/5).  Stage slots and radii r + c h:
//   1 (c = 0): y;  full step: 2 (1/2), 3 (1/2), 4 (1);  first half step: 5 (1/4), 6 (1/4), 7 (1/2);
//   8 (1/2): the first half step's result y_a;  second half step from y_a: 9 (3/4), 10 (3/4), 11 (1).
// Pass p reduces slot p + 2; the final pass forms y_b (two half steps) and y_full, the error, and
// the moments of y_b at r + h (the next step's slot 1).
struct TabCFR {
  static constexpr bool kRichardson = true;
  static constexpr int S = 11;
  static constexpr int kPasses = 11;
  static constexpr bool kAdaptive = true;
  static constexpr int kErrPow = 5;
  static constexpr bool kFinalMoments = true;
  static constexpr int kEvalsPerStep = 11;
  static constexpr bool kEM2 = false;
  __host__ __device__ static constexpr double a(int, int) { return 0.0; }
  __host__ __device__ static constexpr double b(int) { return 0.0; }
  __host__ __device__ static constexpr double e(int) { return 0.0; }
  __host__ __device__ static constexpr double c(int i) {
    return i == 1 ? 0.0 : (i == 2 || i == 3 || i == 7 || i == 8) ? 0.5 : (i == 5 || i == 6) ? 0.25
         : (i == 9 || i == 10) ? 0.75 : 1.0;
  }
};

// Largest finite value of the working precision.
template <typename Real>
__host__ __device__ constexpr Real rbig() { return sizeof(Real) == 4 ? Real(3.0e38) : Real(1.7e308); }

// Geometry of one (stage radius, angle bin): cos, 1/cos, 1 - cos, 1/cos - 1 without cancellation.
// The kernels use q (path-length factor 1/cos of Eq. eom), t1 (the weight of the moment D) and t2
// (the factor of mu J1 in the nu-nu term): K = q [eta omega B + lambda z + mu (D + t2 J1)].
//   bulb: q = 1/cos th, t1 = 1/cos th - 1, t2 = 1 - cos th (Eq. Hnu with the measure in u-bins);
//   single angle: every beam radial (q = 1, D = 0) and t2 = (1 - sqrt(1 - x))^2 / x, the
//     geometric factor of Eq. Hnu integrated over emission uniform in u (x = R^2 / r^2);
//   homogeneous test geometry: q = 1, D = 0, t2 = 1 (H_nunu = mu0 J1, mu0 constant).
struct Geo { double q, t1, t2; };
__device__ __forceinline__ Geo geometry(double u, double x, int geom = kGeomBulb) {
  if (geom == kGeomSingleAngle) {
    const double s = 1.0 + sqrt(1.0 - x);       // (1 - sqrt(1 - x))^2 / x = x / (1 + sqrt(1 - x))^2
    return {1.0, 0.0, x / (s * s)};
  }
  if (geom == kGeomHomogeneous) return {1.0, 0.0, 1.0};
  const double c = sqrt(fma(-u, x, 1.0));
  const double t2 = u * x / (1.0 + c);          // 1 - cos
  const double q = 1.0 / c;                     // 1 / cos
  return {q, t2 * q, t2};                       // t1 = 1/cos - 1 = (1 - cos)/cos
}
__device__ __forceinline__ void geometry_f(double u, double x, float& q, float& t1, float& t2,
                                           int geom = kGeomBulb) {
  if (geom != kGeomBulb) {
    const Geo g = geometry(u, x, geom);
    q = (float)g.q;
    t1 = (float)g.t1;
    t2 = (float)g.t2;
    return;
  }
  const float om = (float)fma(-u, x, 1.0);      // 1 - u x in double (no cancellation), then FP32
  const float ux = (float)(u * x);
  const float c = sqrtf(om);
  q = 1.0f / c;
  t2 = ux / (1.0f + c);
  t1 = t2 * q;
}

// --------------------------------------------------------------------------------------------
// Per-thread moment accumulators.  FP64 kernels add each beam's contribution w s by FMA into a
// double.  Mixed kernels sum the contributions of FP32 weights and states as an unevaluated pair
// hi + lo without rounding loss, four operations a contribution:
//   s = fma(w, y, hi),  z = hi - s,  lo += fma(w, y, z),  hi = s.
// hi starts at a bias 1.5 2^m with 2^(m-1) at least the sum of the contributions' magnitudes, so it
// stays in one binade: z is exact (both are multiples of the same 2^(m-23)), fma(w, y, z) is the part
// of the exact product that hi did not take, rounded to 2^(m-48), and the product itself is not rounded
// first; lo's own roundings are near 2^(m-48) times the square root of the n contributions.  2^m is at most
// 16 (n + 2) wmax (run_pass), so with weights of wbar on average the error of a thread's sum is about
// n 2^-46 wmax / wbar of it, coarser than a double's but below the 2^-24 roundings of the states and weights
// while n wmax / wbar is below 2^22.  (TwoSum on the rounded product takes eight operations and needs no
// bias.)  At the end of a pass hi is an integer count of 2^(m-23) read off its bits (biased_fix) and every
// further sum is an integer addition.  The
// FP32 weights carry a per-instance power-of-two scale (InstConst::acc_unit = 2^-S) so that the
// integers are in units of 2^-S; no FP64 instruction is issued per beam (GB300's FP64 pipe is ~1/68
// of its FP32 rate).  Components come in groups with a bias each (D, J1, and Jc, Js): their weights
// differ by the geometry factor, which far from R is far below one.
__device__ __forceinline__ void biased_add(float& hi, float& lo, float w, float y) {
  const float s = __fmaf_rn(w, y, hi);
  const float z = __fsub_rn(hi, s);
  lo = __fadd_rn(lo, __fmaf_rn(w, y, z));
  hi = s;
}
// The bias for contributions whose magnitudes sum to at most P: 1.5 2^m, 2^(m-2) <= P < 2^(m-1).
__device__ __forceinline__ float sum_bias(float P) {
  return __int_as_float((((__float_as_int(P) >> 23) + 2) << 23) | 0x400000);
}

template <typename Real, int NM> struct MomAcc;
// FP64: within an angle row all weights share their angle factors, so a thread sums g_k s (row, 3 or 9
// FMAs a beam) and multiplies the row's sum by du, du t1, ... when it leaves the row (Phys::flush_row).
template <int NM> struct MomAcc<double, NM> {
  static constexpr bool kRows = true;
  double v[NM], r[NM];                                 // r: as many as a state has components are used
  __device__ __forceinline__ void start(const float*, int nc) {
#pragma unroll
    for (int i = 0; i < NM; ++i) { v[i] = 0.0; if (i < nc) r[i] = 0.0; }
  }
};
template <int NM> struct MomAcc<float, NM> {
  static constexpr bool kRows = false;
  float hi[NM], lo[NM];
  // bias: one per group of nc components
  __device__ __forceinline__ void start(const float* bias, int nc) {
#pragma unroll
    for (int i = 0; i < NM; ++i) { hi[i] = bias[i / nc]; lo[i] = 0.0f; }
  }
  __device__ __forceinline__ void add(int i, float w, float y) { biased_add(hi[i], lo[i], w, y); }
};

// A float that holds a count of 2^-S units (possibly with a fraction) as the nearest int64 (halves
// away from zero), from its bits on the integer pipe, branch-free (no FP64 instruction).  Sets ovf
// when |v| >= 2^52 or v is not finite: a partial that large voids the scale's guarantee.
__device__ __forceinline__ long long f32_to_fix(float v, int& ovf) {
  const unsigned int b = __float_as_uint(v);
  const unsigned int ef = (b >> 23) & 0xffu;
  ovf |= ef >= 127u + 52u ? 1 : 0;
  const unsigned int m = ef ? ((b & 0x7fffffu) | 0x800000u) : 0u;   // below 2^-126: zero
  const int e = (int)ef - 150;                                       // |v| = m 2^e
  const int rs = min(max(-e, 0), 31);
  const unsigned int mr = rs ? ((m + (1u << (rs - 1))) >> rs) : m;
  const unsigned long long r = (unsigned long long)mr << min(max(e, 0), 63);
  return (b >> 31) ? -(long long)r : (long long)r;
}
constexpr long long kFixLimit = 1ll << 52;               // largest block partial accepted

// The sum collected by N biased accumulators (hi starting at bias, lo) in units of 2^-S: hi's distance
// from the bias off its bits, lo rounded.  A hi that left its binade (a state far above unit length) or
// a lo past 32 bits takes the general conversion.
template <int N>
__device__ __forceinline__ long long biased_fix(const float (&hi)[N], float lo, float bias, int& ovf) {
  const int bb = __float_as_int(bias), sh = (bb >> 23) - 127 - 23;
  bool plain = fabsf(lo) < 2.0e9f;
  int k = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const int b = __float_as_int(hi[i]);
    plain = plain && ((b ^ bb) >> 23) == 0;
    k += b - bb;
  }
  if (plain) {
    const int down = min(max(-sh, 0), 62);
    const long long v = ((long long)k << max(sh, 0)) + (down ? 1ll << (down - 1) : 0ll);
    return (v >> down) + (long long)__float2int_rn(lo);
  }
  long long v = f32_to_fix(lo, ovf);
#pragma unroll
  for (int i = 0; i < N; ++i) v += f32_to_fix(__fsub_rn(hi[i], bias), ovf);
  return v;
}

// --------------------------------------------------------------------------------------------
// Physics policies.  "Real" is the working precision of the per-beam algebra.
//
// Two flavours: the state of a beam is the Bloch vector s of P = (1 + s.sigma)/2 (antineutrinos:
// of conj(Pbar)), and every beam obeys ds/dr = K x s with
//   K = [eta omega_k B + lambda(r) z + mu(r) (D + (1 - cos th) J1)] / cos th,
// eta = +1 / -1 for nu / nubar, B = (sin 2 theta_v, 0, -cos 2 theta_v): this is
// d(rho)/dr = -i [H, rho] / cos(th) of Eq. eom with H = (1/2) h.sigma.
//
// A table row belongs to one (stage, angle bin): a geometry part, t1 = 1/cos - 1, q = 1/cos, t2 (see
// Geo), q Bx, q Bz, known from the step's radii alone (fill_geo), and a coupling part G0 = q (lambda z +
// mu D + t2 mu J1), known once the stage's moments are (fill_cpl), so that K = eta omega (q Bx, 0, q Bz)
// + G0.  FP32 rows are in the order and the signs in which PairRK needs the components of K, one
// 128-bit and one 32-bit load a stage; those of the commutator integrators are K times the step size.
template <typename Real>
struct Phys2 {
  static constexpr bool kF32 = sizeof(Real) == 4;
  static constexpr bool kPairable = kF32;       // FP32 passes run beam pairs (PairRK)
  static constexpr int NC = 3, NG = 3, NM = kNM2, NSC = kNSC2, KT = 8;
  static constexpr int kERows = kF32 ? 4 : 3;   // energy table: omega_k, weights of nu and nubar (FP32: by bin, padded)
  enum : int { vT1 = 0, vQ = 1, vQBX = 2, vQBZ = 3, vG0X = 4, vG0Y = 5, vG0Z = 6, vT2 = 7 };   // FP64
  enum : int { oNQBX = 0, oNG0X = 1, oQBZ = 2, oG0Z = 3, oG0Y = 4, oT1 = 5, oT2 = 6, oQ = 7 };                 // FP32
  struct Consts { double B[3]; int geom; };
  struct Beam { Real eo; Real w; };   // eta * omega_k, signed weight du_j * g_{sigma,k} (FP64: g alone)
  template <typename R> using With = Phys2<R>;

  __device__ static inline Real t1(const Real* t) { return kF32 ? t[oT1] : t[vT1]; }

  // hs: factor of the K entries (the step size, or 1)
  __device__ static inline void fill_geo(Real* t, double u, double x, const Consts& C, int, Real hs) {
    if constexpr (kF32) {
      float q, t1v, t2;
      geometry_f(u, x, q, t1v, t2, C.geom);
      const float hq = hs * q;
      t[oNQBX] = -(hq * (float)C.B[0]);
      t[oQBZ] = hq * (float)C.B[2];
      t[oT1] = t1v;
      t[oT2] = t2;
      t[oQ] = hq;
    } else {
      const Geo g = geometry(u, x, C.geom);
      t[vT1] = g.t1;
      t[vQ] = g.q;
      t[vT2] = g.t2;
      t[vQBX] = g.q * C.B[0];
      t[vQBZ] = g.q * C.B[2];
    }
  }
  // sc: mu D (3), mu J1 (3), lambda
  __device__ static inline void fill_cpl(Real* t, const Real* sc) {
    const Real q = kF32 ? t[oQ] : t[vQ], t2 = kF32 ? t[oT2] : t[vT2];
    const Real gx = q * (sc[0] + t2 * sc[3]);
    const Real gy = q * (sc[1] + t2 * sc[4]);
    const Real gz = q * (sc[6] + sc[2] + t2 * sc[5]);
    if constexpr (kF32) {
      t[oNG0X] = -gx;
      t[oG0Z] = gz;
      t[oG0Y] = gy;
    } else {
      t[vG0X] = gx;
      t[vG0Y] = gy;
      t[vG0Z] = gz;
    }
  }
  __device__ static inline void K(const Real* t, const Beam& bm, Real (&Kv)[3]) {
    if constexpr (kF32) {
      Kv[0] = -(bm.eo * t[oNQBX] + t[oNG0X]);
      Kv[1] = t[oG0Y];
      Kv[2] = bm.eo * t[oQBZ] + t[oG0Z];
    } else {
      Kv[0] = bm.eo * t[vQBX] + t[vG0X];
      Kv[1] = t[vG0Y];
      Kv[2] = bm.eo * t[vQBZ] + t[vG0Z];
    }
  }
  __device__ static inline void f(const Real (&Kv)[3], const Real (&y)[3], Real (&k)[3]) {
    k[0] = Kv[1] * y[2] - Kv[2] * y[1];
    k[1] = Kv[2] * y[0] - Kv[0] * y[2];
    k[2] = Kv[0] * y[1] - Kv[1] * y[0];
  }
  // moments D (weight w t1) and J1 (weight w); row sums: w is g_k alone
  template <class Acc>
  __device__ static inline void accum_row(Acc& acc, Real w, const Real* row, const Real (&y)[3]) {
    if constexpr (Acc::kRows) {
#pragma unroll
      for (int i = 0; i < 3; ++i) acc.r[i] = fma(w, y[i], acc.r[i]);
    } else {
      const Real wt = w * t1(row);
#pragma unroll
      for (int i = 0; i < 3; ++i) { acc.add(i, wt, y[i]); acc.add(3 + i, w, y[i]); }
    }
  }
  template <class Acc>
  __device__ static inline void flush_row(Acc& acc, Real du, const Real* row) {
    const Real dt = du * t1(row);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      acc.v[i] = fma(dt, acc.r[i], acc.v[i]);
      acc.v[3 + i] = fma(du, acc.r[i], acc.v[3 + i]);
      acc.r[i] = 0;
    }
  }
  // Frobenius norm^2 of the traceless part of P = (1 + s.sigma)/2: |s|^2 / 2
  __device__ static inline Real tnorm2(const Real (&y)[3]) {
    return Real(0.5) * (y[0] * y[0] + y[1] * y[1] + y[2] * y[2]);
  }
  // The larger norm of two states given by their components' leading 21 bits, or a little less
  __device__ static inline Real norm_floor(const Real (&a)[3], const Real (&b)[3]) {
    return sqrt(fmax(tnorm2(a), tnorm2(b)));
  }
  __device__ static inline void normalise(Real (&y)[3]) {
    const Real n2 = y[0] * y[0] + y[1] * y[1] + y[2] * y[2];
    const Real inv = Real(1) / sqrt(n2);
#pragma unroll
    for (int i = 0; i < 3; ++i) y[i] *= inv;
  }
  // the pure-state projection of the exponential steps: for a Bloch vector, its unit length
  __device__ static inline void purify(Real (&y)[3]) { normalise(y); }
};

// Three flavours: the state is the full 3x3 Hermitian density matrix (9 reals: P00, P11, P22,
// Re P01, Im P01, Re P02, Im P02, Re P12, Im P12) of P (nu) or conj(Pbar) (nubar); the derivative
// is -i [K, P] with the Hermitian
//   K = [eta (omega21 M21 + omega31 M31) + lambda E_ee + mu (D + (1 - cos) J1)] / cos,
// M21/M31 the real unit vacuum matrices U diag(0,1,0) U^T and U diag(0,0,1) U^T.
//
// Commutators and propagators do not see a multiple of the unit matrix in K, so a generator is 8
// reals (NG): K00 - K22, K11 - K22, then real and imaginary parts of K01, K02, K12.  The energy
// table holds the 5 real vacuum entries of each bin (kVac) and a table row the rest of the
// generator, G = q (lambda E_ee + mu D + (1 - cos) mu J1), so an assembled generator is one FMA for
// each real entry, K = q v + G.  These kernels are bound by arithmetic (FP64: the two-lane pipe).
template <typename Real>
struct Phys3 {
  static constexpr bool kPairable = false;
  static constexpr int NC = 9, NG = 8, NM = kNM3, NSC = kNSC3, KT = 11;
  static constexpr int kVac = 5, kERows = kVac + 2;
  enum : int { vT1 = 0, vQ = 1, vG = 2, vT2 = 10 };
  struct Consts { int geom; };
  struct Beam { Real v[kVac]; Real w; };
  template <typename R> using With = Phys3<R>;

  __device__ static inline Real t1(const Real* t) { return t[vT1]; }
  __device__ static inline void fill_geo(Real* t, double u, double x, const Consts& C, int, Real hs) {
    if constexpr (sizeof(Real) == 4) {
      float q, t1v, t2;
      geometry_f(u, x, q, t1v, t2, C.geom);
      t[vT1] = t1v;
      t[vQ] = hs * q;
      t[vT2] = t2;
    } else {
      const Geo g = geometry(u, x, C.geom);
      t[vT1] = g.t1;
      t[vQ] = g.q;
      t[vT2] = g.t2;
    }
  }
  // sc: mu D (9), mu J1 (9), lambda
  __device__ static inline void fill_cpl(Real* t, const Real* sc) {
    const Real q = t[vQ], t2 = t[vT2];
    const Real g22 = sc[2] + t2 * sc[11];
    t[vG + 0] = q * (sc[18] + (sc[0] + t2 * sc[9]) - g22);
    t[vG + 1] = q * (sc[1] + t2 * sc[10] - g22);
#pragma unroll
    for (int i = 2; i < NG; ++i) t[vG + i] = q * (sc[i + 1] + t2 * sc[i + 10]);
  }
  // the generator: v holds eta (omega21 M21 + omega31 M31) of the beam's energy bin (00 - 22,
  // 11 - 22, 01, 02, 12)
  __device__ static inline void K(const Real* t, const Beam& bm, Real (&Kv)[NG]) {
    const Real q = t[vQ];
    const Real* g = t + vG;
    Kv[0] = q * bm.v[0] + g[0];
    Kv[1] = q * bm.v[1] + g[1];
    Kv[2] = q * bm.v[2] + g[2];
    Kv[3] = g[3];
    Kv[4] = q * bm.v[3] + g[4];
    Kv[5] = g[5];
    Kv[6] = q * bm.v[4] + g[6];
    Kv[7] = g[7];
  }
  // Z = -i [K, Y] entry by entry.  With x, y, z = K01, K02, K12 and a, b, c = Y01, Y02, Y12:
  //   [K,Y]_01 = (K00 - K11) a - (Y00 - Y11) x + y conj(c) - b conj(z),
  //   [K,Y]_02 = (K00 - K22) b - (Y00 - Y22) y + x c - a z,
  //   [K,Y]_12 = (K11 - K22) c - (Y11 - Y22) z + conj(x) b - conj(a) y,
  // and the diagonal is 2i Im(x conj(a) + y conj(b)), 2i Im(z conj(c) - x conj(a)), minus their sum:
  // 52 operations where the two full complex products take about 170.  (262,144 beams, FP64 DP45,
  // GB300, a call of 8 steps: 7.80 ms with the full products and 39 operations per assembled K,
  // 4.97 ms so.)
  __device__ static inline void f(const Real (&Kv)[NG], const Real (&y)[9], Real (&z)[9]) {
    const Real d02 = Kv[0], d12 = Kv[1], d01 = d02 - d12;
    const Real xr = Kv[2], xi = Kv[3], yr = Kv[4], yi = Kv[5], zr = Kv[6], zi = Kv[7];
    const Real ar = y[3], ai = y[4], br = y[5], bi = y[6], cr = y[7], ci = y[8];
    const Real e01 = y[0] - y[1], e02 = y[0] - y[2], e12 = y[1] - y[2];
    const Real A = xi * ar - xr * ai, B = yi * br - yr * bi, C = zi * cr - zr * ci;
    const Real z0 = A + B, z2 = B + C, z1 = C - A;
    z[0] = z0 + z0;
    z[1] = z1 + z1;
    z[2] = -(z2 + z2);
    z[3] = d01 * ai - e01 * xi + yi * cr - yr * ci - bi * zr + br * zi;
    z[4] = e01 * xr - d01 * ar - yr * cr - yi * ci + br * zr + bi * zi;
    z[5] = d02 * bi - e02 * yi + xr * ci + xi * cr - ar * zi - ai * zr;
    z[6] = e02 * yr - d02 * br - xr * cr + xi * ci + ar * zr - ai * zi;
    z[7] = d12 * ci - e12 * zi + xr * bi - xi * br - ar * yi + ai * yr;
    z[8] = e12 * zr - d12 * cr - xr * br - xi * bi + ar * yr + ai * yi;
  }
  template <class Acc>
  __device__ static inline void accum_row(Acc& acc, Real w, const Real* row, const Real (&y)[9]) {
    if constexpr (Acc::kRows) {
#pragma unroll
      for (int i = 0; i < 9; ++i) acc.r[i] = fma(w, y[i], acc.r[i]);
    } else {
      const Real wt = w * t1(row);
#pragma unroll
      for (int i = 0; i < 9; ++i) { acc.add(i, wt, y[i]); acc.add(9 + i, w, y[i]); }
    }
  }
  template <class Acc>
  __device__ static inline void flush_row(Acc& acc, Real du, const Real* row) {
    const Real dt = du * t1(row);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      acc.v[i] = fma(dt, acc.r[i], acc.v[i]);
      acc.v[9 + i] = fma(du, acc.r[i], acc.v[9 + i]);
      acc.r[i] = 0;
    }
  }
  // ||P - tr(P)/3||_F^2 with off-diagonal entries counted twice
  __device__ static inline Real tnorm2(const Real (&y)[9]) {
    const Real t = (y[0] + y[1] + y[2]) * Real(1.0 / 3.0);
    const Real d0 = y[0] - t, d1 = y[1] - t, d2 = y[2] - t;
    return d0 * d0 + d1 * d1 + d2 * d2 +
           2 * (y[3] * y[3] + y[4] * y[4] + y[5] * y[5] + y[6] * y[6] + y[7] * y[7] + y[8] * y[8]);
  }
  // The larger norm of two states given by their components' leading 21 bits, or a little less: taking
  // the trace off amplifies the truncation (2^-20 of the diagonal) where a state is nearly 1/3
  __device__ static inline Real norm_floor(const Real (&a)[9], const Real (&b)[9]) {
    const Real d = fabs(a[0]) + fabs(a[1]) + fabs(a[2]) + fabs(b[0]) + fabs(b[1]) + fabs(b[2]);
    return fmax(sqrt(fmax(tnorm2(a), tnorm2(b))) - Real(4e-6) * d, Real(0));
  }
  __device__ static inline void normalise(Real (&)[9]) {}
  // Mixed-precision exponential steps: restore the idempotency of the (pure) density matrix that
  // the FP32 rounding of the propagators erodes step by step, P <- 3 P^2 - 2 P^3 (McWeeny
  // purification: an eigenvalue 1 - e goes to 1 - 3 e^2 + 2 e^3, a small one d to 3 d^2 - 2 d^3),
  // as the two-flavour path renormalises its Bloch vector.
  __device__ static inline void purify(Real (&y)[9]) {
    const Real pr[3][3] = {{y[0], y[3], y[5]}, {y[3], y[1], y[7]}, {y[5], y[7], y[2]}};
    const Real pi[3][3] = {{0, y[4], y[6]}, {-y[4], 0, y[8]}, {-y[6], -y[8], 0}};
    Real qr[3][3], qi[3][3];                          // P^2
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        Real sr = 0, si = 0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          sr += pr[a][c] * pr[c][b] - pi[a][c] * pi[c][b];
          si += pr[a][c] * pi[c][b] + pi[a][c] * pr[c][b];
        }
        qr[a][b] = sr;
        qi[a][b] = si;
      }
    Real outr[3][3], outi[3][3];                      // 3 P^2 - 2 P^3, upper triangle
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = a; b < 3; ++b) {
        Real sr = 0, si = 0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          sr += qr[a][c] * pr[c][b] - qi[a][c] * pi[c][b];
          si += qr[a][c] * pi[c][b] + qi[a][c] * pr[c][b];
        }
        outr[a][b] = Real(3) * qr[a][b] - Real(2) * sr;
        outi[a][b] = Real(3) * qi[a][b] - Real(2) * si;
      }
    y[0] = outr[0][0];
    y[1] = outr[1][1];
    y[2] = outr[2][2];
    y[3] = outr[0][1];
    y[4] = outi[0][1];
    y[5] = outr[0][2];
    y[6] = outi[0][2];
    y[7] = outr[1][2];
    y[8] = outi[1][2];
  }
};
// Two flavours, extended bulb model (Sec. 2, Eq. int-v and Eq. F): beams also carry an azimuthal
// angle phi around the radial direction, the combined angle bin a = j n_phi + p holding u_j,
// du_j / n_phi and phi_p = 2 pi (p + 1/2) / n_phi.  Besides D and J1 the potential needs
//   Jc = sum_b w_b (sin th_b / cos th_b) cos phi_b s_b,   Js = the same with sin phi_b,
// and K = [eta omega B + lambda z + mu (D + (1 - cos th) J1 - sin th (cos phi Jc + sin phi Js))] / cos th.
// Table rows as Phys2's, with the azimuthal moment weights (sin th / cos th) cos phi and
// (sin th / cos th) sin phi.
template <typename Real>
struct Phys2E {
  static constexpr bool kF32 = sizeof(Real) == 4;
  static constexpr bool kPairable = kF32;       // FP32 passes run beam pairs (PairRK)
  static constexpr int NC = 3, NG = 3, NM = 12, NSC = 14, KT = kF32 ? 12 : 10;
  static constexpr int kERows = Phys2<Real>::kERows;
  enum : int { vT1 = 0, vQ = 1, vQBX = 2, vQBZ = 3, vG0X = 4, vG0Y = 5, vG0Z = 6, vSCC = 7, vSCS = 8, vT2 = 9 };   // FP64
  enum : int { oNQBX = 0, oNG0X = 1, oQBZ = 2, oG0Z = 3, oG0Y = 4, oT1 = 5, oT2 = 6, oQ = 7, oSCC = 8, oSCS = 9, oH = 10 };   // FP32
  struct Consts { double B[3]; int n_phi; };
  using Beam = typename Phys2<Real>::Beam;
  template <typename R> using With = Phys2E<R>;

  __device__ static inline Real t1(const Real* t) { return kF32 ? t[oT1] : t[vT1]; }
  __device__ static inline void fill_geo(Real* t, double u, double x, const Consts& C, int a, Real hs) {
    const int pidx = a % C.n_phi;
    if constexpr (kF32) {
      // FP32 rows in FP32 arithmetic (as Phys2's): the table holds floats anyway, and FP64 square
      // roots, divisions and sincospi per row would cost more than the row's beams on GB300
      float q, t1v, t2, sp, cp;
      geometry_f(u, x, q, t1v, t2);
      const float so = sqrtf((float)(u * x)) * q;             // sin th / cos th, sin^2 th = u R^2 / r^2
      sincospif((2.0f * pidx + 1.0f) / C.n_phi, &sp, &cp);   // phi_p = 2 pi (p + 1/2) / n_phi
      const float hq = hs * q;
      t[oNQBX] = -(hq * (float)C.B[0]);
      t[oQBZ] = hq * (float)C.B[2];
      t[oT1] = t1v;
      t[oSCC] = so * cp;
      t[oSCS] = so * sp;
      t[oT2] = t2;
      t[oQ] = hq;
      t[oH] = hs;
    } else {
      const Geo g = geometry(u, x);
      const double so = sqrt(u * x) * g.q;
      double sp, cp;
      sincospi((2.0 * pidx + 1.0) / C.n_phi, &sp, &cp);
      t[vT1] = g.t1;
      t[vQ] = g.q;
      t[vT2] = g.t2;
      t[vQBX] = g.q * C.B[0];
      t[vQBZ] = g.q * C.B[2];
      t[vSCC] = so * cp;
      t[vSCS] = so * sp;
    }
  }
  // sc: mu D (3), mu J1 (3), mu Jc (3), mu Js (3), lambda
  __device__ static inline void fill_cpl(Real* t, const Real* sc) {
    const Real q = kF32 ? t[oQ] : t[vQ], t2 = kF32 ? t[oT2] : t[vT2];
    const Real scc = kF32 ? t[oH] * t[oSCC] : t[vSCC], scs = kF32 ? t[oH] * t[oSCS] : t[vSCS];
    Real g[3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
      g[i] = q * ((i == 2 ? sc[12] : Real(0)) + sc[i] + t2 * sc[3 + i]) - (scc * sc[6 + i] + scs * sc[9 + i]);
    if constexpr (kF32) {
      t[oNG0X] = -g[0];
      t[oG0Z] = g[2];
      t[oG0Y] = g[1];
    } else {
      t[vG0X] = g[0];
      t[vG0Y] = g[1];
      t[vG0Z] = g[2];
    }
  }
  __device__ static inline void K(const Real* t, const Beam& bm, Real (&Kv)[3]) {
    if constexpr (kF32) {
      Kv[0] = -(bm.eo * t[oNQBX] + t[oNG0X]);
      Kv[1] = t[oG0Y];
      Kv[2] = bm.eo * t[oQBZ] + t[oG0Z];
    } else {
      Kv[0] = bm.eo * t[vQBX] + t[vG0X];
      Kv[1] = t[vG0Y];
      Kv[2] = bm.eo * t[vQBZ] + t[vG0Z];
    }
  }
  __device__ static inline void f(const Real (&Kv)[3], const Real (&y)[3], Real (&k)[3]) {
    Phys2<Real>::f(Kv, y, k);
  }
  template <class Acc>
  __device__ static inline void accum_row(Acc& acc, Real w, const Real* t, const Real (&y)[3]) {
    if constexpr (Acc::kRows) {
#pragma unroll
      for (int i = 0; i < 3; ++i) acc.r[i] = fma(w, y[i], acc.r[i]);
    } else {
      const Real wt = w * t1(t), wc = w * t[oSCC], ws = w * t[oSCS];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        acc.add(i, wt, y[i]);
        acc.add(3 + i, w, y[i]);
        acc.add(6 + i, wc, y[i]);
        acc.add(9 + i, ws, y[i]);
      }
    }
  }
  template <class Acc>
  __device__ static inline void flush_row(Acc& acc, Real du, const Real* t) {
    const Real f[4] = {du * t1(t), du, du * t[vSCC], du * t[vSCS]};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
#pragma unroll
      for (int g = 0; g < 4; ++g) acc.v[3 * g + i] = fma(f[g], acc.r[i], acc.v[3 * g + i]);
      acc.r[i] = 0;
    }
  }
  __device__ static inline Real tnorm2(const Real (&y)[3]) { return Phys2<Real>::tnorm2(y); }
  __device__ static inline Real norm_floor(const Real (&a)[3], const Real (&b)[3]) { return Phys2<Real>::norm_floor(a, b); }
  __device__ static inline void normalise(Real (&y)[3]) { Phys2<Real>::normalise(y); }
  __device__ static inline void purify(Real (&y)[3]) { Phys2<Real>::normalise(y); }
};


// --------------------------------------------------------------------------------------------
struct KParams {
  int n_inst;
  int n_pieces;
  const InstConst* ic;
  InstDyn* dyn;
  const Piece* pieces;
  const int* blk_piece;          // [gridDim.x + 1]
  unsigned long long* acc;       // [n_inst][kMaxStages][kNMMax][2] fixed-point accumulators
  unsigned long long* errmax;    // [n_inst] error norm maxima (bit patterns of non-negative doubles)
  int* nonfinite;                // [n_inst]
  void* planeA;
  void* planeB;
  void* escr;                    // FP64 DP45: error partial planes [NC][plane_stride]
  void* kst;                     // FP64 RK4 / DP45: stage derivatives k_1..k_n, then one stage state [n + 1][NC][plane_stride]
  uint64_t plane_stride;         // elements between component planes
  const void* etab;              // energy tables, Real, per instance at e_off: [n_tab][n_energy]
  const double* u_tab;           // angle positions u_j, at a_off
  const double* du_tab;          // angle weights du_j, at a_off
  Barrier* bar;
  unsigned long long timeout_ns;
  int* status;                   // global sticky status
  int* all_done;
  int n_steps;
  int init_only;
  // beam-shard mode (one problem split over several GPUs, the host exchanging the stage moments):
  // 0 off; kShardPass: only pass `shard_pass` of the current step (-1: the moment pass of the
  // current state), no device-wide barrier, no serial section; kShardSerialInit / Final: only the
  // serial section that follows the moment pass or a step's final pass (one block)
  int shard_mode;
  int shard_pass;
  // dynamic scheduling (handles with several instances): instead of a fixed list of pieces per
  // block, every block takes the next piece of the pass from a device-wide counter until none is
  // left, so blocks whose pieces run slower (small angle rows, more set-ups, memory placement) do
  // not hold the whole grid at the pass's barrier
  int dyn_sched;
  int max_jj;
  int integrator;
  // optional pass trace (NULL: off): per pass and block, %globaltimer at pass start, after the
  // block's beams and reduction, after the barrier released it, and 1 if it was the last block
  unsigned long long* trace;
  int trace_passes;
#ifdef XFLAT_BOUNDS
  Span span[kSpanCount];         // checked build: the allocations behind the pointers above
#endif
};

// Checked build (-DXFLAT_BOUNDS): every state-plane, stage-plane, energy-table and angle-table
// access of the pass body, the shared-memory row index of every beam and the piece list are tested
// before use.  An access outside its allocation (or off the alignment of its vector type) is
// skipped, a load yielding zeros; the first one is recorded in the barrier's bounds words and the
// launch status becomes XFLAT_ERR_CUDA.  Without the macro every check is the constant true.
#ifdef XFLAT_BOUNDS
static __device__ __noinline__ void bounds_fault(const KParams& p, int site, long long off) {
  if (atomicCAS(&p.bar->bounds_site, 0, site) == 0)
    atomicExch(reinterpret_cast<unsigned long long*>(&p.bar->bounds_off), (unsigned long long)off);
  atomicCAS(p.status, 0, 3 /* XFLAT_ERR_CUDA */);
}
__device__ __forceinline__ bool span_ok(const KParams& p, int id, const void* ptr, unsigned bytes, int site) {
  const Span sp = p.span[id];
  const char* c = static_cast<const char*>(ptr);
  const bool ok = sp.lo != nullptr && c >= sp.lo && c + bytes <= sp.lo + sp.bytes &&
                  (reinterpret_cast<uintptr_t>(c) % bytes) == 0;
  if (!ok) bounds_fault(p, site, sp.lo ? (long long)(c - sp.lo) : -1ll);
  return ok;
}
__device__ __forceinline__ bool index_ok(const KParams& p, bool ok, int site, long long v) {
  if (!ok) bounds_fault(p, site, v);
  return ok;
}
#define XFLAT_SPAN_OK(p, id, ptr, bytes, site) ::xflat::span_ok((p), (id), (ptr), (bytes), (site))
#define XFLAT_INDEX_OK(p, cond, site, v) ::xflat::index_ok((p), (cond), (site), (long long)(v))
#else
#define XFLAT_SPAN_OK(p, id, ptr, bytes, site) true
#define XFLAT_INDEX_OK(p, cond, site, v) true
#endif

// Add x to the fixed-point accumulators of component c of a stage slot, truncating |x| below 2^-64.
// x = big 2^3 + hi 2^-34 + lo 2^-64 exactly, with |hi| < 2^37 and |lo| < 2^30 in two words of one copy: no
// carry passes between them, and neither addition waits for the other's result.  A piece makes one
// addition; an instance has fewer than 2^31 beams in pieces of 124 and more (but for the ends of slices), so
// fewer than 2^25 pieces, and the sum of all copies of a word stays below 2^62.  big is zero for weights
// that sum to a few units, as normalised ones do; else it goes to the slot's one word for large partials.
// Returns false when x or the running sum leaves the range, 2^63.  (The common range is tested on the bits
// and the rest is a function of its own: an FP64 comparison is one more link in the chain of 65-cycle
// operations that ends every pass.)
__device__ __forceinline__ void fx_add_small(unsigned long long* a, double x) {
  const double hi_d = trunc(x * 17179869184.0);                                      // 2^34
  const long long lo = (long long)((x * 17179869184.0 - hi_d) * 1073741824.0);       // exact difference, 2^30
  atomicAdd(&a[0], (unsigned long long)lo);
  atomicAdd(&a[1], (unsigned long long)(long long)hi_d);
}
static __device__ __noinline__ bool fx_add_large(unsigned long long* slot, int copy, int c, double x) {
  if (!(fabs(x) < 9223372036854775808.0)) return false;
  const double b = trunc(x * 0.125);
  const long long big = (long long)b;
  const long long sum = (long long)atomicAdd(slot + ((size_t)kAccCopies * kNMMax + c) * 2, (unsigned long long)big) + big;
  fx_add_small(slot + ((size_t)copy * kNMMax + c) * 2, fma(-8.0, b, x));
  return sum < (1ll << 60) && sum > -(1ll << 60);
}
__device__ __forceinline__ bool fx_add(unsigned long long* slot, int copy, int c, double x) {
  if ((__double2hiint(x) & 0x7fffffff) >= 0x40200000) return fx_add_large(slot, copy, c, x);   // |x| >= 8
  fx_add_small(slot + ((size_t)copy * kNMMax + c) * 2, x);
  return true;
}

template <class Tab>
__device__ __forceinline__ double stage_c(int i) { return Tab::c(i); }

// 0.9 Err^(-1/P), the unclamped step-size factor, in double (P = 5 for the 5(4) pair, 2 for the
// 2(1) pair).  The caller clamps it to [0.2, 5], which decides alone below Err = (0.9/5)^P and
// above (0.9/0.2)^P, so only (a slightly wider) range is computed: a float seed refined by two
// Newton steps for y^-P = Err, y <- y ((P + 1) - Err y^P) / P, which need no division (one FP64
// pow costs ~5800 cycles of latency on this part, the two steps ~800) and converge to double
// accuracy.
template <int P>
__device__ __forceinline__ double controller_factor(double err) {
  constexpr double lo = P == 5 ? 1.5e-4 : 0.025, hi = P == 5 ? 2000.0 : 25.0;
  if (!(err > lo)) return 5.0;
  if (!(err < hi)) return 0.0;
  double y = (double)powf((float)err, -1.0f / (float)P);
  for (int it = 0; it < 2; ++it) {
    double yp = y;
#pragma unroll
    for (int q = 1; q < P; ++q) yp *= y;
    y = y * fma(err * (-1.0 / P), yp, (P + 1.0) / P);
  }
  return 0.9 * y;
}

// lambda(r) from a matter table: the interval [r_i, r_{i+1}) holding r by binary search, then
// lambda_i (r / r_i)^p_i (the end values outside the table)
__device__ inline double table_strength(const double* t, int n, double r) {
  if (r <= t[0]) return t[1];
  if (r >= t[3 * (n - 1)]) return t[3 * (n - 1) + 1];
  int lo = 0, hi = n - 1;                       // t[3 lo] <= r < t[3 hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (t[3 * mid] <= r) lo = mid; else hi = mid;
  }
  return t[3 * lo + 1] * pow(r / t[3 * lo], t[3 * lo + 2]);
}
// mu(r) and lambda(r) from 1/r
__device__ __forceinline__ void strengths_inv(const InstConst& ic, double inv, double& mu, double& lam) {
  mu = ic.geom == kGeomHomogeneous ? ic.mu_const : ic.mu_coef * inv * inv;
  lam = 0.0;
  if (ic.matter == kMatterPower) {
    const double x = ic.r_ref * inv;
    lam = ic.lam_coef * (ic.power == 3.0 ? x * x * x : pow(x, ic.power));
  } else if (ic.matter == kMatterConst) {
    lam = ic.lam_const;
  } else if (ic.matter == kMatterTable) {
    lam = table_strength(ic.mtab, ic.mt_n, 1.0 / inv);
  }
}
__device__ __forceinline__ void strengths(const InstConst& ic, double r, double& mu, double& lam) {
  strengths_inv(ic, 1.0 / r, mu, lam);
}

// Loads that must not hit a stale L1 line: instance dynamics change across barriers.
__device__ __forceinline__ double ldcg(const double* p) { return __ldcg(p); }
__device__ __forceinline__ int ldcg(const int* p) { return __ldcg(p); }

// Component c of a stage's moments: the kAccCopies fixed-point copies summed as integers (exact,
// so every block that reads them gets the same bits), then converted to double.
template <typename Real>
__device__ __forceinline__ double acc_component(const unsigned long long* acc_slot, int c, double unit) {
  if constexpr (sizeof(Real) == 4) {
    long long sum = 0;
#pragma unroll
    for (int cp = 0; cp < kAccCopies; ++cp) sum += (long long)__ldcg(acc_slot + ((size_t)cp * kNMMax + c) * 2);
    return (double)sum * unit;                                   // 2^-S of the instance
  } else {
    const long long big = (long long)__ldcg(acc_slot + ((size_t)kAccCopies * kNMMax + c) * 2);
    long long hi = 0, lo = 0;
#pragma unroll
    for (int cp = 0; cp < kAccCopies; ++cp) {
      const unsigned long long* w = acc_slot + ((size_t)cp * kNMMax + c) * 2;
      const ulonglong2 v = __ldcg(reinterpret_cast<const ulonglong2*>(w));
      lo += (long long)v.x;
      hi += (long long)v.y;
    }
    const __int128 sum = ((__int128)big << 67) + ((__int128)hi << 30) + lo;   // units of 2^-64 (fx_add)
    return (double)(long long)(sum >> 64) + (double)(unsigned long long)sum * 5.421010862427522e-20;
  }
}

// Hand-off of each instance's new r and h (and whether its next step needs stage geometry) from
// serial_update to serial_geometry inside the last block, through shared memory (instances past
// kGeoShared are read back from global memory).
constexpr int kGeoShared = 64;
struct GeoHandoff {
  double r[kGeoShared], h[kGeoShared];
  int pending[kGeoShared];
};
__device__ __forceinline__ GeoHandoff& geo_handoff() {
  __shared__ GeoHandoff g;
  return g;
}

// Sum of N values over a warp, the N results spread over its lanes: at each halving of the lane
// distance a lane keeps one half of the values and hands the other half to its partner, so N = 6 takes 8
// additions a lane instead of the 30 of six shuffle trees (18: 20 instead of 90; on GB300's two-lane
// FP64 pipe every one costs the SM 16 cycles a warp).  Returns the sum of component *idx; *valid in the
// one lane that reports it.
template <int N, int O, typename T>
__device__ __forceinline__ T reduce_scatter(T (&v)[N], int lane, int& idx, int& left, bool& valid) {
  if constexpr (O == 0) {
    valid = valid && left >= 1;
    return v[0];
  } else if constexpr (N == 1) {
    T w[1] = {v[0] + __shfl_xor_sync(0xffffffffu, v[0], O)};
    valid = valid && (lane & O) == 0;
    return reduce_scatter<1, O / 2, T>(w, lane, idx, left, valid);
  } else {
    constexpr int H = (N + 1) / 2;
    const bool up = (lane & O) != 0;
    T w[H];
#pragma unroll
    for (int i = 0; i < H; ++i) {
      const T lo = v[i], hi = i + H < N ? v[i + H < N ? i + H : 0] : T(0);
      w[i] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, O);
    }
    idx += up ? H : 0;
    left = up ? left - H : min(left, H);
    return reduce_scatter<H, O / 2, T>(w, lane, idx, left, valid);
  }
}

// Block sums of the threads' moment partials v (double, or integers of the instance's unit in the
// mixed kernels) into one copy of the accumulators of an instance's stage slot (mixed: acc_slot is that
// copy): reduce-scatter in each warp, one shared-memory row a warp, a half-warp tree a component over up to
// 16 warps, and one fixed-point addition a component.  In a fixed order, so the result depends on the block
// decomposition only.
// ovf: a thread's partial left the integer range (mixed).  A sum that is not finite or out of range
// (FP64: 2^63 and more) rejects an adaptive trial step (reject) and is fatal otherwise.
template <int NM, typename T>
__device__ __forceinline__ void reduce_moments(T (&v)[NM], int ovf, T* red, unsigned long long* acc_slot, int copy,
                                            unsigned long long* errmax, int* nonfinite, bool reject) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int idx = 0, left = NM;
  bool valid = true;
  const T s = reduce_scatter<NM, 16, T>(v, lane, idx, left, valid);
  if (valid) red[warp * NM + idx] = s;
  int any_ovf = 0;
  if constexpr (sizeof(T) == 8 && T(0.5) == T(0)) any_ovf = __syncthreads_or(ovf);     // integers
  else __syncthreads();
  for (int t = threadIdx.x; t < NM * 16; t += blockDim.x) {
    const int c = t >> 4, w = t & 15;
    T x = w < nw ? red[w * NM + c] : T(0);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (w) continue;
    bool ok;
    if constexpr (T(0.5) == T(0)) {
      ok = !any_ovf && x < kFixLimit && x > -kFixLimit;
      if (ok) atomicAdd(acc_slot + 2 * c, (unsigned long long)x);
    } else {
      ok = fx_add(acc_slot, copy, c, x);
    }
    if (!ok) {
      if (reject) atomicMax(errmax, 0x7ff0000000000000ull);
      else atomicExch(nonfinite, 1);
    }
  }
}

// FP64 kernels share one copy of it over their passes (noinline): inlined, its code was out of the
// instruction cache at every pass.
template <int NM>
__device__ __noinline__ void reduce_moments_shared(double (&v)[NM], double* red, unsigned long long* acc_slot, int copy,
                                                   unsigned long long* errmax, int* nonfinite, bool reject) {
  reduce_moments<NM, double>(v, 0, red, acc_slot, copy, errmax, nonfinite, reject);
}

// The block's largest squared error ratio (FP32; infinity where not finite) and non-finite flag.
__device__ __forceinline__ void reduce_error(float em, int bad, float* red, unsigned long long* errmax, int* nonfinite) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) em = fmaxf(em, __shfl_xor_sync(0xffffffffu, em, o));
  if (lane == 0) red[warp] = em;
  const int any_bad = __syncthreads_or(bad);
  if (warp == 0) {
    float m = lane < nw ? red[lane] : 0.0f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) {
      if (any_bad) atomicExch(nonfinite, 1);
      // the beams gave squared error ratios
      atomicMax(errmax, (unsigned long long)__double_as_longlong(sqrt((double)m)));
    }
  }
}

// The serial section of a step's final barrier and of the moment launch, in the last block: the
// instances' stage constants from the accumulators, the controller and the step bookkeeping.  Every value
// another block may have written since this SM last looked is read through L2 (__ldcg), never from a
// possibly stale L1 line; the loads are issued before any branch on them.
template <class Phys, class Tab, typename Real>
__device__ int serial_update(const KParams& p, int slot, bool final_pass, bool init) {
  constexpr int NM = Phys::NM;
  constexpr int NCOMP = NM / 2;
  int all_finished = 1;                            // over this thread's instances
  for (int i = threadIdx.x; i < p.n_inst; i += blockDim.x) {
    const InstConst& ic = p.ic[i];
    InstDyn& d = p.dyn[i];
    const unsigned long long* acc = p.acc + (size_t)i * acc_words_per_inst(sizeof(Real)) + (size_t)slot * acc_words_per_slot(sizeof(Real));
    const bool have_moments = !(final_pass && !Tab::kFinalMoments);
    const bool adaptive_final = final_pass && Tab::kAdaptive && !Tab::kFinalMoments;   // FSAL
    // ---- every load first (no store may sit between them) -------------------------------
    const int done = __ldcg(&d.done), status = __ldcg(&d.status), nonfin = __ldcg(&p.nonfinite[i]);
    const unsigned long long eb = __ldcg(&p.errmax[i]);
    double m[NM];
    if (have_moments) {
#pragma unroll
      for (int c = 0; c < NM; ++c) m[c] = acc_component<Real>(acc, c, ic.acc_unit);
    }
    double m7[NM], sc7[Phys::NSC];
    if (adaptive_final) {
#pragma unroll
      for (int c = 0; c < NM; ++c) m7[c] = __ldcg(&d.mom[Tab::S][c]);
#pragma unroll
      for (int c = 0; c < Phys::NSC; ++c) sc7[c] = __ldcg(&d.sc[Tab::S][c]);
    }
    const int gslot = slot == 0 ? Tab::S : slot;   // slot 0: new state's moments at r + h
    double mu = __ldcg(&d.mus[gslot]), lam = __ldcg(&d.lams[gslot]);
    double r = __ldcg(&d.r), hh = __ldcg(&d.h);
    const double r_end = __ldcg(&d.r_end), r0f = __ldcg(&d.r0_fixed), hf = __ldcg(&d.h_fixed);
    long long nfix = __ldcg(&d.n_fixed);
    const long long nfix_tot = __ldcg(&d.n_fixed_total);
    int last = __ldcg(&d.last), parity = __ldcg(&d.parity);
    unsigned long long accepted = __ldcg(&d.accepted), rejected = __ldcg(&d.rejected);
    unsigned long long evals = __ldcg(&d.stage_evals);
    const double h_min = ic.h_min, h_max = ic.h_max;
    if (done || status) continue;
    if (nonfin) {
      d.status = 5;  // XFLAT_ERR_NONFINITE
      atomicCAS(p.status, 0, 5);
      continue;
    }
    // ---- stage constants of the stage just reduced (the accumulators are cleared elsewhere) --
    if (have_moments) {
      if (init) strengths(ic, __ldcg(&d.rs[slot]), mu, lam);   // the host set only rs[1], xs[1]
      for (int c = 0; c < NM; ++c) d.mom[slot][c] = m[c];
      for (int c = 0; c < NCOMP; ++c) {
        d.sc[slot][c] = mu * m[c];
        d.sc[slot][NCOMP + c] = mu * m[NCOMP + c];
      }
      d.sc[slot][NM] = lam;
    }
    if (!final_pass && !init) {
      all_finished = 0;
      continue;
    }
    // ---- step bookkeeping ---------------------------------------------------------------
    bool fin = false, step_err = false;
    if (init) {
      evals += Tab::kAdaptive ? 1ull : 0ull;
    } else if (!Tab::kAdaptive) {
      parity ^= 1;
      accepted += 1;
      evals += Tab::kEvalsPerStep;
      nfix += 1;
      fin = nfix >= nfix_tot;
      r = fin ? r_end : r0f + (double)nfix * hf;
      // the final pass reduced the new state's moments at r + h (= stage S radius): stage 1 of
      // the next step
      for (int c = 0; c < NM; ++c) d.mom[1][c] = m[c];
      for (int c = 0; c < NCOMP; ++c) {
        d.sc[1][c] = mu * m[c];
        d.sc[1][NCOMP + c] = mu * m[NCOMP + c];
      }
      d.sc[1][NM] = lam;
    } else {
      const double err = __longlong_as_double((long long)eb);
      p.errmax[i] = 0ull;
      d.err = err;
      evals += Tab::kEvalsPerStep;
      const bool ok = err <= 1.0;
      const double q = controller_factor<Tab::kErrPow>(err);
      if (ok) {
        r = last ? r_end : r + hh;
        parity ^= 1;
        accepted += 1;
        if (Tab::kFinalMoments) {
          // the final pass reduced the new state's moments at r + h: stage 1 of the next step
          for (int c = 0; c < NM; ++c) d.mom[1][c] = m[c];
          for (int c = 0; c < NCOMP; ++c) {
            d.sc[1][c] = mu * m[c];
            d.sc[1][NCOMP + c] = mu * m[NCOMP + c];
          }
          d.sc[1][NM] = lam;
        } else {
          for (int c = 0; c < NM; ++c) d.mom[1][c] = m7[c];
          for (int c = 0; c < Phys::NSC; ++c) d.sc[1][c] = sc7[c];
        }
        fin = last != 0;
      } else {
        rejected += 1;
      }
      const double fac = ok ? fmin(5.0, fmax(0.2, q)) : fmax(0.2, q);
      hh = fmin(hh * fac, h_max);
      if (!fin && hh < h_min) {
        d.status = 6;  // XFLAT_ERR_STEP
        atomicCAS(p.status, 0, 6);
        step_err = true;
      }
    }
    // ---- the next step's clipped step size; its stage geometry follows in serial_geometry ----
    if (!fin && Tab::kAdaptive) {
      last = (r + hh >= r_end) ? 1 : 0;
      if (last) hh = r_end - r;
    }
    d.geo_pending = (!fin && !step_err) ? 1 : 0;
    if (i < kGeoShared) {
      GeoHandoff& g = geo_handoff();
      g.r[i] = r;
      g.h[i] = Tab::kAdaptive ? hh : hf;
      g.pending[i] = d.geo_pending;
    }
    d.r = r;
    d.h = hh;
    d.last = last;
    d.parity = parity;
    d.n_fixed = nfix;
    d.accepted = accepted;
    d.rejected = rejected;
    d.stage_evals = evals;
    if (fin) d.done = 1;
    if (!fin && !step_err) all_finished = 0;
  }
  return all_finished;
}

// Accumulator slots of the stages kPasses..S (no pass of their own index clears them), zeroed by
// the last block of the final barrier: nobody accumulates into or reads them until the next step
// (the fence in serial_geometry publishes the stores before the release).
template <class Tab, typename Real>
__device__ void clear_late_slots(const KParams& p) {
  constexpr int kWords = acc_words_per_slot(sizeof(Real));
  constexpr int kLate = Tab::S - Tab::kPasses + 1;
  for (int t = threadIdx.x; t < p.n_inst * kLate * kWords; t += blockDim.x) {
    const int inst = t / (kLate * kWords), rem = t % (kLate * kWords);
    const int slot = Tab::kPasses + rem / kWords;
    p.acc[(size_t)inst * acc_words_per_inst(sizeof(Real)) + (size_t)slot * kWords + rem % kWords] = 0ull;
  }
}

// The next step's stage radii, R^2/r^2, mu and lambda, one (instance, stage) per thread of the last
// block: FP64 divisions have a long latency on this part, so they run side by side, not in a chain.
// Takes r, h and the pending flag from serial_update (after a __syncthreads), then fences every
// thread's writes (those of serial_update included) before the barrier is released.
template <class Tab>
__device__ void serial_geometry(const KParams& p) {
  const GeoHandoff& g = geo_handoff();
  for (int t = threadIdx.x; t < p.n_inst * Tab::S; t += blockDim.x) {
    const int i = t / Tab::S, s = t % Tab::S + 1;
    InstDyn& d = p.dyn[i];
    const bool shared = i < kGeoShared;
    if (!(shared ? g.pending[i] : ldcg(&d.geo_pending))) continue;
    const InstConst& ic = p.ic[i];
    const double r = shared ? g.r[i] : ldcg(&d.r);
    const double h = shared ? g.h[i] : (Tab::kAdaptive ? ldcg(&d.h) : ldcg(&d.h_fixed));
    const double rs = (s == 1) ? r : __dadd_rn(r, __dmul_rn(stage_c<Tab>(s), h));
    const double inv = 1.0 / rs;
    double mus, lams;
    strengths_inv(ic, inv, mus, lams);
    d.rs[s] = rs;
    d.xs[s] = ic.R2 * inv * inv;
    d.mus[s] = mus;
    d.lams[s] = lams;
  }
  __threadfence();
}


// ---------------------------------------------------------------------------------------------
// State ring of the FP32 two-flavour bulb passes.  Each thread streams its beams' state through a
// private ring of kStateRingDepth + 1 slots in shared memory, filled by cp.async (LDGSTS)
// kStateRingDepth vectors ahead of the one being processed: several vectors' bytes in flight per
// thread without holding registers for them.  (Measured on GB300 against one register-held
// prefetch vector, against 2 and 5 vectors ahead, and against a per-warp ring of 256-byte bulk
// copies completing on mbarriers, which was slower on every launch shape.)  The slots are
// thread-private, so the only ordering needed is the thread's own cp.async.wait_group.
template <class Phys, typename Real>
__host__ __device__ constexpr bool state_ring() {
  return Phys::NC == 3 && Phys::NM == 6 && sizeof(Real) == 4;
}
__device__ __forceinline__ uint32_t smem_addr(const void* ptr) {
  return (uint32_t)__cvta_generic_to_shared(ptr);
}
__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// wait until at most N of this thread's committed groups are pending
template <int N>
__device__ __forceinline__ void cp_async_wait_pending() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Consecutive beams a thread takes at once: two in the FP32 two-flavour kernels (packed pairs), one in
// the others (their pass bodies are long, a second copy for the second beam only fills the instruction
// cache, and FP64 stage planes are then read and written in full 256-byte rows).
template <class Phys, typename Real>
__host__ __device__ constexpr int vec_beams() { return Phys::NC == 3 && sizeof(Real) == 4 ? 2 : 1; }

template <typename Real, int N>
__device__ __forceinline__ void vload(const Real* p, Real (&v)[N]) {
  if constexpr (N == 1) {
    v[0] = __ldcg(p);
  } else {
    const float2 t = __ldcg(reinterpret_cast<const float2*>(p));
    v[0] = t.x;
    v[1] = t.y;
  }
}
template <typename Real, int N>
__device__ __forceinline__ void vstore(Real* p, const Real (&v)[N]) {
  if constexpr (N == 1) __stcg(p, v[0]);
  else __stcg(reinterpret_cast<float2*>(p), make_float2(v[0], v[1]));
}

// Plane accesses of the pass body, checked in the checked build (site: where, for the record).
template <typename Real, int N>
__device__ __forceinline__ void vload_at(const KParams& p, int span, const Real* ptr, Real (&v)[N], int site) {
  if (XFLAT_SPAN_OK(p, span, ptr, N * sizeof(Real), site)) {
    vload(ptr, v);
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = Real(0);
  }
}
template <typename Real, int N>
__device__ __forceinline__ void vstore_at(const KParams& p, int span, Real* ptr, const Real (&v)[N], int site) {
  if (XFLAT_SPAN_OK(p, span, ptr, N * sizeof(Real), site)) vstore(ptr, v);
}

// sqrt(x) and 1/sqrt(x) to rounding: Newton steps from the hardware's FP32 reciprocal square root, no
// division (the library's FP64 square root and division are chains of 673 and 429 cycles on GB300; only an
// FP64 x beyond the seed's range takes them, by a test on its bits: an FP64 comparison there cost 1 % of a
// call of 8 Lie RK4 steps of 4096 beams).  x is at least about 1e-10 (FP32: 1e-6), see rotate.
static __device__ __noinline__ void sqrt_pair_library(double x, double& t, double& r) {
  t = sqrt(x);
  r = 1.0 / t;
}
__device__ __forceinline__ void sqrt_pair(float x, float& t, float& r) {
  r = rsqrtf(x);
  r = fmaf(0.5f * r, fmaf(-x * r, r, 1.0f), r);
  t = x * r;
  t = fmaf(0.5f * r, fmaf(-t, t, x), t);
}
__device__ __forceinline__ void sqrt_pair(double x, double& t, double& r) {
  if (__double2hiint(x) >= 0x47e00000) {                       // 2^127 and more, or not a number
    sqrt_pair_library(x, t, r);
    return;
  }
  r = (double)rsqrtf((float)x);
  r = fma(0.5 * r, fma(-x * r, r, 1.0), r);
  r = fma(0.5 * r, fma(-x * r, r, 1.0), r);
  t = x * r;
  t = fma(0.5 * r, fma(-t, t, x), t);
}

// Rotation of y about Om by |Om| (right-handed): y + a Om x y + b Om x (Om x y), the Bloch form of
// y -> U y U^dagger with U = exp(-i Om.sigma/2), i.e. the propagator of Eq. U; a = sin t / t and
// b = (1 - cos t) / t^2 = (sin(t/2) / t)^2 2 from the half angle, without cancellation.
template <typename Real>
__device__ __forceinline__ void rotate(const Real (&Om)[3], Real (&y)[3]) {
  const Real t2 = Om[0] * Om[0] + Om[1] * Om[1] + Om[2] * Om[2];
  Real a, b;
  bool tiny;
  if constexpr (sizeof(Real) == 4) tiny = !(t2 > Real(1e-3) * Real(1e-3));
  else tiny = __double2hiint(t2) < 0x3ddb7cdf;                 // below about 1e-10, from the leading bits
  if (!tiny) {
    Real t, r, sh, ch;
    sqrt_pair(t2, t, r);
    if constexpr (sizeof(Real) == 4) sincosf(0.5f * t, &sh, &ch);
    else sincos(0.5 * t, &sh, &ch);
    const Real sr = sh * r;
    a = Real(2) * sr * ch;
    b = Real(2) * sr * sr;
  } else {
    a = Real(1) - t2 * Real(1.0 / 6.0);
    b = Real(0.5) - t2 * Real(1.0 / 24.0);
  }
  const Real c0 = Om[1] * y[2] - Om[2] * y[1];
  const Real c1 = Om[2] * y[0] - Om[0] * y[2];
  const Real c2 = Om[0] * y[1] - Om[1] * y[0];
  const Real d0 = Om[1] * c2 - Om[2] * c1;
  const Real d1 = Om[2] * c0 - Om[0] * c2;
  const Real d2 = Om[0] * c1 - Om[1] * c0;
  y[0] += a * c0 + b * d0;
  y[1] += a * c1 + b * d1;
  y[2] += a * c2 + b * d2;
}

// Helpers of propagate3 in the working precision.  expo: the largest biased exponent of the entries,
// from their bits (integer pipe); pow2: the power of two of a biased exponent.
__device__ __forceinline__ int expo_bits(float v) { return __float_as_int(v) & 0x7fffffff; }
__device__ __forceinline__ int expo_bits(double v) { return __double2hiint(v) & 0x7fffffff; }
template <typename Real> __device__ __forceinline__ Real pow2_biased(int e) {
  if constexpr (sizeof(Real) == 4) return __int_as_float(e << 23);
  else return __hiloint2double(e << 20, 0);
}
__device__ __forceinline__ void sincos_of(float x, float& s, float& c) { sincosf(x, &s, &c); }
__device__ __forceinline__ void sincos_of(double x, double& s, double& c) { sincos(x, &s, &c); }
// The root of largest modulus of l^3 - c1 l - c0 = 0 (three real roots, c1 > 0; it is at least
// sqrt(c1) in modulus and the derivative there at least 2 c1, so Newton's iteration is well
// conditioned).  Seed: with l = sqrt(c1) m the equation is m^3 - m = a, a = |c0| c1^-3/2 in
// [0, 0.385], whose root a cubic in a gives to 5e-5.
__device__ __forceinline__ float largest_root_seed(float c1, float c0) {
  const float rn = rsqrtf(c1);
  const float a = fminf(fabsf(c0) * rn * rn * rn, 0.3849002f);
  float m = fmaf(fmaf(fmaf(0.1887236f, a, -0.3171565f), a, 0.4959911f), a, 1.0000473f);
  m -= __fdividef(fmaf(m, fmaf(m, m, -1.0f), -a), fmaf(3.0f * m, m, -1.0f));
  return copysignf(m * (c1 * rn), c0);
}
__device__ __forceinline__ float largest_root(float c1, float c0) {
  const float m = largest_root_seed(c1, c0);
  return m - __fdividef(fmaf(m, fmaf(m, m, -c1), -c0), fmaf(3.0f * m, m, -c1));
}
__device__ __forceinline__ double largest_root(double c1, double c0) {
  // two corrections with the FP32 slope: each multiplies the error (1e-7 at first) by ~1e-7
  const float c1f = (float)c1, mf = largest_root_seed(c1f, (float)c0);
  const double inv = (double)__fdividef(1.0f, fmaf(3.0f * mf, mf, -c1f));
  double m = (double)mf;
  m = fma(-inv, fma(m, fma(m, m, -c1), -c0), m);
  return fma(-inv, fma(m, fma(m, m, -c1), -c0), m);
}
// 1/sqrt(x) of an x of the order of one, and w, 1/w of w2 = w^2 >= 0 (w = 0 where w2 underflows):
// Newton steps from the hardware's FP32 values (GB300's FP64 division and square root are long
// dependent chains)
__device__ __forceinline__ float rnorm1(float x) {
  const float r = rsqrtf(x);
  return fmaf(0.5f * r, fmaf(-x * r, r, 1.0f), r);
}
__device__ __forceinline__ double rnorm1(double x) {
  double r = (double)rsqrtf((float)x);
  r = fma(0.5 * r, fma(-x * r, r, 1.0), r);
  return fma(0.5 * r, fma(-x * r, r, 1.0), r);
}
__device__ __forceinline__ void root_pair(float w2, float& w, float& rw) {
  w = sqrtf(w2);
  rw = __fdividef(1.0f, w);
}
__device__ __forceinline__ void root_pair(double w2, double& w, double& rw) {
  const float f = (float)w2;
  if (!(f >= 1.0e-36f)) { w = w2 == w2 ? 0.0 : w2; rw = w; return; }   // far below the rounding of Q
  double r = (double)rsqrtf(f);
  r = fma(0.5 * r, fma(-w2 * r, r, 1.0), r);
  rw = fma(0.5 * r, fma(-w2 * r, r, 1.0), r);
  w = w2 * rw;
}

// Three flavours: y <- U y U^dagger with U = exp(-i Om) for Hermitian Om (8 reals: the 00 and 11
// entries less the 22 entry, then real and imaginary parts of the 01, 02 and 12 entries), the
// propagator of Eq. U for a 3 x 3 generator; a phase of U and a multiple of the unit matrix in Om
// drop out.
//
// Closed form on the traceless Q = Om / s (s a power of two, largest entry in [1, 2)).  Its
// characteristic polynomial is l^3 - c1 l - c0 (c1 = tr Q^2 / 2, c0 = det Q); m = 2u, the root of
// largest modulus, is at least sqrt(3 c1)/2 away from the other two, -u + w and -u - w, so its
// eigenvector v, a column of Q^2 + m Q + (m^2 - c1) = (3 m^2 - c1) v v^dagger (Cayley-Hamilton), is
// well conditioned even when the other two nearly coincide (matter far above the vacuum
// splittings).  On the complement of P = v v^dagger the generator is -u + C with the traceless
// C = Q + u - 3u P, C^2 = w^2 (1 - P), hence
//   U e^{-ius} = e^{-3ius} P + cos(ws) (1 - P) - i sin(ws)/w C.
// w comes from the entries of C, not from c1 - 3u^2, whose cancellation would cost eps |Om|^2
// instead of eps |Om| in the phases; and C is first projected onto the traceless matrices on the
// complement of v, because the rounding of its entries (eps, where C itself is w) would otherwise
// make U non-unitary by eps |Om|: that moves whole flavours, not only phases, and near the neutrino
// sphere it throttled the adaptive step.  With it U is unitary to about ten roundings at any |Om|.
// About 470 operations, against about 2200 instructions of a cyclic-Jacobi eigen-decomposition
// (262,144 beams, mixed adaptive Lie RK4 on GB300, a call of 5 attempted steps: 5.08 ms with Jacobi
// sweeps, 1.98 ms so; largest error against 64 bits over random Om of norms 1e-8 .. 1e4,
// relative to max(1, |Om|): 0.2e-6 to 0.7e-6 against 1.3e-6 to 1.9e-6 in FP32, 1.5e-15 to 2.7e-15
// against 3e-15 to 5e-15 in FP64).
template <typename Real>
__device__ __noinline__ void propagate3(const Real (&Om)[8], Real (&y)[9]) {
  Real xr = Om[2], xi = Om[3], yr = Om[4], yi = Om[5], zr = Om[6], zi = Om[7];
  const Real t = (Om[0] + Om[1]) * Real(1.0 / 3.0);
  Real q0 = Om[0] - t, q1 = Om[1] - t, q2 = -t;
  constexpr int kMant = sizeof(Real) == 4 ? 23 : 20, kMaxE = sizeof(Real) == 4 ? 253 : 2045;
  int eb = max(max(expo_bits(q0), expo_bits(q1)), expo_bits(q2));
  eb = max(eb, max(max(expo_bits(xr), expo_bits(xi)), max(expo_bits(yr), expo_bits(yi))));
  eb = max(eb, max(expo_bits(zr), expo_bits(zi)));
  const int E = min(eb >> kMant, kMaxE);
  if (E == 0) return;                                       // Om = 0 (or denormal)
  const Real s = pow2_biased<Real>(E), inv = pow2_biased<Real>(kMaxE + 1 - E);
  q0 *= inv; q1 *= inv; q2 *= inv;
  xr *= inv; xi *= inv; yr *= inv; yi *= inv; zr *= inv; zi *= inv;
  // M = Q^2 first, its entries 00, 11, 22, 01, 02, 12
  const Real x2 = xr * xr + xi * xi, y2 = yr * yr + yi * yi, z2 = zr * zr + zi * zi;
  Real m00 = q0 * q0 + (x2 + y2), m11 = q1 * q1 + (x2 + z2), m22 = q2 * q2 + (y2 + z2);
  const Real xzr = xr * zr - xi * zi, xzi = xr * zi + xi * zr;         // x z
  Real m01r = yr * zr + yi * zi - q2 * xr, m01i = yi * zr - yr * zi - q2 * xi;
  Real m02r = xzr - q1 * yr, m02i = xzi - q1 * yi;
  Real m12r = xr * yr + xi * yi - q0 * zr, m12i = xr * yi - xi * yr - q0 * zi;
  const Real c1 = Real(0.5) * (m00 + m11 + m22);
  const Real c0 = q0 * (q1 * q2 - z2) - q1 * y2 - q2 * x2 + Real(2) * (xzr * yr + xzi * yi);
  const Real m = largest_root(c1, c0), u = Real(0.5) * m;
  // M = (3 m^2 - c1) v v^dagger
  const Real e = m * m - c1;
  m00 += m * q0 + e; m11 += m * q1 + e; m22 += m * q2 + e;
  m01r += m * xr; m01i += m * xi; m02r += m * yr; m02i += m * yi; m12r += m * zr; m12i += m * zi;
  // v: the column of M with the largest diagonal entry, normalised
  const bool b1 = m11 > m00 && m11 >= m22, b2 = !b1 && m22 > m00;
  Real v0r = b1 ? m01r : b2 ? m02r : m00, v0i = b1 ? m01i : b2 ? m02i : Real(0);
  Real v1r = b1 ? m11 : b2 ? m12r : m01r, v1i = b1 ? Real(0) : b2 ? m12i : -m01i;
  Real v2r = b1 ? m12r : b2 ? m22 : m02r, v2i = b1 ? -m12i : b2 ? Real(0) : -m02i;
  const Real rn = rnorm1((v0r * v0r + v0i * v0i) + (v1r * v1r + v1i * v1i) + (v2r * v2r + v2i * v2i));
  v0r *= rn; v0i *= rn; v1r *= rn; v1i *= rn; v2r *= rn; v2i *= rn;
  const Real p00 = v0r * v0r + v0i * v0i, p11 = v1r * v1r + v1i * v1i, p22 = v2r * v2r + v2i * v2i;
  const Real p01r = v0r * v1r + v0i * v1i, p01i = v0i * v1r - v0r * v1i;
  const Real p02r = v0r * v2r + v0i * v2i, p02i = v0i * v2r - v0r * v2i;
  const Real p12r = v1r * v2r + v1i * v2i, p12i = v1i * v2r - v1r * v2i;
  // C = Q + u - 3u P (in q0 .. zi), then its projection C - v h^dagger - h v^dagger - (tau/2)(1 - P)
  // with r = C v, h = r - (v^dagger r / 2 + tau / 4) v and tau the trace left on the complement
  const Real k = Real(3) * u;
  q0 = (q0 + u) - k * p00; q1 = (q1 + u) - k * p11; q2 = (q2 + u) - k * p22;
  xr -= k * p01r; xi -= k * p01i; yr -= k * p02r; yi -= k * p02i; zr -= k * p12r; zi -= k * p12i;
  Real w2;
  {
    Real r0r = q0 * v0r + xr * v1r - xi * v1i + yr * v2r - yi * v2i;
    Real r0i = q0 * v0i + xr * v1i + xi * v1r + yr * v2i + yi * v2r;
    Real r1r = xr * v0r + xi * v0i + q1 * v1r + zr * v2r - zi * v2i;
    Real r1i = xr * v0i - xi * v0r + q1 * v1i + zr * v2i + zi * v2r;
    Real r2r = yr * v0r + yi * v0i + zr * v1r + zi * v1i + q2 * v2r;
    Real r2i = yr * v0i - yi * v0r + zr * v1i - zi * v1r + q2 * v2i;
    const Real rho = (v0r * r0r + v0i * r0i) + (v1r * r1r + v1i * r1i) + (v2r * r2r + v2i * r2i);
    const Real tau = (q0 + q1 + q2) - rho;
    const Real hh = Real(0.5) * rho + Real(0.25) * tau, ht = Real(0.5) * tau;
    r0r -= hh * v0r; r0i -= hh * v0i; r1r -= hh * v1r; r1i -= hh * v1i; r2r -= hh * v2r; r2i -= hh * v2i;
    q0 = (q0 - ht) - Real(2) * (v0r * r0r + v0i * r0i);
    q1 = (q1 - ht) - Real(2) * (v1r * r1r + v1i * r1i);
    q2 = (q2 - ht) - Real(2) * (v2r * r2r + v2i * r2i);
    xr -= v0r * r1r + v0i * r1i + r0r * v1r + r0i * v1i;
    xi -= v0i * r1r - v0r * r1i + r0i * v1r - r0r * v1i;
    yr -= v0r * r2r + v0i * r2i + r0r * v2r + r0i * v2i;
    yi -= v0i * r2r - v0r * r2i + r0i * v2r - r0r * v2i;
    zr -= v1r * r2r + v1i * r2i + r1r * v2r + r1i * v2i;
    zi -= v1i * r2r - v1r * r2i + r1i * v2r - r1r * v2i;
    w2 = Real(0.5) * (q0 * q0 + q1 * q1 + q2 * q2) + (xr * xr + xi * xi) + (yr * yr + yi * yi) + (zr * zr + zi * zi);
  }
  Real w, rw, sw, cw, s3, c3;
  root_pair(w2, w, rw);
  sincos_of(w * s, sw, cw);
  sincos_of(k * s, s3, c3);
  const Real g = w == Real(0) ? s : sw * rw;
  const Real br = c3 - cw, bi = -s3;
  // U = cw (1 - P) + e^{-3ius} P - i g C, entry by entry (on the diagonal 1 - P is the sum of the other
  // two entries of P: nothing cancels where P is nearly a flavour)
  const Real u00r = c3 * p00 + cw * (p11 + p22), u00i = bi * p00 - g * q0;
  const Real u11r = c3 * p11 + cw * (p00 + p22), u11i = bi * p11 - g * q1;
  const Real u22r = c3 * p22 + cw * (p00 + p11), u22i = bi * p22 - g * q2;
  Real u01r, u01i, u10r, u10i, u02r, u02i, u20r, u20i, u12r, u12i, u21r, u21i;
  auto pair = [&](Real pr, Real pi, Real qr, Real qi, Real& ur, Real& ui, Real& lr, Real& li) {
    const Real a1 = br * pr, a2 = bi * pi - g * qi, b1 = bi * pr - g * qr, b2 = br * pi;
    ur = a1 - a2; ui = b1 + b2;
    lr = a1 + a2; li = b1 - b2;
  };
  pair(p01r, p01i, xr, xi, u01r, u01i, u10r, u10i);
  pair(p02r, p02i, yr, yi, u02r, u02i, u20r, u20i);
  pair(p12r, p12i, zr, zi, u12r, u12i, u21r, u21i);
  // row a of T = U Y, then the entries (a, b >= a) of T U^dagger
  const Real ar = y[3], ai = y[4], hr = y[5], hi = y[6], cr = y[7], ci = y[8];
  auto row = [&](Real v0r, Real v0i, Real v1r, Real v1i, Real v2r, Real v2i, Real (&tr)[3], Real (&ti)[3]) {
    tr[0] = v0r * y[0] + v1r * ar + v1i * ai + v2r * hr + v2i * hi;
    ti[0] = v0i * y[0] + v1i * ar - v1r * ai + v2i * hr - v2r * hi;
    tr[1] = v0r * ar - v0i * ai + v1r * y[1] + v2r * cr + v2i * ci;
    ti[1] = v0i * ar + v0r * ai + v1i * y[1] + v2i * cr - v2r * ci;
    tr[2] = v0r * hr - v0i * hi + v1r * cr - v1i * ci + v2r * y[2];
    ti[2] = v0i * hr + v0r * hi + v1i * cr + v1r * ci + v2i * y[2];
  };
  Real tr[3], ti[3], n0, n1, n2, n3, n4, n5, n6, n7, n8;
  row(u00r, u00i, u01r, u01i, u02r, u02i, tr, ti);
  n0 = tr[0] * u00r + ti[0] * u00i + tr[1] * u01r + ti[1] * u01i + tr[2] * u02r + ti[2] * u02i;
  n3 = tr[0] * u10r + ti[0] * u10i + tr[1] * u11r + ti[1] * u11i + tr[2] * u12r + ti[2] * u12i;
  n4 = ti[0] * u10r - tr[0] * u10i + ti[1] * u11r - tr[1] * u11i + ti[2] * u12r - tr[2] * u12i;
  n5 = tr[0] * u20r + ti[0] * u20i + tr[1] * u21r + ti[1] * u21i + tr[2] * u22r + ti[2] * u22i;
  n6 = ti[0] * u20r - tr[0] * u20i + ti[1] * u21r - tr[1] * u21i + ti[2] * u22r - tr[2] * u22i;
  row(u10r, u10i, u11r, u11i, u12r, u12i, tr, ti);
  n1 = tr[0] * u10r + ti[0] * u10i + tr[1] * u11r + ti[1] * u11i + tr[2] * u12r + ti[2] * u12i;
  n7 = tr[0] * u20r + ti[0] * u20i + tr[1] * u21r + ti[1] * u21i + tr[2] * u22r + ti[2] * u22i;
  n8 = ti[0] * u20r - tr[0] * u20i + ti[1] * u21r - tr[1] * u21i + ti[2] * u22r - tr[2] * u22i;
  row(u20r, u20i, u21r, u21i, u22r, u22i, tr, ti);
  n2 = tr[0] * u20r + ti[0] * u20i + tr[1] * u21r + ti[1] * u21i + tr[2] * u22r + ti[2] * u22i;
  y[0] = n0; y[1] = n1; y[2] = n2; y[3] = n3; y[4] = n4; y[5] = n5; y[6] = n6; y[7] = n7; y[8] = n8;
}

// The propagator of Eq. U over one step for the generator Om (step length and coefficients folded
// in): y <- exp(-i Om) y exp(i Om).  Two flavours: the rotation of the Bloch vector; three
// flavours: the closed form of propagate3.
template <typename Real>
__device__ __forceinline__ void propagate(const Real (&Om)[3], Real (&y)[3]) { rotate(Om, y); }
template <typename Real>
__device__ __forceinline__ void propagate(const Real (&Om)[8], Real (&y)[9]) { propagate3(Om, y); }

// Per-block shared state of the piece being processed.
template <typename Real, class Phys>
struct BlockShared {
  double xs[kMaxStages];               // R^2 / r_s^2
  int t1max[kMaxStages];               // FP32 kernels: bits of the largest t1 of the piece's rows of a stage
  Real scr[kMaxStages][Phys::NSC];     // stage constants in working precision
  Real hA[kMaxStages][kMaxStages];     // tableau coefficients times h (scaled_rows: the coefficients)
  Real hB[kMaxStages];
  Real hE[kMaxStages];
  Real rtol, atol;
  float rtol_f, atol_f, inv_tol;       // FP64 error filter: tolerances times inv_tol = 1 / (rtol + atol)
  int emax_f;                          // bits of the largest squared error ratio found in the piece so far (rounded down)
  int active;
  int parity;
  int flag;
  int pass_idx;                        // passes run by this block in this launch (pass trace)
  int next_piece;                      // dynamic scheduling: the piece this block processes next
  int keep;                            // single-piece block: launch-invariant set-up already loaded
  unsigned int gen_seen;               // barrier generation this block arrived in
  unsigned int expected;               // arrivals a pass barrier waits for
  unsigned long long pass_next;        // pass_barrier's count
};

// Table view: row (stage s, combined angle index tj) holds Phys::KT values.
template <typename Real, class Phys>
struct TabView {
  const Real* t;
  int n_jj;
  __device__ __forceinline__ const Real* row(int s, int tj) const {
    return t + ((size_t)s * n_jj + tj) * Phys::KT;
  }
};

// The FP32 value of a double's leading 21 bits (truncated), from its high word on the integer pipe;
// zero below 2^-126, infinite or not a number from 2^128 on.
__device__ __forceinline__ float lead_f32(double x) {
  const int h = __double2hiint(x), e = ((h >> 20) & 0x7ff) - 896;
  const int m = (h & 0xfffff) << 3;
  const int bits = e <= 0 ? 0 : e >= 255 ? (0x7f800000 | ((h & 0x7ff00000) == 0x7ff00000 ? m : 0)) : (e << 23) | m;
  return __int_as_float(bits | (h & 0x80000000));
}
__device__ __forceinline__ float lead_f32(float x) { return x; }

// What a pass does (compile time).
enum PassKind : int { kStagePass = 0, kFinalPass = 1, kInitPass = 2 };

// Adaptive FP64 kernels split the last two passes of a step: the pass forming Y_S (= y5, first
// same as last) also stores y5 and the error partial sum over stages 1..S-1, and the final pass only
// adds k_S -- the stage chain costs FP64 instructions on GB300's narrow FP64
// pipe.  FP32 kernels rebuild the chain in the final pass instead: their state, y5 and those
// partials together exceed the L2, and the extra DRAM traffic costs more than the FP32 chain.
template <class Tab, typename Real>
__host__ __device__ constexpr bool split_final() {
  return Tab::kAdaptive && !Tab::kFinalMoments && !Tab::kEM2 && sizeof(Real) == 8;   // DP45 in FP64
}

// FP64 commutator tableaus (RK4, DP45) keep their stage derivatives in HBM: the pass that
// evaluates k_s writes it, later passes of the step read it back instead of rebuilding the chain.
// On GB300 an FP64 stage evaluation costs far more time than moving its 8 bytes per component
// (the FP64 pipe runs at ~1/68 of the FP32 rate), so a DP45 step evaluates 7 stages instead of
// the 28 of the rebuilt chain.  FP32 kernels rebuild: their stage vectors would push the state out
// of the L2.  The stored values are bit-identical to rebuilt ones (same inputs, same arithmetic).
template <class Tab, typename Real>
__host__ __device__ constexpr bool stored_stages() {
  return !Tab::kEM2 && sizeof(Real) == 8;
}
// Stage derivatives a step stores (k_1 .. k_n): every stage whose derivative a later pass needs.
template <class Tab, typename Real>
__host__ __device__ constexpr int stored_stage_count() {
  return split_final<Tab, Real>() ? Tab::S - 2 : Tab::S - 1;
}

template <class Phys, class Tab, typename Real, bool kCF, int kPass, int kKind>
struct PassBody;

// Commutator-form Runge-Kutta (RK4 / DP45) ------------------------------------------------------
template <class Phys, class Tab, typename Real, int kPass, int kKind>
struct PassBody<Phys, Tab, Real, false, kPass, kKind> {
  static constexpr int NC = Phys::NC;
  static constexpr bool kWriteOut = false, kReadOut = false, kReadBoth = false;
  static constexpr bool kSplit = split_final<Tab, Real>();
  // number of stage derivatives the pass needs before its stage state, rebuilt or (stored stages)
  // read back (split final pass: none, the pass forming Y_S left y5 and the error partial behind;
  // unsplit adaptive: S - 1, k_S follows from the new state)
  static constexpr int kChain =
      kKind == kInitPass ? 0
      : (kKind == kFinalPass ? (kSplit ? 0 : Tab::S - (Tab::kAdaptive ? 1 : 0)) : kPass + 1);
  // stored stage derivatives (stored_stages): all of the chain but its last stage are read back,
  // and a stage pass writes the one it evaluates when a later pass of the step reads it
  static constexpr bool kStore = stored_stages<Tab, Real>();
  static constexpr int kLoadK = (kStore && kChain > 0) ? kChain - 1 : 0;
  static constexpr bool kStoreK = kStore && kKind == kStagePass && kChain <= stored_stage_count<Tab, Real>();
  // the stage state the chain evaluates last, Y_kChain, is the one the previous pass formed for its
  // moments: stored there (plane set after the stage derivatives) and read back here
  static constexpr bool kLoadY = kStore && kChain >= 2;
  static constexpr bool kStoreY = kStore && kKind == kStagePass && !(kSplit && kPass + 2 == Tab::S);
  static constexpr int kYPlanes = stored_stage_count<Tab, Real>();
  // y: the step's state.  Split final pass: the pass forming Y_S replaces y by the new state
  // y5 = Y_S and sets ep, the error partial sum over stages 1..S-1; the final pass gets y5 in y, that
  // ep back, and the step's state in yo.  kst: this beam's element of the stage-derivative
  // planes (component i of k_l at kst[((l - 1) NC + i) kstride]), read and written by this thread
  // only.
  template <class BS, class Acc>
  __device__ static inline void beam(BS& bs, const typename Phys::Beam& bm,
                                     const TabView<Real, Phys>& tv, int tj, Real (&y)[NC],
                                     Real (&ep)[NC], const Real (&yo)[NC],
                                     Acc& acc, Real& emax, int& bad, bool mixed,
                                     Real* kst, size_t kstride) {
    Real k[Tab::S + 1][NC];
#pragma unroll
    for (int l = 1; l <= kLoadK; ++l)
#pragma unroll
      for (int i = 0; i < NC; ++i) k[l][i] = kst[((size_t)(l - 1) * NC + i) * kstride];
#pragma unroll
    for (int l = kLoadK + 1; l <= kChain; ++l) {
      Real Y[NC];
      if constexpr (kLoadY) {
#pragma unroll
        for (int i = 0; i < NC; ++i) Y[i] = kst[((size_t)kYPlanes * NC + i) * kstride];
      } else {
#pragma unroll
        for (int i = 0; i < NC; ++i) {
          Real v = y[i];
#pragma unroll
          for (int m = 1; m < l; ++m)
            if (Tab::a(l, m) != 0.0) v += bs.hA[l][m] * k[m][i];
          Y[i] = v;
        }
      }
      Real Kv[Phys::NG];
      Phys::K(tv.row(l, tj), bm, Kv);
      Phys::f(Kv, Y, k[l]);
    }
    if constexpr (kStoreK) {
#pragma unroll
      for (int i = 0; i < NC; ++i) kst[((size_t)(kChain - 1) * NC + i) * kstride] = k[kChain][i];
    }
    if (kKind == kInitPass) {
      Phys::accum_row(acc, bm.w, tv.row(1, tj), y);
      return;
    }
    if (kKind == kStagePass) {
      constexpr int I = kPass + 2;
      Real Y[NC];
#pragma unroll
      for (int i = 0; i < NC; ++i) {
        Real v = y[i];
#pragma unroll
        for (int m = 1; m < I; ++m)
          if (Tab::a(I, m) != 0.0) v += bs.hA[I][m] * k[m][i];
        Y[i] = v;
      }
      if (kSplit && I == Tab::S) {
        // first same as last: Y_S is the new state y5 (row S of A is b).  Its error partial sum
        // over stages 1..S-1 goes with it, so the final pass needs only k_S.
        if (mixed) Phys::normalise(Y);
#pragma unroll
        for (int i = 0; i < NC; ++i) {
          Real v = 0;
#pragma unroll
          for (int m = 1; m < Tab::S; ++m)
            if (Tab::e(m) != 0.0) v += bs.hE[m] * k[m][i];
          ep[i] = v;
        }
        Phys::accum_row(acc, bm.w, tv.row(I, tj), Y);
#pragma unroll
        for (int i = 0; i < NC; ++i) y[i] = Y[i];
        return;
      }
      if (Tab::kAdaptive && I == Tab::S && mixed) Phys::normalise(Y);
      if constexpr (kStoreY) {
#pragma unroll
        for (int i = 0; i < NC; ++i) kst[((size_t)kYPlanes * NC + i) * kstride] = Y[i];
      }
      Phys::accum_row(acc, bm.w, tv.row(I, tj), Y);
      return;
    }
    if (Tab::kAdaptive && !kSplit) {
      // final pass: y5 from the rebuilt chain, k_S = f(y5), the embedded error and the squared
      // error ratio (its square root is taken once per block)
      Real yn[NC];
#pragma unroll
      for (int i = 0; i < NC; ++i) {
        Real v = y[i];
#pragma unroll
        for (int m = 1; m <= kChain; ++m)
          if (Tab::b(m) != 0.0) v += bs.hB[m] * k[m][i];
        yn[i] = v;
      }
      const bool ynok = Phys::tnorm2(yn) <= rbig<Real>();
      if (mixed && ynok) Phys::normalise(yn);
      if (!(Phys::tnorm2(y) <= rbig<Real>())) bad = 1;     // non-finite input state: fatal
      Real Kv[Phys::NG];
      Phys::K(tv.row(Tab::S, tj), bm, Kv);
      Phys::f(Kv, yn, k[Tab::S]);
      Real e[NC];
#pragma unroll
      for (int i = 0; i < NC; ++i) {
        Real v = 0;
#pragma unroll
        for (int m = 1; m <= Tab::S; ++m)
          if (Tab::e(m) != 0.0) v += bs.hE[m] * k[m][i];
        e[i] = v;
      }
      const Real den = bs.atol + bs.rtol * sqrt(fmax(Phys::tnorm2(y), Phys::tnorm2(yn)));
      Real r2 = Phys::tnorm2(e) / (den * den);
      if (!(r2 <= rbig<Real>()) || !ynok) r2 = Real(INFINITY);
      emax = fmax(emax, r2);
#pragma unroll
      for (int i = 0; i < NC; ++i) y[i] = yn[i];
      return;
    }
    if (Tab::kAdaptive) {
      // split final pass (y holds y5, whose moments the pass before reduced): k_S = f(y5), the embedded
      // error, and the squared error ratio (its square root is taken once per block).  Only the largest
      // ratio counts: an FP32 estimate of it (components by their leading 21 bits; never below the ratio
      // by more than the 1e-3 it is raised by, norm_floor) passes over every beam that cannot exceed the
      // largest found so far in the block, so the FP64 norms, square root and division -- a fifth of a
      // DP45 step's FP64 work -- are left for a few beams a block.
      Real Kv[Phys::NG], kS[NC], e[NC];
      Phys::K(tv.row(Tab::S, tj), bm, Kv);
      Phys::f(Kv, y, kS);
#pragma unroll
      for (int i = 0; i < NC; ++i) e[i] = ep[i] + bs.hE[Tab::S] * kS[i];
      float ef[NC], yf[NC], of[NC];
#pragma unroll
      for (int i = 0; i < NC; ++i) {
        ef[i] = lead_f32(e[i]) * bs.inv_tol;
        yf[i] = lead_f32(y[i]);
        of[i] = lead_f32(yo[i]);
      }
      using P32 = typename Phys::template With<float>;
      const float df = bs.atol_f + bs.rtol_f * P32::norm_floor(of, yf);
      const float rf = __fdividef(P32::tnorm2(ef), df * df);
      // also where rf is not a number, and where the squares leave FP32's range: with df above 1e-12 they
      // lose bits only where the squared ratio is below 1e-13
      const float found = __int_as_float(*(volatile int*)&bs.emax_f);
      if (!(rf * 1.001f < found && found > 1.0e-13f && df > 1.0e-12f && df < 1.0e18f)) {
        const Real no = Phys::tnorm2(yo), n5 = Phys::tnorm2(y);
        if (!(no <= rbig<Real>())) bad = 1;                     // non-finite input state: fatal
        const Real den = bs.atol + bs.rtol * sqrt(fmax(no, n5));
        Real r2 = Phys::tnorm2(e) / (den * den);
        // a trial step whose stages overflowed the working precision is rejected, not fatal
        if (!(r2 <= rbig<Real>()) || !(n5 <= rbig<Real>())) r2 = Real(INFINITY);
        emax = fmax(emax, r2);
        atomicMax(&bs.emax_f, __float_as_int(__double2float_rd((double)fmin(r2, Real(3.0e38)))));
      }
      return;
    }
    // final pass of a fixed-step tableau
    Real yn[NC];
#pragma unroll
    for (int i = 0; i < NC; ++i) {
      Real v = y[i];
#pragma unroll
      for (int m = 1; m <= kChain; ++m)
        if (Tab::b(m) != 0.0) v += bs.hB[m] * k[m][i];
      yn[i] = v;
    }
    const bool ynok = Phys::tnorm2(yn) <= rbig<Real>();
    if (mixed && ynok) Phys::normalise(yn);
    Phys::accum_row(acc, bm.w, tv.row(Tab::S, tj), yn);
#pragma unroll
    for (int i = 0; i < NC; ++i) y[i] = yn[i];
  }
};

// Commutator-free Lie RK4 on Bloch vectors (two flavours) ---------------------------------------
template <class Phys, class Tab, typename Real, int kPass, int kKind>
struct PassBody<Phys, Tab, Real, true, kPass, kKind> {
  static constexpr int NC = Phys::NC;          // 3: Bloch vectors; 9: Hermitian 3 x 3 matrices
  static constexpr int NG = Phys::NG;          // reals of a generator: 3, or 8 (a 3 x 3 without its trace)
  static constexpr bool kStore = false;
  // Stage states that later passes start from are kept in the output planes, which nobody reads before
  // the final pass: the commutator-free scheme's Y2, from which Y4 follows by one more propagator, and
  // (Richardson) the first half step's Y5 likewise for Y7, then its result y_a, from which slots 9 to 11
  // and the second half step start.  An attempt takes 16 propagators a beam instead of the 26 that start
  // from y every time (a rejected attempt leaves the output planes as scratch), for three more writes of
  // a state that stays in the L2 (GB300: 4M beams mixed, 4 attempts, 3.18 -> 2.23 ms with rotate's
  // division-free form; three flavours, 262,144 beams, 5 attempts, 1.92 -> 1.60 ms).
  static constexpr int kSlot = kKind == kStagePass && !Tab::kEM2 ? kPass + 2 : 0;
  static constexpr bool kWriteOut = kSlot == 2 || (Tab::kRichardson && (kSlot == 5 || kSlot == 8));
  static constexpr bool kReadOut = kSlot == 4 || (Tab::kRichardson && (kSlot == 7 || kSlot >= 9));
  static constexpr bool kReadBoth = kKind == kFinalPass && Tab::kRichardson;
  // rotation of y by d K (the propagator of Eq. U over the path length d for generator K)
  __device__ static inline void rot(Real (&y)[NC], const Real (&K)[NG], Real d) {
    Real Om[NG];
#pragma unroll
    for (int i = 0; i < NG; ++i) Om[i] = d * K[i];
    propagate(Om, y);
  }
  // the fourth stage state of a CF4 step of size hh from its second, y = exp(hh/2 Ka) y0, with generators
  // Ka (its first stage) and Kc (its third): exp(hh (Kc - Ka/2)) y
  __device__ static inline void cf4_stage4(Real (&y)[NC], const Real (&Ka)[NG], const Real (&Kc)[NG], Real hh) {
    Real D[NG];
#pragma unroll
    for (int i = 0; i < NG; ++i) D[i] = Kc[i] - Real(0.5) * Ka[i];
    rot(y, D, hh);
  }
  // the CF4 update of size hh from y with the step's four generators
  __device__ static inline void cf4_final(Real (&y)[NC], const Real (&K1)[NG], const Real (&K2)[NG],
                                          const Real (&K3)[NG], const Real (&K4)[NG], Real hh) {
    Real Om[NG];
#pragma unroll
    for (int i = 0; i < NG; ++i)
      Om[i] = hh * (Real(0.25) * K1[i] + Real(1.0 / 6.0) * (K2[i] + K3[i]) - Real(1.0 / 12.0) * K4[i]);
    propagate(Om, y);
#pragma unroll
    for (int i = 0; i < NG; ++i)
      Om[i] = hh * (Real(-1.0 / 12.0) * K1[i] + Real(1.0 / 6.0) * (K2[i] + K3[i]) + Real(0.25) * K4[i]);
    propagate(Om, y);
  }
  template <class BS>
  __device__ static inline void gen(const BS& bs, const typename Phys::Beam& bm, const TabView<Real, Phys>& tv,
                                    int tj, int s, Real (&K)[NG]) {
    Phys::K(tv.row(s, tj), bm, K);
  }
  // Richardson-controlled CF4 (TabCFR): pass p forms the stage state of slot p + 2, from y or from the
  // state kept in the output planes (kReadOut); the final pass (y the step's state, ya the first half
  // step's result) forms both results, the error ratio and the moments of the kept result.
  template <class BS, class Acc>
  __device__ static inline void richardson(const BS& bs, const typename Phys::Beam& bm,
                                           const TabView<Real, Phys>& tv, int tj, Real (&y)[NC], const Real (&ya)[NC],
                                           Acc& acc, Real& emax, int& bad, bool mixed) {
    const Real h = bs.hB[0], hh = Real(0.5) * h;
    constexpr int I = kKind == kFinalPass ? 0 : kPass + 2;   // slot formed by this pass
    if constexpr (I == 2 || I == 3) {
      // full step: Y2 = exp(h/2 K1) y, Y3 = exp(h/2 K2) y
      Real K[NG];
      gen(bs, bm, tv, tj, I - 1, K);
      rot(y, K, hh);
    } else if constexpr (I == 5 || I == 6) {
      // first half step: slots 5, 6 as 2, 3 with hh and generators K1, K5
      Real K[NG];
      gen(bs, bm, tv, tj, I == 5 ? 1 : 5, K);
      rot(y, K, Real(0.5) * hh);
    } else if constexpr (I == 4 || I == 7) {
      // y holds Y2 (Y5): Y4 = exp(h (K3 - K1/2)) Y2, Y7 = exp(hh (K6 - K1/2)) Y5
      Real K1[NG], K[NG];
      gen(bs, bm, tv, tj, 1, K1);
      gen(bs, bm, tv, tj, I - 1, K);
      cf4_stage4(y, K1, K, I == 4 ? h : hh);
    } else if constexpr (I == 8) {
      // the first half step's result y_a
      Real K1[NG], K5[NG], K6[NG], K7[NG];
      gen(bs, bm, tv, tj, 1, K1);
      gen(bs, bm, tv, tj, 5, K5);
      gen(bs, bm, tv, tj, 6, K6);
      gen(bs, bm, tv, tj, 7, K7);
      cf4_final(y, K1, K5, K6, K7, hh);
    } else if constexpr (I == 9 || I == 10) {
      // second half step from y_a
      Real K[NG];
      gen(bs, bm, tv, tj, I - 1, K);
      rot(y, K, Real(0.5) * hh);
    } else if constexpr (I == 11) {
      Real K8[NG], K10[NG];
      gen(bs, bm, tv, tj, 8, K8);
      gen(bs, bm, tv, tj, 10, K10);
      rot(y, K8, Real(0.5) * hh);
      cf4_stage4(y, K8, K10, hh);
    }
    if constexpr (I >= 2) {
      Phys::accum_row(acc, bm.w, tv.row(I, tj), y);
      return;
    } else {
      // final pass: y_b = the second half step from y_a, y_full = the full step from y
      Real yb[NC], yf[NC];
#pragma unroll
      for (int i = 0; i < NC; ++i) { yb[i] = ya[i]; yf[i] = y[i]; }
      {
        Real K8[NG], K9[NG], K10[NG], K11[NG];
        gen(bs, bm, tv, tj, 8, K8);
        gen(bs, bm, tv, tj, 9, K9);
        gen(bs, bm, tv, tj, 10, K10);
        gen(bs, bm, tv, tj, 11, K11);
        cf4_final(yb, K8, K9, K10, K11, hh);
      }
      {
        Real K1[NG], K2[NG], K3[NG], K4[NG];
        gen(bs, bm, tv, tj, 1, K1);
        gen(bs, bm, tv, tj, 2, K2);
        gen(bs, bm, tv, tj, 3, K3);
        gen(bs, bm, tv, tj, 4, K4);
        cf4_final(yf, K1, K2, K3, K4, h);
      }
      Real e[NC];
#pragma unroll
      for (int i = 0; i < NC; ++i) e[i] = (yb[i] - yf[i]) * Real(1.0 / 15.0);
      if (!(Phys::tnorm2(y) <= rbig<Real>())) bad = 1;        // non-finite input state: fatal
      const bool ynok = Phys::tnorm2(yb) <= rbig<Real>();
      const Real den = bs.atol + bs.rtol * sqrt(fmax(Phys::tnorm2(y), Phys::tnorm2(yb)));
      Real r2 = Phys::tnorm2(e) / (den * den);
      if (!(r2 <= rbig<Real>()) || !ynok) r2 = Real(INFINITY);
      emax = fmax(emax, r2);
      if (mixed && ynok) Phys::purify(yb);
      Phys::accum_row(acc, bm.w, tv.row(11, tj), yb);
#pragma unroll
      for (int i = 0; i < NC; ++i) y[i] = yb[i];
    }
  }
  template <class BS, class Acc>
  __device__ static inline void beam(const BS& bs, const typename Phys::Beam& bm,
                                     const TabView<Real, Phys>& tv, int tj, Real (&y)[NC],
                                     Real (&)[NC], const Real (&yo)[NC],
                                     Acc& acc, Real& emax, int& bad, bool mixed,
                                     Real*, size_t) {
    if (kKind == kInitPass) {
      Phys::accum_row(acc, bm.w, tv.row(1, tj), y);
      return;
    }
    const Real h = bs.hB[0];
    if constexpr (Tab::kRichardson) {
      richardson(bs, bm, tv, tj, y, yo, acc, emax, bad, mixed);
      return;
    }
    if constexpr (Tab::kEM2) {
      // exponential midpoint rule: half step with K1 -> Y_half (moments at r + h/2); final pass:
      // y' = exp(h K2) y, the estimate exp(h K1) y, the error ratio, moments of y' at r + h
      Real K1[NG], Om[NG];
      Phys::K(tv.row(1, tj), bm, K1);
      if (kKind == kStagePass) {
#pragma unroll
        for (int i = 0; i < NG; ++i) Om[i] = Real(0.5) * h * K1[i];
        propagate(Om, y);
        Phys::accum_row(acc, bm.w, tv.row(2, tj), y);
        return;
      }
      Real K2[NG], yn[NC], ye[NC], e[NC];
      Phys::K(tv.row(2, tj), bm, K2);
#pragma unroll
      for (int i = 0; i < NC; ++i) { yn[i] = y[i]; ye[i] = y[i]; }
#pragma unroll
      for (int i = 0; i < NG; ++i) Om[i] = h * K2[i];
      propagate(Om, yn);
#pragma unroll
      for (int i = 0; i < NG; ++i) Om[i] = h * K1[i];
      propagate(Om, ye);
#pragma unroll
      for (int i = 0; i < NC; ++i) e[i] = yn[i] - ye[i];
      if (!(Phys::tnorm2(y) <= rbig<Real>())) bad = 1;       // non-finite input state: fatal
      const bool ynok = Phys::tnorm2(yn) <= rbig<Real>();
      const Real den = bs.atol + bs.rtol * sqrt(fmax(Phys::tnorm2(y), Phys::tnorm2(yn)));
      Real r2 = Phys::tnorm2(e) / (den * den);
      if (!(r2 <= rbig<Real>()) || !ynok) r2 = Real(INFINITY);
      emax = fmax(emax, r2);
      if (mixed && ynok) Phys::purify(yn);
      Phys::accum_row(acc, bm.w, tv.row(3, tj), yn);
#pragma unroll
      for (int i = 0; i < NC; ++i) y[i] = yn[i];
      return;
    }
    Real K1[NG], K2[NG], K3[NG], K4[NG], Om[NG];
    Phys::K(tv.row(1, tj), bm, K1);
    if (kKind == kStagePass && kPass == 0) {
#pragma unroll
      for (int i = 0; i < NG; ++i) Om[i] = Real(0.5) * h * K1[i];
      propagate(Om, y);
      Phys::accum_row(acc, bm.w, tv.row(2, tj), y);
      return;
    }
    Phys::K(tv.row(2, tj), bm, K2);
    if (kKind == kStagePass && kPass == 1) {
#pragma unroll
      for (int i = 0; i < NG; ++i) Om[i] = Real(0.5) * h * K2[i];
      propagate(Om, y);
      Phys::accum_row(acc, bm.w, tv.row(3, tj), y);
      return;
    }
    Phys::K(tv.row(3, tj), bm, K3);
    if (kKind == kStagePass && kPass == 2) {
      cf4_stage4(y, K1, K3, h);                                // y holds Y2
      Phys::accum_row(acc, bm.w, tv.row(4, tj), y);
      return;
    }
    Phys::K(tv.row(4, tj), bm, K4);
#pragma unroll
    for (int i = 0; i < NG; ++i)
      Om[i] = h * (Real(0.25) * K1[i] + Real(1.0 / 6.0) * (K2[i] + K3[i]) - Real(1.0 / 12.0) * K4[i]);
    propagate(Om, y);
#pragma unroll
    for (int i = 0; i < NG; ++i)
      Om[i] = h * (Real(-1.0 / 12.0) * K1[i] + Real(1.0 / 6.0) * (K2[i] + K3[i]) + Real(0.25) * K4[i]);
    propagate(Om, y);
    if (mixed) Phys::purify(y);
    Phys::accum_row(acc, bm.w, tv.row(4, tj), y);
  }
};

// ----------------------------------------------------------------------------------------------
// FP32 two-flavour beams in pairs with packed f32x2 arithmetic (Blackwell fma/mul.rn.f32x2).
// A thread's two beams are consecutive energy bins of one angle bin, so every table value is shared.
// What bounds these passes (GB300, 4M beams, DP45): with the table values and step coefficients stored
// twice, as packed operands, each pass moved about 110 128-byte wavefronts of shared memory a pair of
// warps, and that, not the FMA pipe (45 % busy) or issue (45 %), set the time; scalar rows of h K with
// compile-time coefficients, and moment sums of four operations a contribution instead of eight, took a
// call of 12 steps from 3.19 to 2.70 ms (64 instances, 28M beams, 8 steps: 16.0 to 13.9 ms; 10
// azimuthal bins, 4M beams, 8 steps: 3.07 to 2.51 ms).
using F2 = unsigned long long;
__device__ __forceinline__ F2 pk(float a, float b) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void upk(F2 r, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
  F2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
  F2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ F2 sub2(F2 a, F2 b) {
  F2 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// biased_add on a pair (each half one beam)
__device__ __forceinline__ void biased_add2(F2& hi, F2& lo, F2 w, F2 y) {
  const F2 s = fma2(w, y, hi);
  const F2 z = sub2(hi, s);
  lo = add2(lo, fma2(w, y, z));
  hi = s;
}
// Moment accumulators of a thread's beam pairs: component i is the unevaluated sum hi[i] + lo[i].
template <int NM>
struct PairAcc {
  F2 hi[NM], lo[NM];
};
// A single (unpaired) beam of a pair kernel accumulates into the first half of the pair
// accumulators, so those kernels keep one set of accumulator registers.
template <int NM>
struct PairHalfAcc {
  static constexpr bool kRows = false;
  PairAcc<NM>& a;
  __device__ __forceinline__ void add(int i, float w, float y) { biased_add2(a.hi[i], a.lo[i], pk(w, 0.0f), pk(y, 0.0f)); }
};

template <class P, class Tab, int kPass, int kKind>
struct PairRK {
  static constexpr int NM = P::NM;                 // 6 (bulb) or 12 (extended: + Jc, Js)
  static_assert(!split_final<Tab, float>(), "FP32 passes rebuild the chain in the final pass");
  static constexpr int kChain =
      kKind == kInitPass ? 0 : (kKind == kFinalPass ? Tab::S - (Tab::kAdaptive ? 1 : 0) : kPass + 1);

  // h k = h K x Y of the row's stage.  The row's values are shared by the two beams and loaded once, as
  // scalars (a value stored twice for a packed operand would cost the shared memory's 128 bytes a cycle
  // twice over, which bound these kernels); the components of K that differ between the beams are made by
  // two scalar FMAs straight into the halves of their operand.  Two components of k are kept with their
  // signs reversed, (-k0, k1, -k2): then K enters as -K0, K2 and both signs of K1 only.
  __device__ static inline void deriv(const float* R, float e0, float e1, const F2 (&Y)[3], F2 (&k)[3]) {
    const float4 a = *reinterpret_cast<const float4*>(R);
    const float g = R[P::oG0Y];
    const F2 nK0 = pk(fmaf(e0, a.x, a.y), fmaf(e1, a.x, a.y)), K2 = pk(fmaf(e0, a.z, a.w), fmaf(e1, a.z, a.w));
    const F2 K1 = pk(g, g), nK1 = pk(-g, -g);
    k[0] = fma2(K2, Y[1], mul2(nK1, Y[2]));
    k[1] = fma2(K2, Y[0], mul2(nK0, Y[2]));
    k[2] = fma2(nK0, Y[1], mul2(K1, Y[0]));
  }
  // Y + c k for k as deriv leaves it
  __device__ static inline void axpy(double cd, const F2 (&k)[3], F2 (&Y)[3]) {
    const float c = (float)cd;
    const F2 cp = pk(c, c), cn = pk(-c, -c);
    Y[0] = fma2(cn, k[0], Y[0]);
    Y[1] = fma2(cp, k[1], Y[1]);
    Y[2] = fma2(cn, k[2], Y[2]);
  }
  // moments of the pair's states with the weights of row R: D (w t1), J1 (w) and, extended model,
  // Jc (w (sin th / cos th) cos phi), Js (w (sin th / cos th) sin phi)
  // (summed without loss: see MomAcc<float>)
  __device__ static inline void accum(PairAcc<NM>& acc, float w0, float w1, const float* R, const F2 (&y)[3]) {
    const float t1 = R[P::oT1];
    const F2 w = pk(w0, w1), wt = pk(w0 * t1, w1 * t1);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      biased_add2(acc.hi[i], acc.lo[i], wt, y[i]);
      biased_add2(acc.hi[3 + i], acc.lo[3 + i], w, y[i]);
    }
    if constexpr (NM == 12) {
      const float sc = R[P::oSCC], ss = R[P::oSCS];
      const F2 wc = pk(w0 * sc, w1 * sc), ws = pk(w0 * ss, w1 * ss);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        biased_add2(acc.hi[6 + i], acc.lo[6 + i], wc, y[i]);
        biased_add2(acc.hi[9 + i], acc.lo[9 + i], ws, y[i]);
      }
    }
  }
  // 1/sqrt(n2) of a pair: hardware reciprocal square root refined by one Newton step
  // r <- r (3 - n2 r^2) / 2 (relative error ~1e-7, as a correctly rounded quotient would give)
  __device__ static inline F2 rnorm(F2 n2) {
    float a, b;
    upk(n2, a, b);
    const F2 r = pk(rsqrtf(a), rsqrtf(b));
    const F2 t = mul2(mul2(n2, r), r);                         // n2 r^2
    return mul2(mul2(r, 0xbf000000bf000000ull), fma2(t, 0x3f8000003f800000ull, 0xc0400000c0400000ull));
  }
  __device__ static inline void normalise(F2 (&y)[3]) {
    F2 n2 = mul2(y[0], y[0]);
    n2 = fma2(y[1], y[1], n2);
    n2 = fma2(y[2], y[2], n2);
    const F2 inv = rnorm(n2);
#pragma unroll
    for (int i = 0; i < 3; ++i) y[i] = mul2(y[i], inv);
  }

  // e0, e1, w0, w1: eta omega and weights of the two beams; rows: table rows of their angle bin, stage s
  // at rows + s * rstride; y as in PassBody::beam
  template <class BS>
  __device__ static inline void run(const BS& bs, float e0, float e1, float w0, float w1, const float* rows, int rstride,
                                    F2 (&y)[3], PairAcc<NM>& acc, float& emax, int& bad) {
    F2 k[Tab::S + 1][3];
    // adaptive final pass: y5 and the error accumulate as soon as each stage derivative exists
    // (same order of operations as summing after the chain), so the derivatives die early
    constexpr bool kFinalAdaptive = kKind == kFinalPass && Tab::kAdaptive;
    F2 yn[3] = {y[0], y[1], y[2]};
    F2 e[3] = {0ull, 0ull, 0ull};
#pragma unroll
    for (int l = 1; l <= kChain; ++l) {
      F2 Y[3] = {y[0], y[1], y[2]};
#pragma unroll
      for (int m = 1; m < l; ++m)
        if (Tab::a(l, m) != 0.0) axpy(Tab::a(l, m), k[m], Y);
      deriv(rows + l * rstride, e0, e1, Y, k[l]);
      if (kFinalAdaptive) {
        if (Tab::b(l) != 0.0) axpy(Tab::b(l), k[l], yn);
        if (Tab::e(l) != 0.0) {            // the error's components carry the signs of k
          const F2 he = pk((float)Tab::e(l), (float)Tab::e(l));
#pragma unroll
          for (int i = 0; i < 3; ++i) e[i] = fma2(he, k[l][i], e[i]);
        }
      }
    }
    if (kKind == kInitPass) {
      accum(acc, w0, w1, rows + rstride * 1, y);
      return;
    }
    if (kKind == kStagePass) {
      constexpr int I = kPass + 2;
      F2 Y[3] = {y[0], y[1], y[2]};
#pragma unroll
      for (int m = 1; m < I; ++m)
        if (Tab::a(I, m) != 0.0) axpy(Tab::a(I, m), k[m], Y);
      if (Tab::kAdaptive && I == Tab::S) normalise(Y);
      accum(acc, w0, w1, rows + rstride * I, Y);
      return;
    }
    if (Tab::kAdaptive) {
      // final pass: y5 from the rebuilt chain, k_S = f(y5), the embedded error and the squared
      // error ratio |e|_F^2 / scale^2 (its square root is taken once per block)
      F2 n2y = mul2(y[0], y[0]);
      n2y = fma2(y[1], y[1], n2y);
      n2y = fma2(y[2], y[2], n2y);
      F2 n2n = mul2(yn[0], yn[0]);
      n2n = fma2(yn[1], yn[1], n2n);
      n2n = fma2(yn[2], yn[2], n2n);
      float a0, a1, c0, c1;
      upk(n2y, a0, a1);
      upk(n2n, c0, c1);
      if (!(a0 <= 3.0e38f) || !(a1 <= 3.0e38f)) bad = 1;    // non-finite input state: fatal
      const bool ok0 = c0 <= 3.0e38f, ok1 = c1 <= 3.0e38f;
      if (ok0 && ok1) {
        const F2 inv = rnorm(n2n);
#pragma unroll
        for (int i = 0; i < 3; ++i) yn[i] = mul2(yn[i], inv);
      }
      deriv(rows + Tab::S * rstride, e0, e1, yn, k[Tab::S]);
      if (Tab::e(Tab::S) != 0.0) {
        const F2 he = pk((float)Tab::e(Tab::S), (float)Tab::e(Tab::S));
#pragma unroll
        for (int i = 0; i < 3; ++i) e[i] = fma2(he, k[Tab::S][i], e[i]);
      }
      F2 e2 = mul2(e[0], e[0]);
      e2 = fma2(e[1], e[1], e2);
      e2 = fma2(e[2], e[2], e2);
      F2 m2 = mul2(yn[0], yn[0]);
      m2 = fma2(yn[1], yn[1], m2);
      m2 = fma2(yn[2], yn[2], m2);
      float e20, e21, m20, m21;
      upk(e2, e20, e21);
      upk(m2, m20, m21);
      // |P~|_F = |s| / sqrt(2), |e|_F^2 = |e|^2 / 2
      const float atol = bs.atol, rtol = bs.rtol;
      const float s0 = atol + rtol * sqrtf(0.5f * fmaxf(a0, m20));
      const float s1 = atol + rtol * sqrtf(0.5f * fmaxf(a1, m21));
      float r0 = __fdiv_rn(0.5f * e20, s0 * s0);
      float r1 = __fdiv_rn(0.5f * e21, s1 * s1);
      if (!(r0 <= 3.0e38f) || !ok0) r0 = INFINITY;
      if (!(r1 <= 3.0e38f) || !ok1) r1 = INFINITY;
      emax = fmaxf(emax, fmaxf(r0, r1));
#pragma unroll
      for (int i = 0; i < 3; ++i) y[i] = yn[i];
      return;
    }
    // final pass of a fixed-step tableau
#pragma unroll
    for (int m = 1; m <= kChain; ++m)
      if (Tab::b(m) != 0.0) axpy(Tab::b(m), k[m], yn);
    float a0[3], a1[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) upk(yn[i], a0[i], a1[i]);
    const bool ok0 = 0.5f * (a0[0] * a0[0] + a0[1] * a0[1] + a0[2] * a0[2]) <= 3.0e38f;
    const bool ok1 = 0.5f * (a1[0] * a1[0] + a1[1] * a1[1] + a1[2] * a1[2]) <= 3.0e38f;
    if (ok0 && ok1) normalise(yn);
    accum(acc, w0, w1, rows + rstride * Tab::S, yn);
#pragma unroll
    for (int i = 0; i < 3; ++i) y[i] = yn[i];
  }
};

// Load the beam constants of (species, energy k) and the angle weight du.
template <typename Real>
__device__ __forceinline__ void load_beam(const Real* et, int ne, int sigma, int k, Real du,
                                          typename Phys2<Real>::Beam& bm) {
  if constexpr (sizeof(Real) == 4) {
    // one 128-bit entry a bin: omega, weights of nu and nubar, pad
    const float4 v = *reinterpret_cast<const float4*>(et + 4 * (size_t)k);
    bm.eo = sigma ? -v.x : v.x;
    bm.w = du * (sigma ? v.z : v.y);
  } else {
    const Real om = et[k];
    bm.eo = sigma ? -om : om;
    bm.w = et[(1 + sigma) * ne + k];                // row sums carry du
  }
}
template <typename Real>
__device__ __forceinline__ void load_beam(const Real* et, int ne, int sigma, int k, Real du,
                                          typename Phys3<Real>::Beam& bm) {
  constexpr int kVac = Phys3<Real>::kVac;
#pragma unroll
  for (int i = 0; i < kVac; ++i) {
    const Real v = et[i * ne + k];
    bm.v[i] = sigma ? -v : v;
  }
  const Real g = et[(kVac + sigma) * ne + k];
  bm.w = sizeof(Real) == 4 ? du * g : g;             // FP64 row sums carry du
}

// Checked build: a beam's energy-table entries (all rows of its bin), its row of the shared angle tables and (stored-stage bodies) its
// elements of the stage planes.  Always true without XFLAT_BOUNDS.
template <class Body, int NC, typename Real>
__device__ __forceinline__ bool beam_in_bounds(const KParams& p, const Real* et, int ne, int k, int tj,
                                               int n_jj, const Real* kst_beam) {
#ifdef XFLAT_BOUNDS
  constexpr int kERowMax = (NC == 3 ? Phys2<double>::kERows : Phys3<Real>::kERows) - 1;
  bool ok = index_ok(p, tj >= 0 && tj < n_jj, 12, tj) && index_ok(p, k >= 0 && k < ne, 10, k) &&
            (NC == 3 && sizeof(Real) == 4
                 ? span_ok(p, kSpanEtab, et + 4 * (size_t)k, 16, 10)
                 : span_ok(p, kSpanEtab, et + k, sizeof(Real), 10) &&
                       span_ok(p, kSpanEtab, et + (size_t)kERowMax * ne + k, sizeof(Real), 11));
  if constexpr (Body::kStore)
    ok = ok && span_ok(p, kSpanKst, kst_beam, sizeof(Real), 8) &&
         span_ok(p, kSpanKst, kst_beam + ((size_t)(Body::kYPlanes + 1) * NC - 1) * p.plane_stride,
                 sizeof(Real), 9);
  return ok;
#else
  return true;
#endif
}

// Dynamic shared memory: reduction scratch, the table rows, the angle weights, the angle positions
// (8-byte aligned) and the state rings.
template <typename Real>
__device__ __forceinline__ Real* table_smem(unsigned char* dyn_smem) {
  return reinterpret_cast<Real*>(dyn_smem + 32 * kNMMax * sizeof(double));
}
template <typename Real>
__device__ __forceinline__ double* angle_smem(Real* after_weights) {
  return reinterpret_cast<double*>((reinterpret_cast<uintptr_t>(after_weights) + 7) & ~uintptr_t(7));
}

// Stages whose table rows a pass reads (bit s set: row s needed).
template <class Tab, int kPass, int kKind>
__device__ __forceinline__ unsigned stages_needed() {
  if (kKind == kInitPass) return 1u << 1;
  if (kKind == kFinalPass) return ((1u << (Tab::S + 1)) - 1u) & ~1u;          // 1..S
  return ((1u << (kPass + 3)) - 1u) & ~1u;                                      // 1..kPass+2
}

// FP32 commutator kernels tabulate h K instead of K, so that the tableau's coefficients are compile-time
// constants of their pass bodies (shared memory's bandwidth bounds them, see PairRK::deriv).
template <typename Real, bool kCF>
__host__ __device__ constexpr bool scaled_rows() { return sizeof(Real) == 4 && !kCF; }

// Set-up of a piece for a pass: flags, step size, coefficients, stage constants and the table rows.
// newest: the stage whose moments the previous pass reduced (0: none of this step); every block derives
// its constants mu m (and lambda) from the accumulators itself (integer sums: the same bits everywhere),
// so that barrier needs no serial section, and the block holding the instance's first beams records
// them for later passes and the host.  need: stages whose rows the pass reads.  single: the block's only
// piece, whose set-up stays in shared memory for the whole step: pass 0 fills the geometry of every
// stage's rows, and after it (incremental) only the newest stage's couplings are still to come.
// One copy of this code serves every pass of a kernel (instruction cache).
template <class Phys, class Tab, typename Real, bool kCF>
__device__ __noinline__ void setup_piece(const KParams& p, BlockShared<Real, Phys>& bs, unsigned char* dyn_smem, int pi,
                                         int newest, unsigned need, bool incremental, bool single) {
  constexpr int kTS = Tab::S + 1;                                    // table stage slots 0..S
  Real* tab = table_smem<Real>(dyn_smem);                            // [kTS][max_jj][KT]
  Real* dut = tab + (size_t)kTS * p.max_jj * Phys::KT;               // [max_jj]
  double* ut = angle_smem(dut + p.max_jj);                           // [max_jj]
  const Piece pc = p.pieces[pi];
  const InstConst& ic = p.ic[pc.inst];
  const InstDyn* d = p.dyn + pc.inst;
  const int n_jj = pc.n_jj;
  // constant c of the newest stage
  auto newest_constant = [&](int c) {
    const unsigned long long* accs = p.acc + (size_t)pc.inst * acc_words_per_inst(sizeof(Real)) + (size_t)newest * acc_words_per_slot(sizeof(Real));
    InstDyn* dw = p.dyn + pc.inst;
    double v = 0.0;
    if (c < Phys::NM) {
      const double m = acc_component<Real>(accs, c, ic.acc_unit);
      v = ldcg(&d->mus[newest]) * m;
      if (pc.start == ic.rec_start) dw->mom[newest][c] = m;
    } else if (c == Phys::NM) {
      v = ldcg(&d->lams[newest]);
    }
    if (pc.start == ic.rec_start && c <= Phys::NM) dw->sc[newest][c] = v;
    return v;
  };
  __syncthreads();
  if constexpr (sizeof(Real) == 8) {
    if (threadIdx.x == 0) bs.emax_f = 0;
  }
  if (incremental) {
    if (threadIdx.x < Phys::NSC) bs.scr[newest][threadIdx.x] = (Real)newest_constant(threadIdx.x);
    __syncthreads();
    for (int tj = threadIdx.x; tj < n_jj; tj += blockDim.x)
      Phys::fill_cpl(tab + ((size_t)newest * n_jj + tj) * Phys::KT, bs.scr[newest]);
    __syncthreads();
    return;
  }
  // one parallel load phase (every load issued before any of them is used, so the phase costs one L2
  // round trip)
  if (threadIdx.x == 0) {
    const int dn = ldcg(&d->done), st = ldcg(&d->status), par = ldcg(&d->parity);
    bs.active = (dn == 0 && st == 0) ? 1 : 0;
    bs.parity = par;
  }
  const double h = Tab::kAdaptive ? ldcg(&d->h) : ldcg(&d->h_fixed);
  for (int t = threadIdx.x; t < kTS * Phys::NSC; t += blockDim.x) {
    const int s = t / Phys::NSC, c = t % Phys::NSC;
    double v = 0.0;
    if (s == newest) v = newest_constant(c);
    else if ((need >> s) & 1u) v = ldcg(&d->sc[s][c]);
    bs.scr[s][c] = (Real)v;
  }
  if (threadIdx.x < kMaxStages) {
    bs.xs[threadIdx.x] = ldcg(&d->xs[threadIdx.x]);
    bs.t1max[threadIdx.x] = 0;
  }
  if constexpr (kCF) {
    if (threadIdx.x == 0) bs.hB[0] = (Real)h;
  } else {
    // the non-zero coefficients of the tableau, one a thread: (i, j) of a, then b_j, then e_j
    constexpr int kA = Tab::S + 1, kCoef = kA * kA + 2 * kA;
    for (int t = threadIdx.x; t < kCoef; t += blockDim.x) {
      double v = 0.0;
#pragma unroll
      for (int i = 1; i < kA; ++i)
#pragma unroll
        for (int j = 1; j < kA; ++j)
          if (Tab::a(i, j) != 0.0) v = t == i * kA + j ? Tab::a(i, j) : v;
#pragma unroll
      for (int j = 1; j < kA; ++j) {
        if (Tab::b(j) != 0.0) v = t == kA * kA + j ? Tab::b(j) : v;
        if (Tab::e(j) != 0.0) v = t == kA * kA + kA + j ? Tab::e(j) : v;
      }
      const Real hv = (Real)(scaled_rows<Real, kCF>() ? v : h * v);
      if (t < kA * kA) bs.hA[t / kA][t % kA] = hv;
      else if (t < kA * kA + kA) bs.hB[t - kA * kA] = hv;
      else bs.hE[t - kA * kA - kA] = hv;
    }
  }
  // launch-invariant part (tolerances, angle tables): a single-piece block loads it once per launch
  if (!(single && bs.keep)) {
    if (threadIdx.x == 0) {
      bs.rtol = (Real)ic.rtol;
      bs.atol = (Real)ic.atol;
      if constexpr (sizeof(Real) == 8) {
        const double inv = fmin(1.0 / (ic.rtol + ic.atol), 1.0e30);      // keeps FP32 squares in range
        bs.inv_tol = (float)inv;
        bs.rtol_f = (float)(ic.rtol * inv);
        bs.atol_f = (float)(ic.atol * inv);
      }
    }
    for (int t = threadIdx.x; t < n_jj; t += blockDim.x) {
      const int jj = pc.jj_lo + t;
      const int j = jj >= (int)ic.n_angle ? jj - (int)ic.n_angle : jj;
      if (!(XFLAT_INDEX_OK(p, j >= 0 && j < (int)ic.n_angle, 15, jj) &&
            XFLAT_SPAN_OK(p, kSpanDu, p.du_tab + ic.a_off + j, sizeof(double), 16) &&
            XFLAT_SPAN_OK(p, kSpanU, p.u_tab + ic.a_off + j, sizeof(double), 16))) {
        dut[t] = Real(0);
        ut[t] = 0.0;
        continue;
      }
      dut[t] = (Real)p.du_tab[ic.a_off + j];
      ut[t] = p.u_tab[ic.a_off + j];
    }
  }
  __syncthreads();
  if (single && threadIdx.x == 0) bs.keep = 1;       // read after later barriers only
  if (!bs.active) return;
  typename Phys::Consts C;
  if constexpr (Phys::NC == 3) {
    C.B[0] = ic.B[0]; C.B[1] = ic.B[1]; C.B[2] = ic.B[2];
    if constexpr (Phys::NM == 12) C.n_phi = (int)ic.n_phi;
    else C.geom = ic.geom;
  } else {
    C.geom = ic.geom;
  }
  const unsigned geo = single && !p.shard_mode ? ((1u << kTS) - 1u) & ~1u : need;
  for (int t = threadIdx.x; t < kTS * n_jj; t += blockDim.x) {
    const int s = t / n_jj, tj = t % n_jj;
    if (!((geo >> s) & 1u)) continue;
    Real* row = tab + ((size_t)s * n_jj + tj) * Phys::KT;
    const int jj = (int)pc.jj_lo + tj;
    const int a = jj >= (int)ic.n_angle ? jj - (int)ic.n_angle : jj;     // angle bin of its species
    Phys::fill_geo(row, ut[tj], bs.xs[s], C, a, scaled_rows<Real, kCF>() ? (Real)h : Real(1));
    if constexpr (sizeof(Real) == 4) atomicMax(&bs.t1max[s], __float_as_int(Phys::t1(row)));   // t1 >= 0
    if ((need >> s) & 1u) Phys::fill_cpl(row, bs.scr[s]);
  }
  __syncthreads();
}

// One pass over all pieces of this block.
template <class Phys, class Tab, typename Real, bool kCF, int kPass, int kKind>
__device__ void run_pass(const KParams& p, BlockShared<Real, Phys>& bs, unsigned char* dyn_smem) {
  constexpr int NC = Phys::NC, NM = Phys::NM, VN = vec_beams<Phys, Real>();
  using Body = PassBody<Phys, Tab, Real, kCF, kPass, kKind>;
  double* red = reinterpret_cast<double*>(dyn_smem);                 // 32 * kNMMax doubles
  constexpr int kTS = Tab::S + 1;                                    // table stage slots 0..S
  Real* tab = table_smem<Real>(dyn_smem);                            // [kTS][max_jj][KT]
  Real* dut = tab + (size_t)kTS * p.max_jj * Phys::KT;               // [max_jj]
  float* ring = reinterpret_cast<float*>(                            // [slots][NC][threads][2], 16-byte aligned
      (reinterpret_cast<uintptr_t>(angle_smem(dut + p.max_jj) + p.max_jj) + 15) & ~uintptr_t(15));
  const bool mixed = sizeof(Real) == 4;
  const int slot = kKind == kInitPass ? 1 : (kKind == kStagePass ? kPass + 2 : 0);
  // Clear accumulator slots nobody reads any more (block 0, while the other blocks already work).
  // Stage s (2 <= s < kPasses) is reduced in pass s - 2 and read by every block in the set-up of
  // pass s - 1, so it is cleared at the start of pass s; pass 0 clears the final pass's slot 0 and
  // the moment launch's slot 1, both read by serial updates that finish before their barrier
  // opens.  Stages with no pass of their own index (kPasses <= s <= S: stage S of RK4 / DP45,
  // stages 2 and 3 of the exponential midpoint rule) are cleared by the final pass's serial section
  // (clear_late_slots) while every other block waits at the final barrier.  Nothing accumulates
  // into a cleared slot until at least one barrier later, and block 0's stores are fenced at its
  // next arrival.
  if (kKind != kInitPass && blockIdx.x == 0) {
    constexpr int kWords = acc_words_per_slot(sizeof(Real));
    constexpr int kSlots = kPass == 0 ? 2 : (kPass >= 2 ? 1 : 0);
    for (int t = threadIdx.x; t < p.n_inst * kSlots * kWords; t += blockDim.x) {
      const int inst = t / (kSlots * kWords), rem = t % (kSlots * kWords), q = rem / kWords;
      const int zslot = kPass == 0 ? q : kPass;
      p.acc[(size_t)inst * acc_words_per_inst(sizeof(Real)) + (size_t)zslot * kWords + rem % kWords] = 0ull;
    }
  }
  const unsigned need = stages_needed<Tab, kPass, kKind>();
  // the stage whose moments the previous pass reduced (0: none of this step, its constants come
  // from the serial update of the previous step or of the moment launch)
  constexpr int kNewest = (kKind != kInitPass && kPass >= 1) ? kPass + 1 : 0;
  const bool dyn = p.dyn_sched != 0;
  const int b0 = dyn ? 0 : p.blk_piece[blockIdx.x], b1 = dyn ? 0 : p.blk_piece[blockIdx.x + 1];
  // a block with a single piece keeps its set-up in shared memory for the whole step (setup_piece)
  const bool single = !dyn && b1 - b0 == 1;
  const bool incremental = single && kNewest >= 1 && !p.shard_mode;
  for (int it = 0;; ++it) {
    int pi = b0 + it;
    if (dyn) {
      __syncthreads();                           // next_piece of the previous piece has been read
      if (threadIdx.x == 0) bs.next_piece = (int)atomicAdd(&p.bar->chunk[(bs.gen_seen >> 1) & 1u], 1u);
      __syncthreads();
      pi = bs.next_piece;
      if (pi >= p.n_pieces) break;
    } else if (pi >= b1) {
      break;
    }
    if (!XFLAT_INDEX_OK(p, pi >= 0 && pi < p.n_pieces, 13, pi)) break;
    const Piece pc = p.pieces[pi];
    if (!XFLAT_INDEX_OK(p, pc.inst >= 0 && pc.inst < p.n_inst && (int)pc.n_jj <= p.max_jj &&
                               (uint64_t)pc.start + pc.len <= p.ic[pc.inst].n_beams, 14, pi))
      continue;
    const InstConst& ic = p.ic[pc.inst];
    setup_piece<Phys, Tab, Real, kCF>(p, bs, dyn_smem, pi, kNewest, need, incremental, single);
    if (!bs.active) continue;
    const int n_jj = pc.n_jj;
    const TabView<Real, Phys> tv{tab, n_jj};
    const Real* et = reinterpret_cast<const Real*>(p.etab) + ic.e_off;
    const Real* yin = reinterpret_cast<const Real*>(bs.parity ? p.planeB : p.planeA) + ic.beam_off;
    Real* yout = reinterpret_cast<Real*>(bs.parity ? p.planeA : p.planeB) + ic.beam_off;
    // split final pass (see split_final): the pass forming Y_S stores y5 (into the output planes),
    // and the error partial; the final pass reads those instead of the chain
    constexpr bool kSplitStore = split_final<Tab, Real>() && kKind == kStagePass && kPass + 2 == Tab::S;
    constexpr bool kSplitLoad = split_final<Tab, Real>() && kKind == kFinalPass;
    Real* escr = reinterpret_cast<Real*>(p.escr) + ic.beam_off;
    Real* kst = Body::kStore ? reinterpret_cast<Real*>(p.kst) + ic.beam_off : nullptr;
    const Real* ysrc = kSplitLoad || Body::kReadOut ? yout : yin;
    const int ne = (int)ic.n_energy, na = (int)ic.n_angle;
    // biases of the mixed sums: a thread adds at most 2 (its + 1) contributions of |w| <= wmax (times the
    // geometry factor), |Y| <= 2, to an accumulator
    auto biases = [&](float (&bias)[NM / NC]) {
      if constexpr (sizeof(Real) == 4) {
        constexpr int kRow = kKind == kInitPass ? 1 : (kKind == kStagePass ? kPass + 2 : Tab::S);
        const float t1m = __int_as_float(bs.t1max[kRow]);
        const float P = 4.0f * (float)(pc.len / (VN * blockDim.x) + 2u) * ic.wmax;
        bias[0] = sum_bias(P * t1m);
        bias[1] = sum_bias(P);
        if constexpr (NM / NC == 4) bias[2] = bias[3] = sum_bias(P * sqrtf(t1m * (t1m + 2.0f)));   // tan th
      }
    };
    float bias[NM / NC];
    biases(bias);
    MomAcc<Real, NM> acc;
    acc.start(bias, NC);
    Real emax = 0;
    int bad = 0;
    // FP32 two-flavour RK passes run beam pairs on packed f32x2 arithmetic (PairRK)
    constexpr bool kPair = Phys::kPairable && !kCF;
    PairAcc<NM> acc2;
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      if constexpr (kPair) acc2.hi[i] = pk(bias[i / NC], bias[i / NC]);
      acc2.lo[i] = 0ull;
    }
    float emax2 = 0.0f;
    // Which beams a thread takes: FP32 passes stride the block over the piece; FP64 passes give each
    // warp a contiguous run of it, so that a thread stays in one angle row for many beams (row sums).
    constexpr bool kRows = MomAcc<Real, NM>::kRows;
    constexpr bool kMoments = kKind != kFinalPass || Tab::kFinalMoments;
    constexpr int kMomRow = kKind == kInitPass ? 1 : (kKind == kStagePass ? kPass + 2 : Tab::S);
    const uint32_t run = kRows ? (pc.len + VN * blockDim.x - 1) / (VN * blockDim.x) * (32u * VN) : 0u;
    const uint32_t first = pc.start + (kRows ? (threadIdx.x >> 5) * run + VN * (threadIdx.x & 31) : VN * threadIdx.x);
    const uint32_t end = kRows ? min(pc.start + pc.len, pc.start + ((threadIdx.x >> 5) + 1) * run) : pc.start + pc.len;
    const uint32_t vstep = kRows ? 32u * VN : VN * blockDim.x;
    int row_cur = -1;                                  // row sums: the row being summed
    // FP32 two-flavour bulb passes: the state comes through the thread's ring, kStateRingDepth vectors
    // ahead (see state_ring).  Other two-flavour passes: the next vector's state is loaded into
    // registers while this one is processed.  Either way the L2/HBM latency of the stream overlaps
    // the arithmetic.
    constexpr bool kRingLoad = state_ring<Phys, Real>();
    constexpr bool kPrefetch = NC == 3 && !kRingLoad;
    Real nxt[NC][VN];
    if (kPrefetch && first < end) {
#pragma unroll
      for (int c = 0; c < NC; ++c) vload_at(p, kSpanPlanes, ysrc + (size_t)c * p.plane_stride + first, nxt[c], 1);
    }
    constexpr int ring_d = kStateRingDepth;
    constexpr uint32_t ring_slots = (uint32_t)ring_d + 1u;
    uint32_t q_fill = 0, q_read = 0;
    // start the copies of the vector at beam l (if it is in the piece) into the next slot; one
    // commit group per vector, empty past the end, so the group count stays in step
    auto ring_fill = [&](uint32_t l) {
      if (l < end) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const Real* src = ysrc + (size_t)c * p.plane_stride + l;
          if (XFLAT_SPAN_OK(p, kSpanPlanes, src, 2 * sizeof(Real), 1))
            cp_async8(ring + (((size_t)q_fill * NC + c) * blockDim.x + threadIdx.x) * 2, src);
        }
      }
      cp_async_commit();
      q_fill = q_fill + 1u == ring_slots ? 0u : q_fill + 1u;
    };
    if constexpr (kRingLoad) {
      for (int j = 0; j < ring_d; ++j) ring_fill(first + (uint32_t)j * vstep);
    }
    for (uint32_t l0 = first; l0 < end; l0 += vstep) {
      Real ys[NC][VN];
      if constexpr (kRingLoad) {
        // the slot filled now is the one read in the previous iteration (kStateRingDepth + 1 slots)
        ring_fill(l0 + (uint32_t)ring_d * vstep);
        cp_async_wait_pending<ring_d>();
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const float2 t = *reinterpret_cast<const float2*>(ring + (((size_t)q_read * NC + c) * blockDim.x + threadIdx.x) * 2);
          ys[c][0] = t.x;
          ys[c][1] = t.y;
        }
        q_read = q_read + 1u == ring_slots ? 0u : q_read + 1u;
      } else if constexpr (kPrefetch) {
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
          for (int v = 0; v < VN; ++v) ys[c][v] = nxt[c][v];
        if (l0 + vstep < end) {
#pragma unroll
          for (int c = 0; c < NC; ++c) vload_at(p, kSpanPlanes, ysrc + (size_t)c * p.plane_stride + l0 + vstep, nxt[c], 2);
        }
      } else {
#pragma unroll
        for (int c = 0; c < NC; ++c) vload_at(p, kSpanPlanes, ysrc + (size_t)c * p.plane_stride + l0, ys[c], 3);
      }
      Real ep[NC][VN], yo[NC][VN];
      if constexpr (kSplitLoad) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          vload_at(p, kSpanEscr, escr + (size_t)c * p.plane_stride + l0, ep[c], 4);
          vload_at(p, kSpanPlanes, yin + (size_t)c * p.plane_stride + l0, yo[c], 17);
        }
      }
      if constexpr (Body::kReadBoth) {
#pragma unroll
        for (int c = 0; c < NC; ++c) vload_at(p, kSpanPlanes, yout + (size_t)c * p.plane_stride + l0, yo[c], 17);
      }
      int jj = (int)fast_div(l0, ic.div_magic);
      int k = (int)l0 - jj * ne;
      bool paired = false;
      if constexpr (kPair) {
        // both beams in the same angle bin (all but the rare pair that straddles two bins)
        if (l0 + 1 < end && k + 1 < ne &&
            beam_in_bounds<Body, NC, Real>(p, et, ne, k, jj - (int)pc.jj_lo, n_jj, nullptr) &&
            beam_in_bounds<Body, NC, Real>(p, et, ne, k + 1, jj - (int)pc.jj_lo, n_jj, nullptr)) {
          paired = true;
          const int sigma = jj >= na ? 1 : 0;
          const int tj = jj - (int)pc.jj_lo;
          typename Phys2<float>::Beam b0, b1;
          load_beam<float>(et, ne, sigma, k, dut[tj], b0);
          load_beam<float>(et, ne, sigma, k + 1, dut[tj], b1);
          F2 y2[3];
#pragma unroll
          for (int c = 0; c < 3; ++c) y2[c] = pk(ys[c][0], ys[c][1]);
          PairRK<Phys, Tab, kPass, kKind>::run(bs, b0.eo, b1.eo, b0.w, b1.w, tab + (size_t)tj * Phys::KT, n_jj * Phys::KT, y2,
                                               acc2, emax2, bad);
#pragma unroll
          for (int c = 0; c < 3; ++c) upk(y2[c], ys[c][0], ys[c][1]);
        }
      }
      if (!paired) {
#pragma unroll
        for (int v = 0; v < VN; ++v) {
          if (l0 + v < end &&
              beam_in_bounds<Body, NC, Real>(p, et, ne, k, jj - (int)pc.jj_lo, n_jj,
                                             Body::kStore ? kst + l0 + v : nullptr)) {
            const int sigma = jj >= na ? 1 : 0;
            const int tj = jj - (int)pc.jj_lo;
            typename Phys::Beam bm;
            load_beam<Real>(et, ne, sigma, k, dut[tj], bm);
            if constexpr (kRows && kMoments) {
              if (tj != row_cur) {
                if (row_cur >= 0) Phys::flush_row(acc, dut[row_cur], tv.row(kMomRow, row_cur));
                row_cur = tj;
              }
            }
            Real y[NC], ev[NC], ov[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) y[c] = ys[c][v];
            if constexpr (kSplitLoad || Body::kReadBoth) {
#pragma unroll
              for (int c = 0; c < NC; ++c) { ev[c] = ep[c][v]; ov[c] = yo[c][v]; }
            }
            if constexpr (kPair) {
              PairHalfAcc<NM> hacc{acc2};
              Body::beam(bs, bm, tv, tj, y, ev, ov, hacc, emax, bad, mixed, nullptr, p.plane_stride);
            } else {
              Body::beam(bs, bm, tv, tj, y, ev, ov, acc, emax, bad, mixed, Body::kStore ? kst + l0 + v : nullptr,
                         p.plane_stride);
            }
#pragma unroll
            for (int c = 0; c < NC; ++c) ys[c][v] = y[c];
            if constexpr (kSplitStore) {
#pragma unroll
              for (int c = 0; c < NC; ++c) ep[c][v] = ev[c];
            }
          }
          if (++k == ne) { k = 0; ++jj; }
        }
      }
      if constexpr ((kKind == kFinalPass && !kSplitLoad) || Body::kWriteOut) {
#pragma unroll
        for (int c = 0; c < NC; ++c) vstore_at(p, kSpanPlanes, yout + (size_t)c * p.plane_stride + l0, ys[c], 5);
      }
      if constexpr (kSplitStore) {
#pragma unroll
        for (int c = 0; c < NC; ++c) vstore_at(p, kSpanPlanes, yout + (size_t)c * p.plane_stride + l0, ys[c], 6);
#pragma unroll
        for (int c = 0; c < NC; ++c) vstore_at(p, kSpanEscr, escr + (size_t)c * p.plane_stride + l0, ep[c], 7);
      }
    }
    if constexpr (kRingLoad) cp_async_wait_pending<0>();  // nothing in flight into the ring after the piece
    if constexpr (kPair) emax = fmax(emax, (Real)emax2);
    if constexpr (kRows && kMoments) {
      if (row_cur >= 0) Phys::flush_row(acc, dut[row_cur], tv.row(kMomRow, row_cur));
    }
    // reduce this piece into the instance accumulators: the error maximum (final pass of an
    // adaptive tableau) and the moments (every pass but a final one without moments); a
    // non-finite moment rejects an adaptive trial step and is fatal for a fixed step and for the moments of
    // the current state (init pass)
    constexpr bool kErrMax = kKind == kFinalPass && Tab::kAdaptive;
    constexpr bool kRejectOverflow = Tab::kAdaptive && kKind != kInitPass;
    unsigned long long* acc_slot =
        p.acc + (size_t)pc.inst * acc_words_per_inst(sizeof(Real)) + (size_t)slot * acc_words_per_slot(sizeof(Real));
    const int copy = blockIdx.x % kAccCopies;
    if constexpr (sizeof(Real) == 4) {
      // mixed precision: each thread's (hi, lo) partial sums go to integers of the instance's
      // acc_unit, and every further sum is an integer addition (exact, order-free).  A thread or block
      // partial of 2^52 units or more (only a runaway or non-finite state reaches it) rejects an
      // adaptive trial step and is fatal for a fixed step.  The error maximum is a max (exact); the
      // square root of the block's maximum is taken in double.
      if constexpr (kErrMax)
        reduce_error((emax <= 3.0e38f) ? (float)emax : INFINITY, bad, reinterpret_cast<float*>(red), &p.errmax[pc.inst],
                     &p.nonfinite[pc.inst]);
      if constexpr (kMoments) {
        if constexpr (kErrMax) __syncthreads();              // the scratch is reused
        int ovf = 0;
        long long v[NM];
        float bias[NM / NC];                                 // again, not held over the loop
        biases(bias);
#pragma unroll
        for (int i = 0; i < NM; ++i) {
          if constexpr (kPair) {
            float h[2], l0, l1;
            upk(acc2.hi[i], h[0], h[1]);
            upk(acc2.lo[i], l0, l1);
            v[i] = biased_fix<2>(h, __fadd_rn(l0, l1), bias[i / NC], ovf);
          } else {
            const float h[1] = {acc.hi[i]};
            v[i] = biased_fix<1>(h, acc.lo[i], bias[i / NC], ovf);
          }
        }
        reduce_moments<NM, long long>(v, ovf, reinterpret_cast<long long*>(red), acc_slot + (size_t)copy * kNMMax * 2, 0, &p.errmax[pc.inst],
                                      &p.nonfinite[pc.inst], kRejectOverflow);
      }
    } else {
      if constexpr (kErrMax) {
        // the maximum over the bits of non-negative doubles (integer pipe)
        long long em = __double_as_longlong((emax <= rbig<Real>()) ? (double)emax : (double)INFINITY);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) em = max(em, __shfl_xor_sync(0xffffffffu, em, o));
        long long* redl = reinterpret_cast<long long*>(red);
        if ((threadIdx.x & 31) == 0) redl[threadIdx.x >> 5] = em;
        const int any_bad = __syncthreads_or(bad);
        if (threadIdx.x == 0) {
          for (int w = 1; w < (int)(blockDim.x >> 5); ++w) em = max(em, redl[w]);
          if (any_bad) atomicExch(&p.nonfinite[pc.inst], 1);
          // the beams gave squared error ratios
          atomicMax(&p.errmax[pc.inst], (unsigned long long)__double_as_longlong(sqrt(__longlong_as_double(em))));
        }
      }
      if constexpr (kMoments) {
        if constexpr (kErrMax) __syncthreads();              // the scratch is reused
        double v[NM];                                        // a copy: the accumulators stay in registers
#pragma unroll
        for (int i = 0; i < NM; ++i) v[i] = acc.v[i];
        reduce_moments_shared<NM>(v, red, acc_slot, copy, &p.errmax[pc.inst], &p.nonfinite[pc.inst], kRejectOverflow);
      }
    }
  }
}

template <class Phys, class Tab, typename Real, bool kCF, int kPass>
__device__ __forceinline__ bool pass_and_sync(const KParams& p, BlockShared<Real, Phys>& bs,
                                              unsigned char* dyn_smem) {
  constexpr bool kFinal = kPass == Tab::kPasses - 1;
  constexpr int kKind = kFinal ? kFinalPass : kStagePass;
  unsigned long long t0 = 0, t1 = 0;
  if (p.trace && threadIdx.x == 0) t0 = globaltimer_ns();
  run_pass<Phys, Tab, Real, kCF, kPass, kKind>(p, bs, dyn_smem);
  if (p.trace && threadIdx.x == 0) t1 = globaltimer_ns();
  if constexpr (!kFinal) {
    // stage pass: every block derives the new stage's constants from the accumulators in its next
    // set-up (run_pass), so the barrier has no serial section (with dynamic scheduling its last block
    // resets the piece counter, below)
    if (!p.dyn_sched) {
      if (!pass_barrier(p.bar, gridDim.x, bs.expected, p.timeout_ns, p.status, &bs.flag, &bs.pass_next)) return false;
      if (p.trace && threadIdx.x == 0) {
        const int idx = bs.pass_idx++;
        if (idx < p.trace_passes) {
          unsigned long long* t = p.trace + ((size_t)idx * gridDim.x + blockIdx.x) * 4;
          t[0] = t0;
          t[1] = t1;
          t[2] = globaltimer_ns();
          t[3] = 0ull;
        }
      }
      return true;
    }
  }
  const int res = barrier_arrive(p.bar, gridDim.x, p.timeout_ns, p.status, &bs.flag, &bs.gen_seen);
  if ((res & 0xf) == kBarAbort) return false;
  if (p.trace && threadIdx.x == 0) {
    const int idx = bs.pass_idx++;
    if (idx < p.trace_passes) {
      unsigned long long* t = p.trace + ((size_t)idx * gridDim.x + blockIdx.x) * 4;
      t[0] = t0;
      t[1] = t1;
      t[2] = globaltimer_ns();
      t[3] = (res & 0xf) == kBarLast ? 1ull : 0ull;
    }
  }
  if ((res & 0xf) == kBarLast && p.dyn_sched && threadIdx.x == 0)
    p.bar->chunk[((bs.gen_seen >> 1) + 1u) & 1u] = 0u;   // the next pass's piece counter (released below)
  if ((res & 0xf) == kBarLast && !kFinal) {
    // the barrier opens at once (a non-finite partial is reported by the final pass's serial update)
    if (threadIdx.x == 0) bs.flag = 0;
    barrier_release(p.bar, 0, &bs.gen_seen);
    if (p.trace && threadIdx.x == 0 && bs.pass_idx - 1 < p.trace_passes)
      p.trace[((size_t)(bs.pass_idx - 1) * gridDim.x + blockIdx.x) * 4 + 3] = globaltimer_ns() | (1ull << 63);
  } else if ((res & 0xf) == kBarLast) {
    const int mine = serial_update<Phys, Tab, Real>(p, 0, true, false);
    const int all = __syncthreads_and(mine);
    clear_late_slots<Tab, Real>(p);
    serial_geometry<Tab>(p);
    if (threadIdx.x == 0) {
      *p.all_done = all;
      bs.flag = all ? 0x10 : 0;
    }
    unsigned long long ts = 0;
    if (p.trace && threadIdx.x == 0) ts = globaltimer_ns();
    barrier_release(p.bar, all, &bs.gen_seen);
    if (p.trace && threadIdx.x == 0 && bs.pass_idx - 1 < p.trace_passes) {
      // last block: stamp 3 = serial work done (bits 0..62), stamp 2 stays its arrival
      p.trace[((size_t)(bs.pass_idx - 1) * gridDim.x + blockIdx.x) * 4 + 3] = ts | (1ull << 63);
    }
  }
  return true;
}

template <class Phys, class Tab, typename Real, bool kCF, int kPass>
__device__ __forceinline__ bool all_passes(const KParams& p, BlockShared<Real, Phys>& bs,
                                           unsigned char* dyn_smem) {
  if constexpr (kPass < Tab::kPasses) {
    if (!pass_and_sync<Phys, Tab, Real, kCF, kPass>(p, bs, dyn_smem)) return false;
    return all_passes<Phys, Tab, Real, kCF, kPass + 1>(p, bs, dyn_smem);
  } else {
    return true;
  }
}

// Beam-shard mode: the beam work of one pass chosen at run time (no barrier, no serial section).
template <class Phys, class Tab, typename Real, bool kCF, int kPass>
__device__ __forceinline__ void one_pass(const KParams& p, BlockShared<Real, Phys>& bs, unsigned char* dyn_smem,
                                         int which) {
  if constexpr (kPass < Tab::kPasses) {
    if (which == kPass) {
      constexpr int kKind = kPass == Tab::kPasses - 1 ? kFinalPass : kStagePass;
      run_pass<Phys, Tab, Real, kCF, kPass, kKind>(p, bs, dyn_smem);
      return;
    }
    one_pass<Phys, Tab, Real, kCF, kPass + 1>(p, bs, dyn_smem, which);
  }
}

// kThreads x kMinB: the block size and resident blocks per SM the register budget is sized for.
// FP64 work runs on GB300's narrow FP64 pipe (about 1/68 of the FP32 rate), which one 256-thread
// block per SM already keeps busy, so FP64 kernels are built for that (whole register file, no spills), the
// two-flavour RK4 and DP45 also for two blocks (kernels_2f.cu).  The FP32 two-flavour kernels are
// latency-bound; they are built for 768 resident threads per SM (256 x 3) and for 512 (256 x 2, or one 512-thread block: the SM's two halves of the work
// then finish together instead of the older block's warps finishing first), and the launch shape
// is chosen by measurement (the autotuner in paper_1912_10596_gb300/autotune.py).
template <class Phys, class Tab, typename Real, bool kCF, int kMinB, int kThreads = 256>
__global__ void __launch_bounds__(kThreads, kMinB) step_kernel(const __grid_constant__ KParams p) {
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  __shared__ BlockShared<Real, Phys> bs;
  if (threadIdx.x == 0) {
    bs.pass_idx = 0;
    bs.keep = 0;
    bs.gen_seen = ld_acquire(&p.bar->gen);        // later barriers track the generation locally
    bs.expected = gridDim.x + p.bar->extra;
    bs.pass_next = pass_barrier_base(p.bar, gridDim.x);
  }
  if (p.shard_mode == kShardPass) {
    if (p.shard_pass < 0) run_pass<Phys, Tab, Real, kCF, 0, kInitPass>(p, bs, dyn_smem);
    else one_pass<Phys, Tab, Real, kCF, 0>(p, bs, dyn_smem, p.shard_pass);
    return;
  }
  if (p.shard_mode == kShardSerialInit || p.shard_mode == kShardSerialFinal) {
    // one block; the host has replaced the pass's partial sums by the totals over all shards
    if (blockIdx.x != 0) return;
    const bool init = p.shard_mode == kShardSerialInit;
    const int mine = serial_update<Phys, Tab, Real>(p, init ? 1 : 0, !init, init);
    const int all = __syncthreads_and(mine);
    if (!init) clear_late_slots<Tab, Real>(p);
    serial_geometry<Tab>(p);
    if (threadIdx.x == 0) *p.all_done = all;
    return;
  }
  if (p.init_only) {
    run_pass<Phys, Tab, Real, kCF, 0, kInitPass>(p, bs, dyn_smem);
    const int res = barrier_arrive(p.bar, gridDim.x, p.timeout_ns, p.status, &bs.flag, &bs.gen_seen);
    if ((res & 0xf) == kBarLast) {
      if (p.dyn_sched && threadIdx.x == 0) p.bar->chunk[((bs.gen_seen >> 1) + 1u) & 1u] = 0u;
      const int mine = serial_update<Phys, Tab, Real>(p, 1, false, true);
      const int all = __syncthreads_and(mine);
      serial_geometry<Tab>(p);
      if (threadIdx.x == 0) *p.all_done = all;
      barrier_release(p.bar, 0, &bs.gen_seen);
    }
    return;
  }
  for (int step = 0; step < p.n_steps; ++step) {
    if (!all_passes<Phys, Tab, Real, kCF, 0>(p, bs, dyn_smem)) return;
    // the release of the final pass carried "every instance finished" in bit 4 of bs.flag
    if (bs.flag & 0x10) return;
  }
}

}  // namespace xflat
