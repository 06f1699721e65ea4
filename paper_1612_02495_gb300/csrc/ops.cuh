// Per-point stencil operators of the three schemes, in a fixed operation order.
//
// Every floating-point operation is an explicit round-to-nearest intrinsic
// (__fma_rn, __dadd_rn, __dmul_rn, __ddiv_rn, __dsqrt_rn and the float forms),
// so the compiler cannot contract or reorder them; the swept kernels and the
// classic kernels call the same operator, which is what makes the two paths
// agree bit for bit.  Constants are stored and multiplied instead of divided by
// (Section "Results", Fig. divisionComparison).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "fixadd.cuh"
#include "swept_geom.cuh"

namespace swept {

__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float sub_rn(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float div_rn(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ double div_rn(double a, double b) { return __ddiv_rn(a, b); }
__device__ __forceinline__ float sqrt_rn(float a) { return __fsqrt_rn(a); }
__device__ __forceinline__ double sqrt_rn(double a) { return __dsqrt_rn(a); }

// ---------------------------------------------------------------------------
// Heat, FTCS (Eq. HeatDisc): T' = Fo (T_{i+1} + T_{i-1}) + (1 - 2 Fo) T_i
// order: s = T_{i+1} + T_{i-1};  T' = fma(Fo, s, c1 * T_i)
// ---------------------------------------------------------------------------
template <typename T>
struct HeatOp {
  static constexpr int R = 1, S = 1, C = 1;
  struct K {
    T fo, c1;
  };
  // v[0..2] = T_{i-1}, T_i, T_{i+1} at the previous tier
  template <int STAGE>
  __device__ __forceinline__ static T point_fp(const T* v, T /*prev2*/, const K& k) {
    const T s = add_rn(v[2], v[0]);
    return fma_rn(k.fo, s, mul_rn(k.c1, v[1]));
  }
  template <int STAGE>
  __device__ __forceinline__ static T point(const T* v, T prev2, const K& k) {
    return point_fp<STAGE>(v, prev2, k);
  }
};

// ---------------------------------------------------------------------------
// Kuramoto-Sivashinsky, Eq. KSDisc (u_i term read as -2 u_i, factor nu on the
// fourth difference), midpoint RK2 (Appendix).  f = -g with
//   sp1 = u_{i+1} + u_{i-1};  sp2 = u_{i+2} + u_{i-2}
//   nl  = fma(u_{i+1}, u_{i+1}, -(u_{i-1} u_{i-1}))
//   d2  = fma(-2, u_i, sp1);  d4 = fma(6, u_i, fma(-4, sp1, sp2))
//   g   = fma(c_4, d4, fma(c_2, d2, c_a nl))
// stage 0 (predictor, odd tiers):  P  = fma(-dt/2, g(u), u_i)
// stage 1 (final, even tiers):     u' = fma(-dt,   g(P), u_i)   u_i from two tiers back
// ---------------------------------------------------------------------------
template <typename T>
struct KsOp {
  static constexpr int R = 2, S = 2, C = 1;
  struct K {
    T ca, c2, c4, mdth, mdt;
  };
  // the common end of g: from u_{i+1}, u_{i-1}^2 and the two differences
  __device__ __forceinline__ static T combine(T up, T um2, T d2, T d4, const K& k) {
    return fma_rn(k.c4, d4, fma_rn(k.c2, d2, mul_rn(k.ca, fma_rn(up, up, -um2))));
  }
  __device__ __forceinline__ static T g(const T* v, const K& k) {
    const T sp1 = add_rn(v[3], v[1]);
    const T sp2 = add_rn(v[4], v[0]);
    const T d2 = fma_rn(T(-2), v[2], sp1);
    const T d4 = fma_rn(T(6), v[2], fma_rn(T(-4), sp1, sp2));
    return combine(v[3], mul_rn(v[1], v[1]), d2, d4, k);
  }
  // v[0..4] = u_{i-2} .. u_{i+2} at the previous tier; prev2 = u_i two tiers back.
  // point_fp: every operation on the floating-point pipes.
  template <int STAGE>
  __device__ __forceinline__ static T point_fp(const T* v, T prev2, const K& k) {
    return fma_rn(STAGE == 0 ? k.mdth : k.mdt, g(v, k), STAGE == 0 ? v[2] : prev2);
  }
  // FP64: the sums, differences and the square on the integer pipes (fixadd.cuh),
  // five of the eleven operations on the FP64 pipe.  False (r meaningless) where
  // the integer arithmetic does not handle an operand; the caller then takes
  // point_fp, behind a real branch: a FP64 instruction whose guard predicate is
  // false holds the pipe as long as one that runs (77 cycles).
  template <int STAGE>
  __device__ __forceinline__ static bool point_int(const T* v, T prev2, const K& k, T& r) {
    T d2, d4, um2;
    const bool lin = fix::second_fourth(v[0], v[1], v[2], v[3], v[4], d2, d4);
    const bool sq = fix::square(v[1], um2);
    r = fma_rn(STAGE == 0 ? k.mdth : k.mdt, combine(v[3], um2, d2, d4, k), STAGE == 0 ? v[2] : prev2);
    return lin && sq;
  }
  // u_{i-1}^2 and the two differences in FP64, out of line: a call is never turned into
  // predicated instructions
  struct Parts {
    T um2, d2, d4;
  };
  __device__ __noinline__ static Parts parts_fp(T a, T b, T c, T d, T e) {
    const T sp1 = add_rn(d, b), sp2 = add_rn(e, a);
    return Parts{mul_rn(b, b), fma_rn(T(-2), c, sp1), fma_rn(T(6), c, fma_rn(T(-4), sp1, sp2))};
  }
  // One point by itself (the classic kernels, whose warps keep nothing from one sub-timestep to the
  // next).  The integer form is tried where it is likely to hold for the whole warp: operands in its
  // range, and differences that do not vanish beside them in single precision (bits cut off, no FP64
  // instruction).  The branch for a point that fails all the same comes before the common end, so that it
  // issues the eleven FP64 operations once.
  template <int STAGE>
  __device__ __forceinline__ static T point(const T* v, T prev2, const K& k) {
    if constexpr (sizeof(T) == 8) {
      if (!__all_sync(__activemask(), fix::differ(v[0], v[1], v[2], v[3], v[4]))) return point_fp<STAGE>(v, prev2, k);
      Parts p;
      const bool lin = fix::second_fourth(v[0], v[1], v[2], v[3], v[4], p.d2, p.d4);
      const bool sq = fix::square(v[1], p.um2);
      if (!(lin && sq)) p = parts_fp(v[0], v[1], v[2], v[3], v[4]);
      return fma_rn(STAGE == 0 ? k.mdth : k.mdt, combine(v[3], p.um2, p.d2, p.d4, k), STAGE == 0 ? v[2] : prev2);
    } else {
      return point_fp<STAGE>(v, prev2, k);
    }
  }
};

// ---------------------------------------------------------------------------
// 1D Euler, finite volume (not in the paper): MUSCL-minmod on primitives,
// Rusanov flux, SSP-RK2.  Order (per face i+1/2 from cells i-1..i+2):
//   cell:   u = m / rho;  p = gm1 fma(-(0.5 m), u, E)
//   qL = q_i + 0.5 minmod(q_i - q_{i-1}, q_{i+1} - q_i)
//   qR = q_{i+1} - 0.5 minmod(q_{i+1} - q_i, q_{i+2} - q_{i+1})
//   mX = rhoX uX;  EX = fma(0.5 mX, uX, pX igm1);  cX = sqrt((gamma pX) / rhoX)
//   s  = max(|uL| + cL, |uR| + cR)
//   F  = 0.5 fma(-s, UR - UL, FL + FR),  F = (m, fma(m, u, p), u (E + p))
//   stage 0:  U1 = fma(-dt/dx, F+ - F-, U)
//   stage 1:  t = fma(-dt/dx, F+ - F-, U1);  U' = 0.5 (U + t)
// Across a reflective wall a cell is read as its mirror with u negated.
// ---------------------------------------------------------------------------
// minmod(a, b): the argument of smaller magnitude when a and b are both
// positive or both negative, else 0.  Evaluated on the integer pipe from the
// IEEE bit patterns: for values of one sign, magnitude order is the order of
// the patterns' magnitude fields, and with equal sign bits a <= b (both
// positive) and a >= b (both negative) are both "bits(a) <= bits(b)" as signed
// integers.  The selection equals the comparison form for every non-NaN input
// (signed zeros, subnormals, infinities included), without spending FP64 issue
// slots on sign tests and compares.
__device__ __forceinline__ double minmod(double a, double b) {
  const long long ia = __double_as_longlong(a), ib = __double_as_longlong(b);
  const long long mag = 0x7fffffffffffffffLL;
  const bool same_sign_nonzero = ((ia ^ ib) >= 0) && (ia & mag) != 0 && (ib & mag) != 0;
  return same_sign_nonzero ? (ia <= ib ? a : b) : 0.0;
}
__device__ __forceinline__ float minmod(float a, float b) {
  const int ia = __float_as_int(a), ib = __float_as_int(b);
  const int mag = 0x7fffffff;
  const bool same_sign_nonzero = ((ia ^ ib) >= 0) && (ia & mag) != 0 && (ib & mag) != 0;
  return same_sign_nonzero ? (ia <= ib ? a : b) : 0.0f;
}
// the larger of two non-negative values, by their bit patterns (same rule)
__device__ __forceinline__ double max_nonneg(double a, double b) {
  return __double_as_longlong(a) >= __double_as_longlong(b) ? a : b;
}
__device__ __forceinline__ float max_nonneg(float a, float b) { return __float_as_int(a) >= __float_as_int(b) ? a : b; }

// 0.5 x, in FP64 on the integer pipe
__device__ __forceinline__ float half_of(float x) { return mul_rn(0.5f, x); }
__device__ __forceinline__ double half_of(double x) { return fix::half(x); }

template <typename T>
struct EulerOp {
  static constexpr int R = 2, S = 2, C = 3;
  struct K {
    T gamma, gm1, igm1, mdtdx;
  };
  struct Prim {
    T r, u, p;
  };
  __device__ __forceinline__ static Prim prim(T r, T m, T e, const K& k) {
    Prim w;
    w.r = r;
    w.u = div_rn(m, r);
    w.p = mul_rn(k.gm1, fma_rn(-half_of(m), w.u, e));
    return w;
  }
  // One side of a face: the MUSCL-minmod reconstructed state with its
  // momentum, energy and wave-speed bound.  Left side from cells a, b, c
  // (value at the right end of b), right side from b, c, d (left end of c).
  struct Side {
    T r, u, p, m, E, sp;
  };
  __device__ __forceinline__ static T speed(T r, T u, T p, T gamma) {
    return add_rn(fabs(u), sqrt_rn(div_rn(mul_rn(gamma, p), r)));
  }
  __device__ __noinline__ static T speed_cold(T r, T u, T p, T gamma) { return speed(r, u, p, gamma); }
  __device__ __forceinline__ static void finish_state(Side& X, const K& k) {
    X.m = mul_rn(X.r, X.u);
    X.E = fma_rn(half_of(X.m), X.u, mul_rn(X.p, k.igm1));
  }
  __device__ __forceinline__ static void finish_side(Side& X, const K& k) {
    finish_state(X, k);
    X.sp = speed(X.r, X.u, X.p, k.gamma);
  }
  // the reconstructed states, without momentum, energy and speed
  __device__ __forceinline__ static void left_state(Side& L, const Prim& a, const Prim& b, const Prim& c) {
    L.r = add_rn(b.r, half_of(minmod(sub_rn(b.r, a.r), sub_rn(c.r, b.r))));
    L.u = add_rn(b.u, half_of(minmod(sub_rn(b.u, a.u), sub_rn(c.u, b.u))));
    L.p = add_rn(b.p, half_of(minmod(sub_rn(b.p, a.p), sub_rn(c.p, b.p))));
  }
  __device__ __forceinline__ static void right_state(Side& R, const Prim& b, const Prim& c, const Prim& d) {
    R.r = sub_rn(c.r, half_of(minmod(sub_rn(c.r, b.r), sub_rn(d.r, c.r))));
    R.u = sub_rn(c.u, half_of(minmod(sub_rn(c.u, b.u), sub_rn(d.u, c.u))));
    R.p = sub_rn(c.p, half_of(minmod(sub_rn(c.p, b.p), sub_rn(d.p, c.p))));
  }
  // Rusanov flux from the two sides: 1/2 (F(L) + F(R)) - 1/2 s (U_R - U_L),
  // s = the larger of |u| + c over the two sides
  // sp = |u| + c >= 0 on both sides
  __device__ __forceinline__ static T smax(const Side& L, const Side& R) { return max_nonneg(L.sp, R.sp); }
  // The same, from the states alone.  A division and a square root are 26 of the
  // 127 FP64 pipe slots a cell and sub-step took with both sides' speeds, so in
  // FP64 only the faster side's is computed: which it is shows in single
  // precision (from truncated bits, no FP64 instruction) when the estimates differ
  // by more than 2^-20 of their sum.  In units of 2^-23: truncated gamma and p make the quotient smaller by 2 and
  // truncated rho larger by 1, the product's rounding is 1/2 and __fdividef's 2, together 4.5 at most; the root
  // halves them and adds 1, truncated |u| is within 1 and the sum's rounding 1/2.  So an estimate is within 3.75 units,
  // 2^-21.1, of its speed, and their difference within 2^-21.1 of the sum of the speeds.  gamma > 1 (swept_init)
  // keeps the quotient a normal float and makes |u| < 2^-100 nothing beside c.
  // On smooth flow the sides are closer than that and both speeds are computed, the second out of line
  // (2^16 cells, one sine wave, 200 steps: 6.81 ms; with both inline and the halvings on the FP64 pipe 7.53).
  // Sides with the same bits have the same speed; everything else computes both.
  __device__ __forceinline__ static T speed_max(const Side& L, const Side& R, const K& k) {
    if constexpr (sizeof(T) == 8) {
      const uint32_t ml = fix::mag(L.u), mr = fix::mag(R.u);
      const float g = fix::float_bits(k.gamma);
      const float ul = ml < (923u << 20) ? 0.f : fabsf(fix::float_bits(L.u));  // below 2^-100: nothing beside c
      const float ur = mr < (923u << 20) ? 0.f : fabsf(fix::float_bits(R.u));
      float cl, cr;
      asm("sqrt.approx.f32 %0, %1;" : "=f"(cl) : "f"(__fdividef(g * fix::float_bits(L.p), fix::float_bits(L.r))));
      asm("sqrt.approx.f32 %0, %1;" : "=f"(cr) : "f"(__fdividef(g * fix::float_bits(R.p), fix::float_bits(R.r))));
      const float sl = ul + cl, sr = ur + cr;
      const bool left = sl > sr;
      // p, rho and gamma within 2^-60 .. 2^59 (positive), |u| below 2^60
      const bool fits = fix::mid(L.p) && fix::mid(L.r) && fix::mid(R.p) && fix::mid(R.r) && fix::mid(k.gamma) &&
                        fix::umax(ml, mr) < (1083u << 20);
      const bool same = __double_as_longlong(L.p) == __double_as_longlong(R.p) &&
                        __double_as_longlong(L.r) == __double_as_longlong(R.r) &&
                        __double_as_longlong(L.u) == __double_as_longlong(R.u);
      T s = speed(left ? L.r : R.r, left ? L.u : R.u, left ? L.p : R.p, k.gamma);
      if (!((fits && fabsf(sl - sr) > (sl + sr) * 0x1p-20f) || same))
        s = max_nonneg(s, speed_cold(left ? R.r : L.r, left ? R.u : L.u, left ? R.p : L.p, k.gamma));
      return s;
    } else {
      return max_nonneg(speed(L.r, L.u, L.p, k.gamma), speed(R.r, R.u, R.p, k.gamma));
    }
  }
  __device__ __forceinline__ static T flux0(const Side& L, const Side& R, T s) {
    return half_of(fma_rn(-s, sub_rn(R.r, L.r), add_rn(L.m, R.m)));
  }
  __device__ __forceinline__ static T flux1(const Side& L, const Side& R, T s) {
    return half_of(fma_rn(-s, sub_rn(R.m, L.m), add_rn(fma_rn(L.m, L.u, L.p), fma_rn(R.m, R.u, R.p))));
  }
  __device__ __forceinline__ static T flux2(const Side& L, const Side& R, T s) {
    return half_of(
        fma_rn(-s, sub_rn(R.E, L.E), add_rn(mul_rn(L.u, add_rn(L.E, L.p)), mul_rn(R.u, add_rn(R.E, R.p)))));
  }
  // Rusanov flux through the face between cells b and c, from cells a, b, c, d
  __device__ __forceinline__ static void flux(const Prim& a, const Prim& b, const Prim& c, const Prim& d, const K& k,
                                              T& F0, T& F1, T& F2) {
    Side L, R;
    left_state(L, a, b, c);
    right_state(R, b, c, d);
    const T s = speed_max(L, R, k);
    finish_state(L, k);
    finish_state(R, k);
    F0 = flux0(L, R, s);
    F1 = flux1(L, R, s);
    F2 = flux2(L, R, s);
  }
  template <int STAGE>
  __device__ __forceinline__ static T update(T fp, T fm, T in_self, T prev2, const K& k) {
    if (STAGE == 0) return fma_rn(k.mdtdx, sub_rn(fp, fm), in_self);
    const T t = fma_rn(k.mdtdx, sub_rn(fp, fm), in_self);
    return half_of(add_rn(prev2, t));
  }
};

// ---------------------------------------------------------------------------
// Discrete adjoints (not in the paper): the exact transposes of the forward
// operation sequence, run backwards in time as the same two-stage, radius-r
// stencil, with the forward state of each tier read from a tape.
//
// KS, reverse of one step m (lam' = dL/du^{m+1}):
//   gT(lam; w)_j = fma(c_4, d4, fma(c_2, d2, (2 c_a w_j)(lam_{j-1} - lam_{j+1})))
//     with sp1, sp2, d2, d4 of lam as in the forward operator
//   stage 0:  mu  = -dt gT(lam'; P^m)                       (odd reverse tiers)
//   stage 1:  lam = fma(-dt/2, gT(mu; u^m), lam' + mu)      (even reverse tiers)
// dL/dnu = sum -dt k4 lam'_j d4(P^m)_j - (dt/2) k4 mu_j d4(u^m)_j, accumulated as
// the equal sums -dt k4 d4(lam')_j P^m_j and -(dt/2) k4 d4(mu)_j u^m_j (the
// periodic fourth difference is symmetric), so the d4 already computed in gT
// is reused.
// ---------------------------------------------------------------------------
// Compensated (Kahan) accumulation of the parameter derivative: the error is
// about 2 eps sum|terms|, independent of the number of terms; the value is
// the double-double (s, -c).
struct KahanAcc {
  double s = 0.0, c = 0.0;
  __device__ __forceinline__ void add(double x) {
    const double y = __dsub_rn(x, c);
    const double t = __dadd_rn(s, y);
    c = __dsub_rn(__dsub_rn(t, s), y);
    s = t;
  }
};

template <typename T>
struct KsAdjOp {
  static constexpr int R = 2, S = 2, C = 1;
  struct K {
    T ca2, c2, c4, mdt, mdth, mdtk4, mdthk4;
  };
  // v[0..4] = lam_{j-2} .. lam_{j+2}; w = forward state at j; d4 returned for dnu
  __device__ __forceinline__ static T gT(const T* v, T w, const K& k, T& d4) {
    const T sp1 = add_rn(v[3], v[1]);
    const T sp2 = add_rn(v[4], v[0]);
    const T dl = sub_rn(v[1], v[3]);
    const T nl = mul_rn(mul_rn(k.ca2, w), dl);
    const T d2 = fma_rn(T(-2), v[2], sp1);
    d4 = fma_rn(T(6), v[2], fma_rn(T(-4), sp1, sp2));
    return fma_rn(k.c4, d4, fma_rn(k.c2, d2, nl));
  }
  // FP64: the three sums and differences on the integer pipes (fixadd.cuh), 11 or
  // 12 of the 17 or 18 operations on the FP64 pipe.  False, with nothing
  // accumulated, where they do not handle an operand; the caller then takes point.
  template <int STAGE>
  __device__ __forceinline__ static bool point_int(const T* v, T prev2, T w, const K& k, KahanAcc& acc, T& r) {
    T d2, d4, dl;
    const bool ok = fix::second_fourth(v[0], v[1], v[2], v[3], v[4], d2, d4, &dl);
    const T g = fma_rn(k.c4, d4, fma_rn(k.c2, d2, mul_rn(mul_rn(k.ca2, w), dl)));
    r = STAGE == 0 ? mul_rn(k.mdt, g) : fma_rn(k.mdth, g, add_rn(prev2, v[2]));
    KahanAcc sum = acc;
    sum.add((double)mul_rn(mul_rn(STAGE == 0 ? k.mdtk4 : k.mdthk4, d4), w));
    acc.s = ok ? sum.s : acc.s;
    acc.c = ok ? sum.c : acc.c;
    return ok;
  }
  template <int STAGE>
  __device__ __forceinline__ static T point(const T* v, T prev2, T w, const K& k, KahanAcc& acc) {
    T d4;
    const T g = gT(v, w, k, d4);
    if (STAGE == 0) {
      acc.add((double)mul_rn(mul_rn(k.mdtk4, d4), w));
      return mul_rn(k.mdt, g);
    }
    acc.add((double)mul_rn(mul_rn(k.mdthk4, d4), w));
    return fma_rn(k.mdth, g, add_rn(prev2, v[2]));
  }
};

// Heat: FTCS is linear with a symmetric stencil, so the reverse step is the
// forward update applied to lam:  lam_j = fma(Fo, lam'_{j+1} + lam'_{j-1}, c1 lam'_j).
// dL/dalpha = sum (dt/dx^2) lam'_j (T_{j+1} + T_{j-1} - 2 T_j)^m, accumulated as
// the equal sum (dt/dx^2) (lam'_{j+1} + lam'_{j-1} - 2 lam'_j) T^m_j.
template <typename T>
struct HeatAdjOp {
  static constexpr int R = 1, S = 1, C = 1;
  struct K {
    T fo, c1, kk;
  };
  template <int STAGE>
  __device__ __forceinline__ static T point(const T* v, T /*prev2*/, T w, const K& k, KahanAcc& acc) {
    const T s = add_rn(v[2], v[0]);
    acc.add((double)mul_rn(mul_rn(k.kk, fma_rn(T(-2), v[1], s)), w));
    return fma_rn(k.fo, s, mul_rn(k.c1, v[1]));
  }
};

}  // namespace swept
