// lj_minimize.cuh -- one team minimises one LJ cluster with L-BFGS.
//
// Method (arXiv 2510.25938, Methodology, "Algorithm Overview" step 2 and
// "Implementation Notes": L-BFGS-B from scipy, no bounds), read as:
//   direction   two-loop recursion, H0 = (s^T y / y^T y) I of the newest pair
//               (Nocedal & Wright Alg. 7.4); steepest descent when the
//               history is empty or the direction is not a descent direction;
//   first trial alpha = min(1, 1/||d||_2) with an empty history, else 1;
//   line search strong Wolfe, c1 = 1e-3, c2 = 0.9, bracketing with doubling
//               (N&W Alg. 3.5) and zoom with safeguarded cubic interpolation
//               (N&W Alg. 3.6, eq. 3.59); a non-finite energy fails the
//               sufficient-decrease test; after max_ls evaluations the best
//               sufficient-decrease point is taken if it strictly lowers E;
//               on failure one retry along -g with an empty history;
//   curvature   the pair (s, y) is stored only if s^T y > eps_mach y^T y;
//   stopping    ||g||_inf < gtol after each accepted step (and at the start).
//
// Precision (GB300: FP64 issues ~1/62 of FP32, the FP64 reciprocal less):
//   FP64 path   every operation in FP64.
//   MIXED path  phase 1: coordinates, gradient, directions and history in
//               FP32, energy as float-float, line-search scalars in FP32, no
//               FP64 instruction at all; it ends when ||g32||_inf <
//               switch_gtol, when the predicted decrease falls below the FP32
//               energy resolution, or when its line search fails.
//               phase 2 (polish): coordinates and pair terms in double-float
//               arithmetic (FP32 pipes, ~1e-14 relative), gradient FP32
//               (only its relative precision is used there), energies
//               float-float, line-search scalars FP32: no FP64 instruction.
//               It hands over once the predicted decrease falls below the
//               double-float energy resolution (~32 * 2^-48 |E|).
//               phase 3: FP64 coordinates, gradient, energy and pair terms
//               for the last iterations (FP32 directions and scalars); the
//               convergence test and the returned energy are always FP64.
#pragma once
#include <type_traits>

#include "lj_device.cuh"
#include "lj_teams.cuh"
#include "lj_consts.h"
#include "../../include/lj_bh.h"

namespace ljd {

struct MinParams {
  int m, max_iter, max_ls;
  double gtol, c1, c2, alpha_max, switch_gtol;
  long long deadline;
  ljh::LjConsts k;         // pair-potential constants (host-derived)
  int layout;              // what hbuf holds (PairLayout)
  int ring_ks;             // ... its ring chunk, in shifts
  double f32_resolution;   // FP32 phase hands over below this predicted decrease / |E|
  double df_resolution;    // double-float polish hands over below this / |E|
};

struct MinResult {
  double E;
  int status;
  int iters;
  int evals32, evals64, evals_df, iters32, iters64;
  long long vec32, vec64;   // sum over iterations of (history used) * 3N
  long long cyc32, cycdf, cyc64;   // SM clock cycles spent in each tier
  long long cycdir, cycls;          // ... in direction computations and line searches
};

enum : int { PH_CONVERGED = 0, PH_MAXITER = 1, PH_LSFAIL = 2, PH_SWITCH = 3, PH_TIMEOUT = 4 };

// FP32-tier iterations after which gradient-only FP32 steps hand over: a
// safety net for a switch_gtol below the FP32 gradient noise (~3e-5 eps/sigma
// on LJ clusters); normal minimisations stay far below it
constexpr int kFP32GradIters = 2000;

// Precision policy of an L-BFGS tier.
//   XP positions (float, double, or ff = double-float), XG gradient, V search
//   directions and history, PM pair arithmetic (0: XP's own, 1: double-float).
//   S line-search scalars: FP64 only on the all-FP64 path.  F energies: FP64
//   when positions are FP64, float-float otherwise (FP32 pipes only).
template <typename XP_, typename XG_, typename V_, int PM_, int POT_ = LJ_POT_LJ>
struct Prec {
  using XP = XP_;
  using XG = XG_;
  using V = V_;
  static constexpr int PM = PM_;
  static constexpr int POT = POT_;   // pair potential: LJ_POT_LJ or LJ_POT_MORSE
  using S = std::conditional_t<sizeof(V_) == 8, double, float>;
  using F = std::conditional_t<std::is_same<XP_, double>::value, double, ff>;
};
// trial position x + a d and step xt - x for each position type
__device__ __forceinline__ float pos_step(float x, float a, float d) { return x + a * d; }
template <typename SA, typename VD>
__device__ __forceinline__ double pos_step(double x, SA a, VD d) {
  return x + (double)a * (double)d;
}
__device__ __forceinline__ ff pos_step(ff x, float a, float d) {
  return df_add(x, df_two_prod(a, d));
}
template <typename V> __device__ __forceinline__ V pos_diff(float xt, float x) { return (V)(xt - x); }
template <typename V> __device__ __forceinline__ V pos_diff(double xt, double x) { return (V)(xt - x); }
template <typename V> __device__ __forceinline__ V pos_diff(ff xt, ff x) {
  const ff d = df_sub(xt, x);
  return (V)(d.hi + d.lo);
}

template <typename V> __device__ __forceinline__ V eps_mach();
template <> __device__ __forceinline__ float eps_mach<float>() { return 1.1920928955078125e-7f; }
template <> __device__ __forceinline__ double eps_mach<double>() { return 2.220446049250313e-16; }

__device__ __forceinline__ float S_sqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double S_sqrt(double x) { return sqrt(x); }

// history element (slot, atom slot a, component c) of this thread: a slot is
// the flattened 3N vector for FP32 history of teams whose first warp runs the
// recursion (it reads 16 bytes a lane), one plane per (a, c) otherwise
template <int T, int A, typename V>
__device__ __forceinline__ int hidx(int slot, int a, int c, int rank) {
  if constexpr (T <= 128 && sizeof(V) == 4) return (slot * A * T + a * T + rank) * 3 + c;
  else return ((slot * A + a) * 3 + c) * T + rank;
}

// ---------------------------------------------------------------------------
// Energy and gradient at x (owned atoms), and dphi = g . d when d != nullptr.
// ---------------------------------------------------------------------------
// PM = 0: pair terms in X precision; PM = 1 (X = double only): pair terms in
// double-float arithmetic on coordinates scaled by 1/sigma.
// hbuf: the team's pair buffer, laid out as p.layout says, or nullptr (FP64 path from
// 65 to 256 atoms, one-sided rows chosen above); FP64 and double-float
// evaluations with one compute each pair once, others in one-sided rows.
// Mixed-precision teams of up to 256 atoms always have one; their rows stay compiled
// because without them the rest is scheduled worse (LJ38 Basin Hopping, 64 walkers x
// 8, 25 steps: 10.48 against 10.14 ms).
// ---------------------------------------------------------------------------
// Morse pair potential (Morse 1929, cluster form), the pair-potential
// extension of the method: V(r) = eps e (e - 2), e = exp(rho (1 - r / re)),
// re in the sigma slot.  FP32 (and FP64 without a pair buffer) in one-sided rows:
// every thread sums, for each atom it owns, the terms of all other atoms;
// E = (eps / 2) sum_i sum_{j != i} e (e - 2), and
// g_i = -(2 eps rho / re) sum_{j != i} e (e - 1) (x_i - x_j) / r.
// FP32 (first tier of the mixed path; compensated energy), double-float
// (evaluate_morse_df, the polish tier) and FP64; those two take each pair once
// through the team's buffer where there is one, up to 256 atoms, as for Eq. (1)
// (half pairs, ring).
// Coincident atoms give E = +inf (and a non-finite gradient), as for Eq. (1).
// ---------------------------------------------------------------------------
__device__ __forceinline__ float to_value(ff v) { return v.hi + v.lo; }
__device__ __forceinline__ double to_value(double v) { return v; }

// FP64 half pairs and row sums; V: the tier's direction type (double: the FP64 path)
template <int T, typename V, typename Term>
__device__ __forceinline__ void half_f64(const Team<T>& tm, int n, double* vb, Term&& term,
                                         double gs, double* gsum, dd& e) {
  if constexpr (sizeof(V) == 8) {
    tri_pairs<T>(tm.rank, n, vb, term, e);
    tm.sync();
    tri_rows<T>(tm.rank, n, vb, gs, gsum);
  } else {
    half_pairs<T>(tm.rank, n, vb, term, [&](double ep) { dd_acc(e, ep); });
    tm.sync();
    half_rows<T>(tm.rank, n, vb, -gs, gsum);
  }
}

// gradient of the owned atoms from the ring's sums, and this thread's g.d
template <int T, int A, typename P, typename F, typename G>
__device__ __forceinline__ void ring_gradient(const Team<T>& tm, int n, const F (&acc)[A][3],
                                              G scale, typename P::XG (&g)[A][3],
                                              const typename P::V (*d)[3], typename P::V& dp) {
  using V = typename P::V;
#pragma unroll
  for (int a = 0; a < A; ++a) {
    const bool in = tm.rank + a * T < n;
#pragma unroll
    for (int c = 0; c < 3; ++c) g[a][c] = in ? scale * to_value(acc[a][c]) : (typename P::XG)0;
    if (d) dp += (V)g[a][0] * d[a][0] + (V)g[a][1] * d[a][1] + (V)g[a][2] * d[a][2];
  }
}

__device__ __forceinline__ void pair_term_morse_f64(const PosD& a, const PosD& b, double rho,
                                                    double rr, double& vx, double& vy,
                                                    double& vz, double& e) {
  const double dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z;
  const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
  const double r = sqrt(r2);
  const double ex = exp(fma(-rr, r, rho));
  e = r2 > 0.0 ? ex * (ex - 2.0) : __longlong_as_double(0x7ff0000000000000LL);
  const double c = ex * (ex - 1.0) / r;
  vx = c * dx; vy = c * dy; vz = c * dz;
}

// Double-float Morse evaluation (the mixed path's polish tier): positions
// scaled by 1/re, pair terms by pair_term_morse_df (double-float exponential
// and square root); each pair once through the team's buffer up to 256 atoms
// (half pairs, ring), one-sided rows above.
template <int T, int A, typename P>
__device__ __forceinline__ void evaluate_morse_df(const Team<T>& tm, int n,
                                                  const typename P::XP (&x)[A][3],
                                                  typename P::XG (&g)[A][3], void* posv,
                                                  void* hbuf, const MinParams& p,
                                                  const typename P::V (*d)[3],
                                                  typename P::F& E, typename P::S& dphi) {
  using V = typename P::V;
  using S = typename P::S;
  PosDF* pos = static_cast<PosDF*>(posv);
  tm.sync();  // previous readers of pos are done
#pragma unroll
  for (int a = 0; a < A; ++a) {
    const int i = tm.rank + a * T;
    if (i < n) {
      ff qx = x[a][0], qy = x[a][1], qz = x[a][2];
      if (p.k.sigma != 1.0) {
        const ff is{p.k.is_hi, p.k.is_lo};
        qx = df_mul(qx, is); qy = df_mul(qy, is); qz = df_mul(qz, is);
      }
      pos[i] = PosDF{qx.hi, qy.hi, qz.hi, 0.f, qx.lo, qy.lo, qz.lo, 0.f};
    }
  }
  tm.sync();
  const ff rho{p.k.rho_f, p.k.rho_lo};
  const float gs = p.k.m_g_f;
  V dp = (V)0;
  ff e{0.f, 0.f};
  if (hbuf != nullptr && p.layout == LAYOUT_HALF) {
    ff* vb = static_cast<ff*>(hbuf);
    float* gsum = static_cast<float*>(posv);
    half_pairs<T>(tm.rank, n, vb,
                  [&](int i, int j, ff& vx, ff& vy, ff& vz, ff& ep) {
                    pair_term_morse_df(pos[i], pos[j], rho, vx, vy, vz, ep);
                  },
                  [&](ff ep) { df_acc(e, ep); });
    tm.sync();
    half_rows<T>(tm.rank, n, vb, -gs, gsum);
    tm.sync();
#pragma unroll
    for (int a = 0; a < A; ++a) {
      const int ii = tm.rank + a * T;
      if (ii < n) {
        g[a][0] = gsum[3 * ii]; g[a][1] = gsum[3 * ii + 1]; g[a][2] = gsum[3 * ii + 2];
      } else {
        g[a][0] = 0.f; g[a][1] = 0.f; g[a][2] = 0.f;
      }
      if (d) dp += (V)g[a][0] * d[a][0] + (V)g[a][1] * d[a][1] + (V)g[a][2] * d[a][2];
    }
    E = ff_scale(team_sum_ff<T>(tm, e), p.k.eps_f);
  } else if (T * A <= 256 && hbuf != nullptr && p.layout == LAYOUT_RING) {
    ff acc[A][3];
    ring_pairs<T, A>(tm, n, p.ring_ks, static_cast<ff*>(hbuf),
                     [&](int i, int j, ff& vx, ff& vy, ff& vz, ff& ep) {
                       pair_term_morse_df(pos[i], pos[j], rho, vx, vy, vz, ep);
                     },
                     [&](ff ep) { df_acc(e, ep); }, acc);
    ring_gradient<T, A, P>(tm, n, acc, -gs, g, d, dp);
    E = ff_scale(team_sum_ff<T>(tm, e), p.k.eps_f);
  } else {
#pragma unroll
    for (int a = 0; a < A; ++a) {
      const int i = tm.rank + a * T;
      if (i < n) {
        const PosDF pi = pos[i];
        ff ax{0.f, 0.f}, ay{0.f, 0.f}, az{0.f, 0.f};
        for (int j = 0; j < n; ++j) {
          ff vx, vy, vz, ep;
          pair_term_morse_df(pi, pos[j], rho, vx, vy, vz, ep);
          if (j != i) {
            df_acc(ax, vx); df_acc(ay, vy); df_acc(az, vz);
            df_acc(e, ep);
          }
        }
        g[a][0] = -gs * (ax.hi + ax.lo);
        g[a][1] = -gs * (ay.hi + ay.lo);
        g[a][2] = -gs * (az.hi + az.lo);
      } else {
        g[a][0] = 0.f; g[a][1] = 0.f; g[a][2] = 0.f;
      }
      if (d) dp += (V)g[a][0] * d[a][0] + (V)g[a][1] * d[a][1] + (V)g[a][2] * d[a][2];
    }
    E = ff_scale(team_sum_ff<T>(tm, e), p.k.m_half_f);
  }
  if (d) dphi = (S)team_sum1<T, V>(tm, dp);
}

template <int T, int A, typename P>
__device__ __forceinline__ void evaluate_morse(const Team<T>& tm, int n,
                                               const typename P::XP (&x)[A][3],
                                               typename P::XG (&g)[A][3], void* posv,
                                               void* hbuf, const MinParams& p,
                                               const typename P::V (*d)[3],
                                               typename P::F& E, typename P::S& dphi) {
  using X = typename P::XP;
  using V = typename P::V;
  using S = typename P::S;
  if constexpr (P::PM == 1) {
    evaluate_morse_df<T, A, P>(tm, n, x, g, posv, hbuf, p, d, E, dphi);
    return;
  } else {
  using Q = typename PosOf<X>::type;
  tm.sync();  // previous readers of pos are done
#pragma unroll
  for (int a = 0; a < A; ++a) {
    const int i = tm.rank + a * T;
    if (i < n) {
      if constexpr (sizeof(X) == 4) {
        stage_f32x2(static_cast<PosF2*>(posv), n, i, x[a][0], x[a][1], x[a][2]);   // packed
      } else {
        Q q;
        q.x = x[a][0]; q.y = x[a][1]; q.z = x[a][2]; q.w = (X)0;
        static_cast<Q*>(posv)[i] = q;
      }
    }
  }
  tm.sync();
  V dp = (V)0;
  if constexpr (sizeof(X) == 4) {
    // packed rows: two pair terms per instruction, as for Eq. (1)
    const PosF2* pos = static_cast<const PosF2*>(posv);
    const float gsc = p.k.m_g_f;
    ff e{0.f, 0.f};
#pragma unroll
    for (int a = 0; a < A; ++a) {
      const int i = tm.rank + a * T;
      if (i < n) {
        float bx, by, bz;
        ff ea{0.f, 0.f};
        morse_row_f32x2(n, i, x[a][0], x[a][1], x[a][2], pos, p.k.rho_f, p.k.rho_re_f, bx, by,
                        bz, ea);
        g[a][0] = gsc * bx; g[a][1] = gsc * by; g[a][2] = gsc * bz;
        e = ff_add(e, ea);
      } else {
        g[a][0] = 0.f; g[a][1] = 0.f; g[a][2] = 0.f;
      }
      if (d) dp += (V)g[a][0] * d[a][0] + (V)g[a][1] * d[a][1] + (V)g[a][2] * d[a][2];
    }
    if constexpr (std::is_same<V, float>::value) {
      if (d) {                  // energy and g.d in one team reduction
        team_sum_ff_f<T>(tm, e, dp);
        E = ff_scale(e, p.k.m_half_f);
        dphi = (S)dp;
        return;
      }
    }
    E = ff_scale(team_sum_ff<T>(tm, e), p.k.m_half_f);
  } else if (hbuf != nullptr && p.layout == LAYOUT_HALF) {
    // ---- half-pair FP64 evaluation (pair phase, then row sums) -------------
    const PosD* pos = static_cast<const PosD*>(posv);
    double* vb = static_cast<double*>(hbuf);
    double* gsum = static_cast<double*>(posv);
    const double rho = p.k.rho, rr = p.k.rho_re;
    dd e{0.0, 0.0};
    auto term = [&](int i, int j, double& vx, double& vy, double& vz, double& ep) {
      pair_term_morse_f64(pos[i], pos[j], rho, rr, vx, vy, vz, ep);
    };
    half_f64<T, V>(tm, n, vb, term, p.k.m_g, gsum, e);
    tm.sync();
#pragma unroll
    for (int a = 0; a < A; ++a) {
      const int ii = tm.rank + a * T;
      if (ii < n) {
        g[a][0] = gsum[3 * ii]; g[a][1] = gsum[3 * ii + 1]; g[a][2] = gsum[3 * ii + 2];
      } else {
        g[a][0] = 0.0; g[a][1] = 0.0; g[a][2] = 0.0;
      }
      if (d) dp += (V)g[a][0] * d[a][0] + (V)g[a][1] * d[a][1] + (V)g[a][2] * d[a][2];
    }
    E = team_sum_dd<T>(tm, e) * p.k.eps;
  } else if (T * A <= 256 && sizeof(V) == 4 && hbuf != nullptr && p.layout == LAYOUT_RING) {
    const PosD* pos = static_cast<const PosD*>(posv);
    const double rho = p.k.rho, rr = p.k.rho_re;
    double acc[A][3];
    dd e{0.0, 0.0};
    ring_pairs<T, A>(tm, n, p.ring_ks, static_cast<double*>(hbuf),
                     [&](int i, int j, double& vx, double& vy, double& vz, double& ep) {
                       pair_term_morse_f64(pos[i], pos[j], rho, rr, vx, vy, vz, ep);
                     },
                     [&](double ep) { dd_acc(e, ep); }, acc);
    ring_gradient<T, A, P>(tm, n, acc, -p.k.m_g, g, d, dp);
    E = team_sum_dd<T>(tm, e) * p.k.eps;
  } else {
    const Q* pos = static_cast<const Q*>(posv);
    const double rho = p.k.rho, rr = p.k.rho_re, gsc = p.k.m_g;
    const double kInf = __longlong_as_double(0x7ff0000000000000LL);
    dd e{0.0, 0.0};
#pragma unroll
    for (int a = 0; a < A; ++a) {
      const int i = tm.rank + a * T;
      if (i < n) {
        const double xi = x[a][0], yi = x[a][1], zi = x[a][2];
        double ax = 0.0, ay = 0.0, az = 0.0;
        for (int j = 0; j < n; ++j) {
          const Q q = pos[j];
          const double dx = xi - q.x, dy = yi - q.y, dz = zi - q.z;
          const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
          const double r = sqrt(r2);
          const double ex = exp(fma(-rr, r, rho));
          double term = ex * (ex - 2.0);
          double c = ex * (ex - 1.0) / r;
          if (j == i) {
            term = 0.0;
            c = 0.0;
          } else if (!(r2 > 0.0)) {
            term = kInf;
          }
          dd_acc(e, term);                        // compensated energy
          ax = fma(c, dx, ax);
          ay = fma(c, dy, ay);
          az = fma(c, dz, az);
        }
        g[a][0] = -gsc * ax; g[a][1] = -gsc * ay; g[a][2] = -gsc * az;
      } else {
        g[a][0] = 0.0; g[a][1] = 0.0; g[a][2] = 0.0;
      }
      if (d) dp += (V)g[a][0] * d[a][0] + (V)g[a][1] * d[a][1] + (V)g[a][2] * d[a][2];
    }
    E = team_sum_dd<T>(tm, e) * p.k.m_half;
  }
  if (d) dphi = (S)team_sum1<T, V>(tm, dp);
  }
}

template <int T, int A, typename P>
__device__ __forceinline__ void evaluate(const Team<T>& tm, int n,
                                         const typename P::XP (&x)[A][3],
                                         typename P::XG (&g)[A][3], void* posv, void* hbuf,
                                         const MinParams& p, const typename P::V (*d)[3],
                                         typename P::F& E, typename P::S& dphi) {
  using X = typename P::XP;
  using XG = typename P::XG;
  using V = typename P::V;
  using S = typename P::S;
  constexpr int PM = P::PM;
  if constexpr (P::POT != LJ_POT_LJ) {
    evaluate_morse<T, A, P>(tm, n, x, g, posv, hbuf, p, d, E, dphi);
    return;
  }
  tm.sync();  // previous readers of pos are done
#pragma unroll
  for (int a = 0; a < A; ++a) {
    const int i = tm.rank + a * T;
    if (i < n) {
      if constexpr (PM == 1) {
        // double-float positions, scaled by 1/sigma (exact for sigma = 1)
        ff qx = x[a][0], qy = x[a][1], qz = x[a][2];
        if (p.k.sigma != 1.0) {
          const ff is{p.k.is_hi, p.k.is_lo};
          qx = df_mul(qx, is); qy = df_mul(qy, is); qz = df_mul(qz, is);
        }
        static_cast<PosDF*>(posv)[i] = PosDF{qx.hi, qy.hi, qz.hi, 0.f, qx.lo, qy.lo, qz.lo, 0.f};
      } else if constexpr (sizeof(X) == 4) {
        stage_f32x2(static_cast<PosF2*>(posv), n, i, x[a][0], x[a][1], x[a][2]);   // packed
      } else {
        typename PosOf<X>::type q;
        q.x = x[a][0]; q.y = x[a][1]; q.z = x[a][2]; q.w = (X)0;
        static_cast<typename PosOf<X>::type*>(posv)[i] = q;
      }
    }
  }
  tm.sync();
  V dp = (V)0;
  if constexpr (PM == 1 || std::is_same<X, double>::value) {
    ff e_df{0.f, 0.f};          // PM == 1: this thread's pair energies
    if (hbuf != nullptr && p.layout == LAYOUT_HALF) {
      // ---- half-pair evaluation: pairs, then one (atom, axis) sum a thread,
      // written over the position buffer (no longer needed) and read back by
      // the owners
      XG* gsum = static_cast<XG*>(posv);
      if constexpr (PM == 1) {
        const PosDF* pos = static_cast<const PosDF*>(posv);
        ff* vb = static_cast<ff*>(hbuf);
        half_pairs<T>(tm.rank, n, vb,
                      [&](int i, int j, ff& vx, ff& vy, ff& vz, ff& ep) {
                        pair_term_df(pos[i], pos[j], vx, vy, vz, ep);
                      },
                      [&](ff ep) { df_acc(e_df, ep); });   // reduced below, with g.d
        tm.sync();
        half_rows<T>(tm.rank, n, vb, -p.k.gs_f, gsum);
        tm.sync();
      } else {
        const PosD* pos = static_cast<const PosD*>(posv);
        double* vb = static_cast<double*>(hbuf);
        const double sig2 = p.k.sig2;
        dd e{0.0, 0.0};
        auto term = [&](int i, int j, double& vx, double& vy, double& vz, double& ep) {
          pair_term_f64(pos[i], pos[j], sig2, vx, vy, vz, ep);
        };
        half_f64<T, V>(tm, n, vb, term, p.k.gscale, gsum, e);
        tm.sync();
        E = team_sum_dd<T>(tm, e) * p.k.e4;
      }
#pragma unroll
      for (int a = 0; a < A; ++a) {
        const int ii = tm.rank + a * T;
        if (ii < n) {
          g[a][0] = gsum[3 * ii]; g[a][1] = gsum[3 * ii + 1]; g[a][2] = gsum[3 * ii + 2];
        } else {
          g[a][0] = 0.0; g[a][1] = 0.0; g[a][2] = 0.0;
        }
        if (d) dp += (V)g[a][0] * d[a][0] + (V)g[a][1] * d[a][1] + (V)g[a][2] * d[a][2];
      }
      if constexpr (PM == 1) {
        // float-float team sum (FP32 pipes): its ~2^-47 relative error is far
        // below the double-float handover resolution; g.d in the same pass
        if constexpr (std::is_same<V, float>::value) {
          if (d) {
            team_sum_ff_f<T>(tm, e_df, dp);
            E = ff_scale(e_df, p.k.e4_f);
            dphi = (S)dp;
            return;
          }
        }
        E = ff_scale(team_sum_ff<T>(tm, e_df), p.k.e4_f);
      }
      if (d) dphi = (S)team_sum1<T, V>(tm, dp);
      return;
    }
  }
  if constexpr ((PM == 1 || std::is_same<X, double>::value) && sizeof(V) == 4 && T * A <= 256) {
    if (hbuf != nullptr && p.layout == LAYOUT_RING) {
      if constexpr (PM == 1) {
        const PosDF* pos = static_cast<const PosDF*>(posv);
        ff acc[A][3], e{0.f, 0.f};
        ring_pairs<T, A>(tm, n, p.ring_ks, static_cast<ff*>(hbuf),
                         [&](int i, int j, ff& vx, ff& vy, ff& vz, ff& ep) {
                           pair_term_df(pos[i], pos[j], vx, vy, vz, ep);
                         },
                         [&](ff ep) { df_acc(e, ep); }, acc);
        ring_gradient<T, A, P>(tm, n, acc, -p.k.gs_f, g, d, dp);
        if constexpr (std::is_same<V, float>::value) {
          if (d) {
            team_sum_ff_f<T>(tm, e, dp);
            E = ff_scale(e, p.k.e4_f);
            dphi = (S)dp;
            return;
          }
        }
        E = ff_scale(team_sum_ff<T>(tm, e), p.k.e4_f);
      } else {
        const PosD* pos = static_cast<const PosD*>(posv);
        const double sig2 = p.k.sig2;
        double acc[A][3];
        dd e{0.0, 0.0};
        ring_pairs<T, A>(tm, n, p.ring_ks, static_cast<double*>(hbuf),
                         [&](int i, int j, double& vx, double& vy, double& vz, double& ep) {
                           pair_term_f64(pos[i], pos[j], sig2, vx, vy, vz, ep);
                         },
                         [&](double ep) { dd_acc(e, ep); }, acc);
        ring_gradient<T, A, P>(tm, n, acc, -p.k.gscale, g, d, dp);
        E = team_sum_dd<T>(tm, e) * p.k.e4;
      }
      if (d) dphi = (S)team_sum1<T, V>(tm, dp);
      return;
    }
  }
  if constexpr (PM == 1) {
    const PosDF* pos = static_cast<const PosDF*>(posv);
    const float gs = p.k.gs_f;
    ff e{0.f, 0.f};
    // ---- tiled half-pair evaluation (teams for more than 256 atoms; compiled
    // only for team shapes that can hold them) ------------------------------
    if constexpr (T * A > 256) {
    if (hbuf != nullptr && p.layout == LAYOUT_TILES) {
      ff* acc = static_cast<ff*>(hbuf);
      df_tile_eval<T>(tm, n, pos, acc, e);
#pragma unroll
      for (int a = 0; a < A; ++a) {
        const int i = tm.rank + a * T;
        if (i < n) {
          const ff sx = acc[i], sy = acc[n + i], sz = acc[2 * n + i];
          g[a][0] = -gs * (sx.hi + sx.lo);
          g[a][1] = -gs * (sy.hi + sy.lo);
          g[a][2] = -gs * (sz.hi + sz.lo);
        } else {
          g[a][0] = (XG)0; g[a][1] = (XG)0; g[a][2] = (XG)0;
        }
        if (d) dp += (V)g[a][0] * d[a][0] + (V)g[a][1] * d[a][1] + (V)g[a][2] * d[a][2];
      }
      if constexpr (std::is_same<V, float>::value) {
        if (d) {
          team_sum_ff_f<T>(tm, e, dp);
          E = ff_scale(e, p.k.e4_f);
          dphi = (S)dp;
          return;
        }
      }
      E = ff_scale(team_sum_ff<T>(tm, e), p.k.e4_f);
      if (d) dphi = (S)team_sum1<T, V>(tm, dp);
      return;
    }
    }
#pragma unroll
    for (int a = 0; a < A; ++a) {
      const int i = tm.rank + a * T;
      if (i < n) {
        const PosDF q = pos[i];
        ff ax, ay, az, ea{0.f, 0.f};
        pair_row_df(n, i, ff{q.xh, q.xl}, ff{q.yh, q.yl}, ff{q.zh, q.zl}, pos, ax, ay, az, ea);
        g[a][0] = -gs * (ax.hi + ax.lo);
        g[a][1] = -gs * (ay.hi + ay.lo);
        g[a][2] = -gs * (az.hi + az.lo);
        e = df_add(e, ea);
      } else {
        g[a][0] = (XG)0; g[a][1] = (XG)0; g[a][2] = (XG)0;
      }
      if (d) dp += (V)g[a][0] * d[a][0] + (V)g[a][1] * d[a][1] + (V)g[a][2] * d[a][2];
    }
    E = ff_scale(team_sum_ff<T>(tm, e), p.k.e2_f);
  } else if constexpr (sizeof(X) == 4) {
    const PosF2* pos = static_cast<const PosF2*>(posv);
    const float gs = p.k.gscale_f;
    const bool unit = p.k.sigma == 1.0;
    ff e{0.f, 0.f};
#pragma unroll
    for (int a = 0; a < A; ++a) {
      const int i = tm.rank + a * T;
      if (i < n) {
        float bx, by, bz;
        ff ea{0.f, 0.f};
        if (unit)
          pair_row_f32x2<false>(n, i, x[a][0], x[a][1], x[a][2], pos, 1.f, bx, by, bz, ea);
        else
          pair_row_f32x2<true>(n, i, x[a][0], x[a][1], x[a][2], pos, p.k.sig2_f, bx, by, bz, ea);
        g[a][0] = gs * bx; g[a][1] = gs * by; g[a][2] = gs * bz;
        e = ff_add(e, ea);
      } else {
        g[a][0] = 0.f; g[a][1] = 0.f; g[a][2] = 0.f;
      }
      if (d) dp += (V)g[a][0] * d[a][0] + (V)g[a][1] * d[a][1] + (V)g[a][2] * d[a][2];
    }
    if constexpr (std::is_same<V, float>::value) {
      if (d) {                  // energy and g.d in one team reduction
        team_sum_ff_f<T>(tm, e, dp);
        E = ff_scale(e, p.k.e2_f);
        dphi = (S)dp;
        return;
      }
    }
    ff et = team_sum_ff<T>(tm, e);
    E = ff_scale(et, p.k.e2_f);
  } else {
    const PosD* pos = static_cast<const PosD*>(posv);
    dd e{0.0, 0.0};
    // ---- tiled FP64 evaluation (teams for more than 256 atoms) -------------
    if constexpr (T * A > 256) {
    if (hbuf != nullptr && p.layout == LAYOUT_TILES) {
      double* acc = static_cast<double*>(hbuf);
      d_tile_eval<T>(tm, n, pos, p.k.sig2, acc, e);
#pragma unroll
      for (int a = 0; a < A; ++a) {
        const int i = tm.rank + a * T;
        if (i < n) {
          g[a][0] = -p.k.gscale * acc[i];
          g[a][1] = -p.k.gscale * acc[n + i];
          g[a][2] = -p.k.gscale * acc[2 * n + i];
        } else {
          g[a][0] = 0.0; g[a][1] = 0.0; g[a][2] = 0.0;
        }
        if (d) dp += (V)g[a][0] * d[a][0] + (V)g[a][1] * d[a][1] + (V)g[a][2] * d[a][2];
      }
      E = team_sum_dd<T>(tm, e) * p.k.e4;
      if (d) dphi = (S)team_sum1<T, V>(tm, dp);
      return;
    }
    }
#pragma unroll
    for (int a = 0; a < A; ++a) {
      const int i = tm.rank + a * T;
      if (i < n) {
        double ax, ay, az;
        pair_row_f64(n, i, x[a][0], x[a][1], x[a][2], pos, p.k.sig2, ax, ay, az, e);
        g[a][0] = -p.k.gscale * ax; g[a][1] = -p.k.gscale * ay; g[a][2] = -p.k.gscale * az;
      } else {
        g[a][0] = 0.0; g[a][1] = 0.0; g[a][2] = 0.0;
      }
      if (d) dp += (V)g[a][0] * d[a][0] + (V)g[a][1] * d[a][1] + (V)g[a][2] * d[a][2];
    }
    E = team_sum_dd<T>(tm, e) * p.k.e2;
  }
  if (d) dphi = (S)team_sum1<T, V>(tm, dp);
}

// largest |g| of this thread as its bit pattern (NaN: above infinity's): bits of
// non-negative floats order as integers, so maxima run on the integer pipe
template <int A>
__device__ __forceinline__ unsigned max_bits(const float (&g)[A][3]) {
  unsigned m = 0;
#pragma unroll
  for (int a = 0; a < A; ++a)
#pragma unroll
    for (int c = 0; c < 3; ++c) m = max(m, __float_as_uint(g[a][c]) & 0x7fffffffu);
  return m;
}
template <int A>
__device__ __forceinline__ unsigned long long max_bits(const double (&g)[A][3]) {
  unsigned long long m = 0;
#pragma unroll
  for (int a = 0; a < A; ++a)
#pragma unroll
    for (int c = 0; c < 3; ++c)
      m = max(m, (unsigned long long)__double_as_longlong(g[a][c]) & 0x7fffffffffffffffULL);
  return m;
}
// back to a value; a NaN anywhere gives infinity
__device__ __forceinline__ float from_bits(unsigned b) {
  return __uint_as_float(min(b, 0x7f800000u));
}
__device__ __forceinline__ double from_bits(unsigned long long b) {
  return __longlong_as_double((long long)min(b, 0x7ff0000000000000ULL));
}

template <int T, int A, typename X>
__device__ __forceinline__ X grad_max(const Team<T>& tm, const X (&g)[A][3]) {
  return from_bits(team_max_bits(tm, max_bits(g)));
}

// Sufficient decrease f(a) <= f(0) + c1 a phi'(0).  FP64-valued energies use
// exactly that expression (the right side rounded to FP64, as the oracle does:
// near the FP64 floor a threshold below half an ulp of f(0) then asks only
// f(a) <= f(0)); float-float energies compare the exact difference.
__device__ __forceinline__ bool armijo_ok(double fa, double f0, double t) {
  return isfinite(fa) && fa <= f0 + t;
}
__device__ __forceinline__ bool armijo_ok(ff fa, ff f0, float t) {
  return fisfinite(fa) && fdiff(fa, f0) <= t;
}

// safeguarded cubic interpolation (N&W eq. 3.59), kept 10% inside the bracket
template <typename S, typename F>
__device__ __forceinline__ S cubic_step(S a, F fa, S ga, S b, F fb, S gb) {
  const S lo = a < b ? a : b;
  const S hi = a < b ? b : a;
  const S w = hi - lo;
  const S mid = (S)0.5 * (a + b);
  if (!(fisfinite(fa) && fisfinite(fb) && isfinite(ga) && isfinite(gb))) return mid;
  const S d1 = ga + gb - (S)3 * ((S)fdiff(fa, fb) / (a - b));
  const S disc = d1 * d1 - ga * gb;
  if (!(disc >= (S)0)) return mid;
  S d2 = S_sqrt(disc);
  if (b - a < (S)0) d2 = -d2;
  const S den = gb - ga + (S)2 * d2;
  if (den == (S)0) return mid;
  S t = b - (b - a) * ((gb + d2 - d1) / den);
  if (!isfinite(t)) return mid;
  const S tlo = lo + (S)0.1 * w;
  const S thi = hi - (S)0.1 * w;
  if (t < tlo) t = tlo;
  if (t > thi) t = thi;
  return t;
}

// ---------------------------------------------------------------------------
// Two-loop recursion by the team's first warp (teams of 1 to 4 warps; float
// history staged through the idle position buffer, FP64 history through the
// idle pair buffer).  The recursion is a chain of 2 cnt + 1 dependent inner products;
// done by the whole team, each one crosses warps through shared memory and a
// barrier.  Instead every thread stages its gradient in `xb` (the idle
// position buffer, 12 A T + 4 bytes), warp 0 runs the recursion over all T
// ranks' entries (lane l covers ranks l, l + 32, ...: the history is
// addressable by rank) with shuffle-only reductions, and stages d and
// g.d back: two team barriers per direction instead of 2 cnt + 1.
//
// Pairs are taken two at a time, so that one two-value reduction serves two
// steps of each loop.  With q the vector before pair t (first loop, newest
// first) the next pair's product follows from this one's:
//   s_{t-1}.(q - alpha_t y_t) = s_{t-1}.q - alpha_t (s_{t-1}.y_t),
// and in the second loop (oldest first), with r before pair t,
//   y_{t+1}.(r + c_t s_t) = y_{t+1}.r + c_t (s_t.y_{t+1}),  c_t = alpha_t - beta_t.
// s_{t-1}.y_t -- the previous pair's s against this pair's y -- is reduced
// when pair t is stored (`sup`).  The same quantities as the one-at-a-time
// recursion (Algorithm 7.4 of Nocedal & Wright), half as many dependent
// reductions.
// ---------------------------------------------------------------------------
template <typename V>
__device__ __forceinline__ V warp_sum(V v) {   // xor butterfly: every lane gets the sum
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

template <typename V>
__device__ __forceinline__ void warp_sum2(V& v0, V& v1) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v0 += __shfl_xor_sync(kFull, v0, o);
    v1 += __shfl_xor_sync(kFull, v1, o);
  }
}

// FP32 vectors lie flat (3 N values, zeros behind them): lane l holds 16 bytes
// of every 512, one vector load and at most four values a lane for LJ38 where
// a lane with the atoms l and l + 32 had six; while a block's products are
// being reduced its other vectors and the next block's are on their way.  1/s.y, s.y/y.y,
// s_{t-1}.y_t and alpha are a register each, slot t's in lane t.
// In isolation (one team, m = 10, N = 38) a direction takes 3.5k cycles: ~290 a
// block of two pairs, 175 of them the two-value reduction, and ~570 once.
// LJ38 Basin Hopping near its minima (64 walkers x 8, 25 steps, mixed): 11.8 ms a
// launch before this form, one evaluation in the line search (run_phase) and the
// ring order of the half pairs, 10.1 after.
// ---------------------------------------------------------------------------
// a lane's part of a vector, of a dot product and of an update: FP32 16 bytes,
// two values an instruction; FP64 one value
template <typename V>
struct HistVec;
template <>
struct HistVec<float> {
  float2 a, b;
  __device__ __forceinline__ void load(const float* p) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    a = make_float2(q.x, q.y);
    b = make_float2(q.z, q.w);
  }
  __device__ __forceinline__ void store(float* p) const {
    *reinterpret_cast<float4*>(p) = make_float4(a.x, a.y, b.x, b.y);
  }
  __device__ __forceinline__ void zero() { a = f2(0.f); b = f2(0.f); }
  __device__ __forceinline__ void scale(float c) { a = __fmul2_rn(a, f2(c)); b = __fmul2_rn(b, f2(c)); }
  __device__ __forceinline__ void add(float c, const HistVec& o) {
    a = __ffma2_rn(f2(c), o.a, a);
    b = __ffma2_rn(f2(c), o.b, b);
  }
};
template <>
struct HistVec<double> {
  double a;
  __device__ __forceinline__ void load(const double* p) { a = *p; }
  __device__ __forceinline__ void store(double* p) const { *p = a; }
  __device__ __forceinline__ void zero() { a = 0.0; }
  __device__ __forceinline__ void scale(double c) { a *= c; }
  __device__ __forceinline__ void add(double c, const HistVec& o) { a = fma(c, o.a, a); }
};
template <int NC>
__device__ __forceinline__ float hist_dot(const HistVec<float> (&x)[NC], const HistVec<float> (&y)[NC]) {
  float2 s = __fmul2_rn(x[0].a, y[0].a);
  s = __ffma2_rn(x[0].b, y[0].b, s);
#pragma unroll
  for (int c = 1; c < NC; ++c) {
    s = __ffma2_rn(x[c].a, y[c].a, s);
    s = __ffma2_rn(x[c].b, y[c].b, s);
  }
  return __fadd_rn(s.x, s.y);
}
template <int NC>
__device__ __forceinline__ double hist_dot(const HistVec<double> (&x)[NC],
                                           const HistVec<double> (&y)[NC]) {
  double s = x[0].a * y[0].a;
#pragma unroll
  for (int c = 1; c < NC; ++c) s = fma(x[c].a, y[c].a, s);
  return s;
}

// 1 / s.y, s.y / y.y and s_prev.y of the stored pairs.  LANES: slot t's in
// lane t of every warp, read by a shuffle (teams whose first warp runs the
// recursion); else in an array of every thread.
template <typename V, bool LANES>
struct PairScalars {
  V rho = (V)0, gam = (V)0, sup = (V)0;
  __device__ __forceinline__ V rho_of(int sl) const { return __shfl_sync(kFull, rho, sl); }
  __device__ __forceinline__ V gam_of(int sl) const { return __shfl_sync(kFull, gam, sl); }
  __device__ __forceinline__ V sup_of(int sl) const { return __shfl_sync(kFull, sup, sl); }
  __device__ __forceinline__ void set(int rank, int sl, V r, V g, V u) {
    if ((rank & 31) == sl) { rho = r; gam = g; sup = u; }
  }
};
template <typename V>
struct PairScalars<V, false> {
  V rho[LJ_MAX_M], gam[LJ_MAX_M];
  __device__ __forceinline__ V rho_of(int sl) const { return rho[sl]; }
  __device__ __forceinline__ V gam_of(int sl) const { return gam[sl]; }
  __device__ __forceinline__ void set(int, int sl, V r, V g, V) { rho[sl] = r; gam[sl] = g; }
};

// the recursion of the lead warp on vectors of NC parts a lane: q (the
// gradient, in xb) to the direction (in xb), returns g.d.  FP32: chunks of 512
// bytes of the flat vector.  FP64: the values of the atom slots (w, a) of a lane, w
// the warp that owns them, in the order of w, a and component -- the order in
// which the products are summed (see tri_pairs on why it matters).
template <int T, int A, int NC, typename V>
__device__ __forceinline__ V lead_recursion(int lane, int m, int cnt, int head,
                                            const V* __restrict__ Sh, const V* __restrict__ Yh,
                                            const PairScalars<V, true>& ps, V* xb) {
  using Vec = HistVec<V>;
  constexpr int L3 = 3 * A * T;              // values of a slot
  constexpr bool FLAT = sizeof(V) == 4;
  auto at = [&](int c) {
    return FLAT ? (c * 32 + lane) * 4 : c % (3 * A) * T + c / (3 * A) * 32 + lane;
  };
  auto in = [&](int c) { return !FLAT || (c + 1) * 128 <= L3 || at(c) < L3; };
  Vec q[NC], d0[NC], d1[NC], u0[NC], u1[NC];
  auto load = [&](const V* base, Vec (&o)[NC]) {
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      if (FLAT && (c + 1) * 128 > L3) o[c].zero();   // not a whole chunk
      if (in(c)) o[c].load(base + at(c));
    }
  };
  // slots of the pairs t (newest: cnt - 1); where there is no such pair, the
  // nearest one, whose factor is then zero: a branch around a shuffle or a
  // load, whose condition the compiler cannot know to be uniform, costs more
  // than reading a pair too many
  auto older = [&](int k, bool is) { return !is ? k : k == 0 ? m - 1 : k - 1; };
  auto newer = [&](int k, bool is) { return !is ? k : k == m - 1 ? 0 : k + 1; };
  load(xb, q);
  V alpha = (V)0;
  // ---- first loop, newest first ----------------------------------------------
  int k0 = head + cnt - 1;
  if (k0 >= m) k0 -= m;
  const V gam = ps.gam_of(k0);
  int k1 = older(k0, cnt >= 2);
  constexpr bool kAhead = NC * sizeof(Vec) <= 48;   // registers for the next block's vectors
  if (kAhead) {
    load(Sh + k0 * L3, d0);
    load(Sh + k1 * L3, d1);
  }
  for (int t = cnt - 1; t >= 0; t -= 2) {
    if (!kAhead) {
      load(Sh + k0 * L3, d0);
      load(Sh + k1 * L3, d1);
    }
    V p0 = hist_dot(d0, q), p1 = hist_dot(d1, q);
    // in flight during the reduction: this block's y, the next block's s
    load(Yh + k0 * L3, u0);
    load(Yh + k1 * L3, u1);
    const V r0 = ps.rho_of(k0), u = ps.sup_of(k0);
    V r1 = ps.rho_of(k1);
    if (t < 1) r1 = (V)0;
    k0 = older(k1, t >= 2);
    k1 = older(k0, t >= 3);
    if (kAhead) {
      load(Sh + k0 * L3, d0);
      load(Sh + k1 * L3, d1);
    }
    warp_sum2(p0, p1);
    const V a0 = r0 * p0;
    const V a1 = r1 * (p1 - a0 * u);
    if (lane == t) alpha = a0;
    if (lane == t - 1) alpha = a1;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      q[c].add(-a0, u0[c]);
      q[c].add(-a1, u1[c]);
    }
  }
#pragma unroll
  for (int c = 0; c < NC; ++c) q[c].scale(gam);
  // ---- second loop, oldest first ----------------------------------------------
  k0 = head;
  k1 = newer(k0, cnt >= 2);
  if (kAhead) {
    load(Yh + k0 * L3, d0);
    load(Yh + k1 * L3, d1);
  }
  for (int t = 0; t < cnt; t += 2) {
    if (!kAhead) {
      load(Yh + k0 * L3, d0);
      load(Yh + k1 * L3, d1);
    }
    V p0 = hist_dot(d0, q), p1 = hist_dot(d1, q);
    load(Sh + k0 * L3, u0);
    load(Sh + k1 * L3, u1);
    const V r0 = ps.rho_of(k0), r1 = ps.rho_of(k1), u = ps.sup_of(k1);
    const V al0 = __shfl_sync(kFull, alpha, t), al1 = __shfl_sync(kFull, alpha, (t + 1) & 31);
    k0 = newer(k1, t + 2 < cnt);
    k1 = newer(k0, t + 3 < cnt);
    if (kAhead) {
      load(Yh + k0 * L3, d0);
      load(Yh + k1 * L3, d1);
    }
    warp_sum2(p0, p1);
    const V c0 = al0 - r0 * p0;
    V c1 = al1 - r1 * (p1 + c0 * u);
    if (t + 1 >= cnt) c1 = (V)0;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      q[c].add(c0, u0[c]);
      q[c].add(c1, u1[c]);
    }
  }
  load(xb, d0);
  const V dphi = -warp_sum(hist_dot(d0, q));
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    q[c].scale((V)-1);
    if (in(c)) q[c].store(xb + at(c));
  }
  return dphi;
}

template <int T, int A, typename XG, typename V>
__device__ __forceinline__ V lead_two_loop(const Team<T>& tm, int n, int m, int cnt, int head,
                                           const V* __restrict__ Sh, const V* __restrict__ Yh,
                                           const PairScalars<V, true>& ps, const XG (&g)[A][3],
                                           V* xb, V (&d)[A][3]) {
  constexpr int L3 = 3 * A * T;               // values of a slot
#pragma unroll
  for (int a = 0; a < A; ++a)
#pragma unroll
    for (int c = 0; c < 3; ++c) xb[hidx<T, A, V>(0, a, c, tm.rank)] = (V)g[a][c];
  tm.sync();
  if (tm.rank < 32) {
    V dphi;
    if constexpr (sizeof(V) == 4) {
      // clusters that leave the last third or more of the chunks empty: fewer
      constexpr int NC = (L3 + 127) / 128, ND = NC > 2 ? NC * 2 / 3 : 1;
      const bool few = NC > 1 && 3 * n <= ND * 128;
      dphi = few ? lead_recursion<T, A, ND, V>(tm.rank, m, cnt, head, Sh, Yh, ps, xb)
                 : lead_recursion<T, A, NC, V>(tm.rank, m, cnt, head, Sh, Yh, ps, xb);
      if (few)                                // zeros behind the chunks that were taken
        for (int f = ND * 128 + tm.rank; f < L3; f += 32) xb[f] = (V)0;
    } else {
      dphi = lead_recursion<T, A, L3 / 32, V>(tm.rank, m, cnt, head, Sh, Yh, ps, xb);
    }
    if (tm.rank == 0) xb[L3] = dphi;
  }
  tm.sync();
#pragma unroll
  for (int a = 0; a < A; ++a)
#pragma unroll
    for (int c = 0; c < 3; ++c) d[a][c] = xb[hidx<T, A, V>(0, a, c, tm.rank)];
  return xb[L3];
}

// ---------------------------------------------------------------------------
// One L-BFGS phase: iterate from (x, g, f) until a stop condition.
// X: coordinates/gradient precision, V: direction/history precision,
// PM: pair arithmetic (0 native X, 1 double-float).
// MODE 0 (FP64, final): stops on ||g||_inf < gtol (CONVERGED) or a failed
//   line search (LSFAIL).
// MODE 1 (mixed, FP32 phase): hands over (SWITCH) once ||g||_inf <
//   switch_gtol or when a line search fails; never converges.  Once the
//   predicted decrease -alpha phi'(0) is below f32_resolution |E| (default 4
//   FP32 ulps) its line searches accept steps on the gradient alone.
// MODE 2 (mixed, double-float polish): CONVERGED on ||g||_inf < gtol (to be
//   confirmed in FP64); once the predicted decrease is below df_resolution
//   |E| (default 32 * 2^-48) its line searches accept steps on the gradient
//   alone (approximate Wolfe conditions); hands over to FP64 when a line
//   search fails.
// In MODE 1, gradient-only steps past kFP32GradIters tier iterations also
// hand over (a switch_gtol below the FP32 gradient noise).
// ---------------------------------------------------------------------------
template <int T, int A, typename P, int MODE>
__device__ __forceinline__ int run_phase(const Team<T>& tm, int n, typename P::XP (&x)[A][3],
                         typename P::XG (&g)[A][3], typename P::F& f,
                         typename P::V* __restrict__ Sh, typename P::V* __restrict__ Yh,
                         PairScalars<typename P::V, (T <= 128)>& ps, int& cnt, int& head, int& iters,
                         int& evals, int& phase_iters, long long& vec, void* pos,
                         void* hbuf, const MinParams& p, long long t0, long long (&cyc)[2]) {
  using X = typename P::XP;
  using XG = typename P::XG;
  using V = typename P::V;
  using S = typename P::S;
  using F = typename P::F;
  const int m = p.m;
  const S c1 = (S)p.c1, c2 = (S)p.c2, amax = (S)p.alpha_max;
  const S resolution = (S)(MODE == 1 ? p.f32_resolution : p.df_resolution);
  const XG stop_gtol = MODE == 1 ? (XG)p.switch_gtol : (XG)p.gtol;
  V d[A][3];
  bool gmode = false;   // MODE 1, 2: energy below resolution, gradient-only line search
  X xt[A][3];
  XG gt[A][3];
  while (iters < p.max_iter) {
    // ---- search direction -------------------------------------------------
    long long tc = clock64();
    S dphi0 = (S)1;
    bool led = false;
    if constexpr (T <= 128) {
      // staging buffer for the lead warp: the idle position buffer (32 n
      // bytes) for float history, the idle pair buffer (half pairs: 24 bytes per
      // pair) for double history
      V* xb = nullptr;
      if constexpr (std::is_same<V, float>::value) {
        if (12 * A * T + 4 <= 32 * n) xb = static_cast<V*>(pos);
      } else {
        if (hbuf != nullptr && p.layout == LAYOUT_HALF && 24 * A * T + 8 <= 24 * n_pairs(n))
          xb = static_cast<V*>(hbuf);
      }
      if (cnt > 0 && xb != nullptr) {
        dphi0 = (S)lead_two_loop<T, A, XG, V>(tm, n, m, cnt, head, Sh, Yh, ps, g, xb, d);
        vec += (long long)cnt * 3 * n;
        led = true;
      }
    }
    if (cnt > 0 && !led) {
      V q[A][3];
#pragma unroll
      for (int a = 0; a < A; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c) q[a][c] = (V)g[a][c];
      // two-loop recursion; each step prefetches the next pair's vectors and
      // 1/s.y before its own team reduction, so loads overlap the reduction
      auto slot_of = [&](int t) { const int sl = head + t; return sl >= m ? sl - m : sl; };
      V alpha[LJ_MAX_M];
      V sc[A][3], yc[A][3], sn[A][3], yn[A][3];
      {
        const int sl = slot_of(cnt - 1);
#pragma unroll
        for (int a = 0; a < A; ++a)
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            sc[a][c] = Sh[hidx<T, A, V>(sl, a, c, tm.rank)];
            yc[a][c] = Yh[hidx<T, A, V>(sl, a, c, tm.rank)];
          }
      }
      V rho_c = ps.rho_of(slot_of(cnt - 1));
      for (int t = cnt - 1; t >= 0; --t) {
        const int nsl = slot_of(t > 0 ? t - 1 : 0);
#pragma unroll
        for (int a = 0; a < A; ++a)
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            sn[a][c] = Sh[hidx<T, A, V>(nsl, a, c, tm.rank)];
            yn[a][c] = Yh[hidx<T, A, V>(nsl, a, c, tm.rank)];
          }
        const V rho_n = ps.rho_of(nsl);
        V part = (V)0;
#pragma unroll
        for (int a = 0; a < A; ++a)
#pragma unroll
          for (int c = 0; c < 3; ++c) part += sc[a][c] * q[a][c];
        const V al = rho_c * team_sum1<T, V>(tm, part);
        alpha[t] = al;
#pragma unroll
        for (int a = 0; a < A; ++a)
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            q[a][c] -= al * yc[a][c];
            sc[a][c] = sn[a][c];
            yc[a][c] = yn[a][c];
          }
        rho_c = rho_n;
      }
      const int newest = slot_of(cnt - 1);
      const V gam = ps.gam_of(newest);
#pragma unroll
      for (int a = 0; a < A; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c) q[a][c] *= gam;
      // (sc, yc) now hold the oldest pair, the first one of the second loop
      rho_c = ps.rho_of(slot_of(0));
      for (int t = 0; t < cnt; ++t) {
        const int nsl = slot_of(t + 1 < cnt ? t + 1 : t);
#pragma unroll
        for (int a = 0; a < A; ++a)
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            sn[a][c] = Sh[hidx<T, A, V>(nsl, a, c, tm.rank)];
            yn[a][c] = Yh[hidx<T, A, V>(nsl, a, c, tm.rank)];
          }
        const V rho_n = ps.rho_of(nsl);
        V part = (V)0;
#pragma unroll
        for (int a = 0; a < A; ++a)
#pragma unroll
          for (int c = 0; c < 3; ++c) part += yc[a][c] * q[a][c];
        const V coef = alpha[t] - rho_c * team_sum1<T, V>(tm, part);
#pragma unroll
        for (int a = 0; a < A; ++a)
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            q[a][c] += coef * sc[a][c];
            sc[a][c] = sn[a][c];
            yc[a][c] = yn[a][c];
          }
        rho_c = rho_n;
      }
      V part = (V)0;
#pragma unroll
      for (int a = 0; a < A; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          d[a][c] = -q[a][c];
          part += (V)g[a][c] * d[a][c];
        }
      dphi0 = (S)team_sum1<T, V>(tm, part);
      vec += (long long)cnt * 3 * n;
    }
    if (!(dphi0 < (S)0)) {  // empty history or not a descent direction
      cnt = 0;
      head = 0;
      V part = (V)0;
#pragma unroll
      for (int a = 0; a < A; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          d[a][c] = -(V)g[a][c];
          part += d[a][c] * d[a][c];
        }
      dphi0 = -(S)team_sum1<T, V>(tm, part);
    }
    bool ok = false;
    F ft;
    {
      const long long t1 = clock64();
      cyc[0] += t1 - tc;
      tc = t1;
    }
    for (int attempt = 0; attempt < 2 && !ok; ++attempt) {
      if (attempt == 1) {
        if (cnt == 0) break;  // already steepest descent: no retry
        cnt = 0;
        head = 0;
        V part = (V)0;
#pragma unroll
        for (int a = 0; a < A; ++a)
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            d[a][c] = -(V)g[a][c];
            part += d[a][c] * d[a][c];
          }
        dphi0 = -(S)team_sum1<T, V>(tm, part);
      }
      S a1 = (S)1;
      if (cnt == 0) {
        a1 = (S)1 / S_sqrt(-dphi0);
        if (a1 > (S)1) a1 = (S)1;
      }
      if constexpr (MODE == 1 || MODE == 2) {
        // predicted decrease below this tier's energy resolution: from here
        // on, steps are accepted on the gradient instead (the FP32 gradient
        // is trusted down to switch_gtol, the double-float one to ~1e-11)
        if (-dphi0 * a1 < resolution * fabsf(f.hi)) gmode = true;
      }
      // ---- line search --------------------------------------------------------
      // One loop with one evaluation in it: its four kinds of trial (bracketing
      // and zoom of the strong-Wolfe search, the gradient-only search, and the
      // best point once more when the budget is spent) share the code of the
      // evaluation, which inlined at each of them filled the instruction cache.
      enum { BRACKET, ZOOM, GRAD, LAST };
      int kind = BRACKET, ev = 0;
      S a_prev = (S)0, dp_prev = dphi0;
      F f_prev = f;
      S a = a1;
      bool have_best = false;
      S best_a = (S)0, last_a = (S)-1;
      F best_f = f;
      S lo = 0, hi = 0, dp_lo = 0, dp_hi = 0;
      F f_lo = f, f_hi = f;
      bool done = false;
      // gradient-only search (approximate Wolfe conditions, Hager and Zhang
      // 2005): accept |phi'(a)| <= c2 |phi'(0)| with the energy no more than
      // the resolution above f(0) (which, for a near-quadratic phi, also
      // implies the Armijo decrease); bracket on the sign of phi' and
      // interpolate by secant steps on phi'.  lo, dp_lo: the last point too
      // short; hi, dp_hi: the first too long (hi < 0: none)
      S tol_f = (S)0;
      bool hi_slope = false;
      if constexpr (MODE == 1 || MODE == 2) {
        if (gmode) {
          kind = GRAD;
          tol_f = (S)2 * resolution * fabsf(f.hi);
          hi = (S)-1;
          dp_lo = dphi0;
        }
      }
      for (int i = 1;; ++i) {
        if (ev >= p.max_ls) {
          // out of budget: the best point with sufficient decrease, if it is lower
          if (kind == GRAD || !have_best || !((S)fdiff(best_f, f) < (S)0)) break;
          if (last_a == best_a) {
            ft = best_f;
            done = true;
            break;
          }
          kind = LAST;
          a = best_a;
        }
        F fa;
        S dp;
#pragma unroll
        for (int aa = 0; aa < A; ++aa)
#pragma unroll
          for (int c = 0; c < 3; ++c) xt[aa][c] = pos_step(x[aa][c], a, d[aa][c]);
        evaluate<T, A, P>(tm, n, xt, gt, pos, hbuf, p, d, fa, dp);
        ++ev;
        last_a = a;
        if (kind == LAST) {
          ft = fa;
          done = true;
          break;
        }
        if constexpr (MODE == 1 || MODE == 2) {
          if (kind == GRAD) {
            const bool eok = fisfinite(fa) && isfinite(dp) && (S)fdiff(fa, f) <= tol_f;
            if (!eok || dp > -c2 * dphi0) {          // too long
              hi = a; dp_hi = dp; hi_slope = eok;
            } else if (dp < c2 * dphi0) {            // too short
              lo = a; dp_lo = dp;
            } else {
              ft = fa;
              done = true;
              break;
            }
            if (hi < (S)0) {
              a = (S)2 * a;
              if (a > amax) a = amax;
            } else {
              const S w = hi - lo;
              S t = (hi_slope && dp_hi > dp_lo) ? lo - dp_lo * w / (dp_hi - dp_lo)
                                                : lo + (S)0.5 * w;
              const S tlo = lo + (S)0.1 * w, thi = hi - (S)0.1 * w;
              if (!(t >= tlo)) t = tlo;
              if (!(t <= thi)) t = thi;
              a = t;
            }
            continue;
          }
        }
        const bool armijo = armijo_ok(fa, f, c1 * a * dphi0);
        if (armijo && (!have_best || (S)fdiff(fa, best_f) < (S)0)) {
          have_best = true; best_f = fa; best_a = a;
        }
        if (kind == BRACKET) {
          if (!armijo || (i > 1 && (S)fdiff(fa, f_prev) >= (S)0)) {
            lo = a_prev; f_lo = f_prev; dp_lo = dp_prev;
            hi = a; f_hi = fa; dp_hi = dp;
            kind = ZOOM;
          } else if (fabs(dp) <= -c2 * dphi0) {
            ft = fa;
            done = true;
            break;
          } else if (dp >= (S)0) {
            lo = a; f_lo = fa; dp_lo = dp;
            hi = a_prev; f_hi = f_prev; dp_hi = dp_prev;
            kind = ZOOM;
          } else {
            a_prev = a; f_prev = fa; dp_prev = dp;
            a = (S)2 * a;
            if (a > amax) a = amax;
            continue;
          }
        } else if (!armijo || (S)fdiff(fa, f_lo) >= (S)0) {
          hi = a; f_hi = fa; dp_hi = dp;
        } else {
          if (fabs(dp) <= -c2 * dphi0) {
            ft = fa;
            done = true;
            break;
          }
          if (dp * (hi - lo) >= (S)0) {
            hi = lo; f_hi = f_lo; dp_hi = dp_lo;
          }
          lo = a; f_lo = fa; dp_lo = dp;
        }
        a = cubic_step<S, F>(lo, f_lo, dp_lo, hi, f_hi, dp_hi);
      }
      evals += ev;
      ok = done;
    }
    cyc[1] += clock64() - tc;
    if (!ok) return MODE == 0 ? PH_LSFAIL : PH_SWITCH;

    // ---- curvature pair, then move ------------------------------------------
    V sv[A][3], yv[A][3];
    // s.y, y.y and s_prev.y (the newest stored pair's s against the new y:
    // the superdiagonal entry the blocked two-loop recursion uses)
    V pr[3] = {(V)0, (V)0, (V)0};
    const int prev = cnt > 0 ? (head + cnt - 1 >= m ? head + cnt - 1 - m : head + cnt - 1) : -1;
#pragma unroll
    for (int a = 0; a < A; ++a)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        sv[a][c] = pos_diff<V>(xt[a][c], x[a][c]);
        yv[a][c] = (V)(gt[a][c] - g[a][c]);
        pr[0] += sv[a][c] * yv[a][c];
        pr[1] += yv[a][c] * yv[a][c];
        if (prev >= 0) pr[2] += Sh[hidx<T, A, V>(prev, a, c, tm.rank)] * yv[a][c];
      }
    // stopping-test values of the new point (||g||_inf, deadline), reduced
    // in the same pass as the curvature pair's s.y and y.y
    auto gmax = max_bits(gt);
    bool late = p.deadline > 0 && (clock64() - t0) > p.deadline;
    team_sums_max(tm, pr, gmax, late);
    if (pr[0] > eps_mach<V>() * pr[1]) {
      int slot;
      if (cnt < m) {
        slot = head + cnt;
        if (slot >= m) slot -= m;
        ++cnt;
      } else {
        slot = head;
        head = head + 1 == m ? 0 : head + 1;
      }
#pragma unroll
      for (int a = 0; a < A; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          Sh[hidx<T, A, V>(slot, a, c, tm.rank)] = sv[a][c];
          Yh[hidx<T, A, V>(slot, a, c, tm.rank)] = yv[a][c];
        }
      // 1 / s.y and the scaling s.y / y.y, formed once here instead of in every
      // recursion step; s_prev . y (undefined for the oldest pair: unused)
      ps.set(tm.rank, slot, (V)1 / pr[0], pr[0] / pr[1], pr[2]);
    }
#pragma unroll
    for (int a = 0; a < A; ++a)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        x[a][c] = xt[a][c];
        g[a][c] = gt[a][c];
      }
    f = ft;
    ++iters;
    ++phase_iters;
    // ---- stopping tests (values reduced above) -----------------------------
    if (from_bits(gmax) < stop_gtol) return MODE == 1 ? PH_SWITCH : PH_CONVERGED;
    if (late) return PH_TIMEOUT;
    if constexpr (MODE == 1) {
      // a switch_gtol below the FP32 gradient noise would keep gradient-only
      // FP32 steps iterating on noise: past kFP32GradIters iterations of the
      // tier the double-float tier takes over
      if (gmode && phase_iters >= kFP32GradIters) return PH_SWITCH;
    }
  }
  return PH_MAXITER;
}

// ---------------------------------------------------------------------------
// Minimise the cluster whose owned coordinates are in x64 (in place).
// hist: this team's history slot (2 m A 3 T values of the phase's V type).
// pos:  this team's shared position buffer (n entries of 32 bytes).
// hbuf: this team's pair buffer (see evaluate) or nullptr.
// MIXED: FP32 phase, then polish iterations whose evaluations run in
// double-float arithmetic; convergence is confirmed, and the returned energy
// computed, by a true FP64 evaluation (if FP64 disagrees, polishing goes on).
// ---------------------------------------------------------------------------
__device__ __forceinline__ int status_of(int code) {
  return code == PH_CONVERGED ? ST_CONVERGED
       : code == PH_LSFAIL   ? ST_LS_FAIL
       : code == PH_TIMEOUT  ? ST_TIMEOUT : ST_MAXITER;
}

template <int T, int A, bool MIXED, int POT = LJ_POT_LJ>
__device__ __forceinline__ void minimise(const Team<T>& tm, int n, double (&x64)[A][3], const MinParams& p,
                         void* hist, void* pos, void* hbuf, MinResult& r) {
  using P32 = Prec<float, float, float, 0, POT>;       // mixed: FP32 tier
  using PDF = Prec<ff, float, float, 1, POT>;          // mixed: double-float tier
  using P64m = Prec<double, double, float, 0, POT>;    // mixed: FP64 tier
  using P64 = Prec<double, double, double, 0, POT>;    // FP64 path
  r.E = 0.0; r.status = ST_CONVERGED; r.iters = 0;
  r.evals32 = 0; r.evals64 = 0; r.evals_df = 0; r.iters32 = 0; r.iters64 = 0;
  r.vec32 = 0; r.vec64 = 0;
  r.cyc32 = 0; r.cycdf = 0; r.cyc64 = 0; r.cycdir = 0; r.cycls = 0;
  long long cyc[2] = {0, 0};
  if (n <= 1) return;
  const long long t0 = clock64();
  long long tmark = t0;
  auto lap = [&](long long& acc) {
    const long long t = clock64();
    acc += t - tmark;
    tmark = t;
    r.cycdir = cyc[0];
    r.cycls = cyc[1];
  };
  int cnt = 0, head = 0, iters = 0;
  const size_t hstride = (size_t)p.m * A * 3 * T;
  const double kInf = __longlong_as_double(0x7ff0000000000000LL);
  if constexpr (!MIXED) {
    double g[A][3];
    double f, dummy;
    evaluate<T, A, P64>(tm, n, x64, g, pos, hbuf, p, nullptr, f, dummy);
    r.evals64 = 1;
    const double gm = grad_max<T, A, double>(tm, g);
    if (!isfinite(f) || !(gm < kInf)) {
      r.E = f; r.status = ST_NONFINITE; lap(r.cyc64); return;
    }
    if (gm < p.gtol) { r.E = f; lap(r.cyc64); return; }
    PairScalars<double, (T <= 128)> ps;
    double* Sh = (double*)hist;
    const int code = run_phase<T, A, P64, 0>(tm, n, x64, g, f, Sh, Sh + hstride, ps, cnt,
                                                 head, iters, r.evals64, r.iters64, r.vec64, pos,
                                                 hbuf, p, t0, cyc);
    r.E = f;
    r.iters = iters;
    r.status = status_of(code);
    lap(r.cyc64);
  } else {
    float* Sh = (float*)hist;
    float* Yh = Sh + hstride;
    PairScalars<float, (T <= 128)> ps;
    int code = PH_SWITCH;
    float dummy32;
    // ---- tier 1: FP32 -------------------------------------------------------
    float x32[A][3];
    bool moved32 = false;
    {
      float g32[A][3];
#pragma unroll
      for (int a = 0; a < A; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c) x32[a][c] = (float)x64[a][c];
      ff f32;
      evaluate<T, A, P32>(tm, n, x32, g32, pos, nullptr, p, nullptr, f32, dummy32);
      r.evals32 = 1;
      const float gm = grad_max<T, A, float>(tm, g32);
      if (fisfinite(f32) && gm < __int_as_float(0x7f800000) && !(gm < (float)p.switch_gtol)) {
        code = run_phase<T, A, P32, 1>(tm, n, x32, g32, f32, Sh, Yh, ps, cnt, head,
                                           iters, r.evals32, r.iters32, r.vec32, pos, nullptr, p,
                                           t0, cyc);
        moved32 = r.iters32 > 0;
      }
    }
    lap(r.cyc32);
    int status = -1;
    bool need_fp64 = false;
    if (code == PH_MAXITER || code == PH_TIMEOUT) {
      status = status_of(code);
      if (moved32) {
#pragma unroll
        for (int a = 0; a < A; ++a)
#pragma unroll
          for (int c = 0; c < 3; ++c) x64[a][c] = (double)x32[a][c];
      }
    } else {
      // ---- tier 2: double-float positions and pair terms, FP32 elsewhere -----
      ff xdf[A][3];
      float gdf[A][3];
#pragma unroll
      for (int a = 0; a < A; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c)
          xdf[a][c] = moved32 ? ff{x32[a][c], 0.f} : df_from_double(x64[a][c]);
      ff fdf;
      evaluate<T, A, PDF>(tm, n, xdf, gdf, pos, hbuf, p, nullptr, fdf, dummy32);
      r.evals_df += 1;
      float gm = grad_max<T, A, float>(tm, gdf);
      if (!fisfinite(fdf) || !(gm < __int_as_float(0x7f800000))) need_fp64 = true;
      while (status < 0 && !need_fp64) {
        if (gm < (float)p.gtol) {
          need_fp64 = true;               // confirm (and finish) in FP64
          break;
        }
        code = run_phase<T, A, PDF, 2>(tm, n, xdf, gdf, fdf, Sh, Yh, ps, cnt, head, iters,
                                          r.evals_df, r.iters64, r.vec64, pos, hbuf, p, t0, cyc);
        if (code == PH_CONVERGED) {
          gm = 0.f;
        } else if (code == PH_SWITCH) {
          need_fp64 = true;
        } else {
          status = status_of(code);
        }
      }
#pragma unroll
      for (int a = 0; a < A; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c) x64[a][c] = (double)xdf[a][c].hi + (double)xdf[a][c].lo;
    }
    lap(r.cycdf);
    double g[A][3];
    double f, dummy;
    if (need_fp64) {
      // ---- tier 3: FP64 -------------------------------------------------------
      evaluate<T, A, P64m>(tm, n, x64, g, pos, hbuf, p, nullptr, f, dummy32);
      r.evals64 += 1;
      const double gm = grad_max<T, A, double>(tm, g);
      if (!isfinite(f) || !(gm < kInf)) {
        r.E = f; r.iters = iters; r.status = ST_NONFINITE; lap(r.cyc64); return;
      }
      if (gm < p.gtol) {
        r.E = f; r.iters = iters; r.status = ST_CONVERGED; lap(r.cyc64); return;
      }
      code = run_phase<T, A, P64m, 0>(tm, n, x64, g, f, Sh, Yh, ps, cnt, head, iters,
                                          r.evals64, r.iters64, r.vec64, pos, hbuf, p, t0, cyc);
      r.E = f;
      r.iters = iters;
      r.status = status_of(code);
      lap(r.cyc64);
      return;
    }
    // final energy (and the non-finite test) in FP64
    evaluate<T, A, P64>(tm, n, x64, g, pos, hbuf, p, nullptr, f, dummy);
    r.evals64 += 1;
    const double gm = grad_max<T, A, double>(tm, g);
    r.E = f;
    r.iters = iters;
    if (!isfinite(f) || !(gm < kInf)) {
      r.status = ST_NONFINITE;
    } else if (gm < p.gtol) {
      r.status = ST_CONVERGED;
    } else {
      r.status = status;
    }
    lap(r.cyc64);
  }
}

}  // namespace ljd
