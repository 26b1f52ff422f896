// lj_device.cuh -- sm_103a device building blocks: teams, team reductions,
// Philox4x32-10, float-float energies and the Eq. (1) pair loops.
//
// A "team" is the group of T threads that owns one candidate cluster:
// one warp (T = 32) or a multiple of 32 threads synchronised by a named
// barrier.  Thread `rank` of a team owns atoms rank, rank + T, ... (A slots)
// and exactly the 3 coordinates / gradient components of those atoms, so
// every vector operation of L-BFGS is thread-local and only the pair loop
// reads other threads' atoms (from shared memory).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace ljd {

constexpr unsigned kFull = 0xffffffffu;

enum : int32_t {
  ST_CONVERGED = 0, ST_MAXITER = 1, ST_LS_FAIL = 2, ST_NONFINITE = 3, ST_TIMEOUT = 4,
  ST_BAD_INPUT = 5
};

// ---------------------------------------------------------------------------
// Team
// ---------------------------------------------------------------------------
template <int T>
struct Team {
  static_assert(T % 32 == 0 && T >= 32 && T <= 1024, "team size");
  int rank;       // 0 .. T-1
  int bar;        // named barrier id (T > 32); 1..15
  double* red;    // shared scratch for cross-warp reductions: 2 x 8 x (T/32) doubles
  mutable int flip = 0;   // which half of `red` the next reduction uses
  __device__ __forceinline__ void sync() const {
    if constexpr (T == 32) {
      __syncwarp();
    } else {
      asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(T) : "memory");
    }
  }
  // Scratch half for the next cross-warp reduction.  Alternating halves
  // makes a barrier before the write unnecessary: a thread can only reach
  // the reduction after next (same half) once every thread has passed the
  // next reduction's barrier, i.e. has finished reading this one.
  __device__ __forceinline__ double* scratch() const {
    double* b = red + (flip ? 8 * (T / 32) : 0);
    flip ^= 1;
    return b;
  }
};

template <typename V>
__device__ __forceinline__ V shfl_xor(V v, int o) { return __shfl_xor_sync(kFull, v, o); }

// Sum of NV values over the team; every thread receives the same bits
// (xor butterfly: partners add the same operands; the cross-warp stage sums
// the per-warp results in the same order on every thread).
template <int T, int NV, typename V>
__device__ __forceinline__ void team_sum(const Team<T>& tm, V (&v)[NV]) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] += shfl_xor(v[k], o);
  }
  if constexpr (T > 32) {
    static_assert(NV * sizeof(V) <= 8 * sizeof(double), "reduction scratch");
    constexpr int NW = T / 32;
    V* buf = reinterpret_cast<V*>(tm.scratch());
    if ((tm.rank & 31) == 0) {
#pragma unroll
      for (int k = 0; k < NV; ++k) buf[(tm.rank >> 5) * NV + k] = v[k];
    }
    tm.sync();
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      V s = buf[k];
#pragma unroll
      for (int w = 1; w < NW; ++w) s += buf[w * NV + k];
      v[k] = s;
    }
  }
}

template <int T, typename V>
__device__ __forceinline__ V team_sum1(const Team<T>& tm, V x) {
  V v[1] = {x};
  team_sum<T, 1, V>(tm, v);
  return v[0];
}

// ---------------------------------------------------------------------------
// Float-float energy values (FP32 phase): hi + lo, |lo| <= ulp(hi)/2.
// The FP32 phase keeps its energies in this form so that the line search can
// form energy differences without any FP64 instruction.
// ---------------------------------------------------------------------------
struct ff {
  float hi, lo;
};

__device__ __forceinline__ ff ff_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return ff{s, e};
}
__device__ __forceinline__ ff ff_add(ff a, ff b) {
  ff s = ff_two_sum(a.hi, b.hi);
  const float lo = __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo));
  return ff_two_sum(s.hi, lo);
}
__device__ __forceinline__ ff ff_add_f(ff a, float b) {
  ff s = ff_two_sum(a.hi, b);
  return ff_two_sum(s.hi, __fadd_rn(s.lo, a.lo));
}
// a c for a float-float a and an FP32 constant c: the high product exact by
// TwoProd (FMA), the low word's product and that error added, renormalised;
// ~2^-47 relative for any c (for a power of two it is the exact product)
__device__ __forceinline__ ff ff_scale(ff a, float c) {
  const float p = __fmul_rn(a.hi, c);
  const float lo = fmaf(a.lo, c, fmaf(a.hi, c, -p));
  const float s = __fadd_rn(p, lo);
  return ff{s, __fsub_rn(lo, __fsub_rn(s, p))};
}

// energy-value traits: difference, finiteness, conversion
__device__ __forceinline__ float fdiff(ff a, ff b) {
  return __fadd_rn(__fsub_rn(a.hi, b.hi), __fsub_rn(a.lo, b.lo));
}
__device__ __forceinline__ double fdiff(double a, double b) { return a - b; }
__device__ __forceinline__ bool fisfinite(ff a) { return isfinite(a.hi); }
__device__ __forceinline__ bool fisfinite(double a) { return isfinite(a); }
__device__ __forceinline__ double fto_double(ff a) { return (double)a.hi + (double)a.lo; }
__device__ __forceinline__ double fto_double(double a) { return a; }

// s += v for a running double-float sum: TwoSum of the high words, every
// rounding error and low word gathered in s.lo (Ogita, Rump and Oishi 2005,
// Sum2); the chain of the high words is one addition a term.  s.lo is
// renormalised where the sum is stored or scaled.
__device__ __forceinline__ void df_acc(ff& s, ff v) {
  const ff t = ff_two_sum(s.hi, v.hi);
  s.hi = t.hi;
  s.lo = __fadd_rn(s.lo, __fadd_rn(t.lo, v.lo));
}

template <int T>
__device__ __forceinline__ ff team_sum_ff(const Team<T>& tm, ff v) {
  // both partners of a butterfly step form the same sums: TwoSum's results
  // and (v.lo + w.lo) do not depend on the order of the operands.  Every step
  // renormalises: the threads' low words, gathered over hundreds of pairs, are
  // far above an ulp of the high ones, and plain FP32 sums of them round by
  // about as much as the line search resolves (Morse, 400 atoms: 9 of 1,500
  // quenches failed their last line search).
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = ff_add(v, ff{shfl_xor(v.hi, o), shfl_xor(v.lo, o)});
  if constexpr (T > 32) {
    constexpr int NW = T / 32;
    float* buf = reinterpret_cast<float*>(tm.scratch());
    if ((tm.rank & 31) == 0) {
      buf[2 * (tm.rank >> 5)] = v.hi;
      buf[2 * (tm.rank >> 5) + 1] = v.lo;
    }
    tm.sync();
    ff s{buf[0], buf[1]};
#pragma unroll
    for (int w = 1; w < NW; ++w) s = ff_add(s, ff{buf[2 * w], buf[2 * w + 1]});
    v = s;
  }
  return v;
}

// Maximum of bit patterns over the team (bits of non-negative floats order as
// integers): one or two REDUX instead of five shuffles with floating-point
// maxima, which for FP64 each take the FP64 unit.
__device__ __forceinline__ unsigned warp_max_bits(unsigned m) {
  return __reduce_max_sync(kFull, m);
}
__device__ __forceinline__ unsigned long long warp_max_bits(unsigned long long m) {
  const unsigned hi = (unsigned)(m >> 32);
  const unsigned mh = __reduce_max_sync(kFull, hi);
  const unsigned ml = __reduce_max_sync(kFull, hi == mh ? (unsigned)m : 0u);
  return ((unsigned long long)mh << 32) | ml;
}
template <int T, typename B>
__device__ __forceinline__ B team_max_bits(const Team<T>& tm, B m) {
  m = warp_max_bits(m);
  if constexpr (T > 32) {
    constexpr int NW = T / 32;
    B* buf = reinterpret_cast<B*>(tm.scratch());
    if ((tm.rank & 31) == 0) buf[tm.rank >> 5] = m;
    tm.sync();
    m = buf[0];
#pragma unroll
    for (int w = 1; w < NW; ++w) m = max(m, buf[w]);
  }
  return m;
}

// team_sum of s[0..NS-1], the maximum of the bit patterns m and the
// disjunction of f in one pass, one cross-warp exchange
template <int T, typename V, typename B, int NS>
__device__ __forceinline__ void team_sums_max(const Team<T>& tm, V (&s)[NS], B& m, bool& f) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int k = 0; k < NS; ++k) s[k] += shfl_xor(s[k], o);
  }
  m = warp_max_bits(m);
  f = __any_sync(kFull, f);
  if constexpr (T > 32) {
    constexpr int NW = T / 32;
    static_assert((NS + 1) * sizeof(V) + sizeof(B) + 8 <= 8 * sizeof(double), "reduction scratch");
    double* raw = tm.scratch();
    B* bm = reinterpret_cast<B*>(raw);
    unsigned* bf = reinterpret_cast<unsigned*>(raw + NW);
    V* bs = reinterpret_cast<V*>(raw + 2 * NW);
    if ((tm.rank & 31) == 0) {
#pragma unroll
      for (int k = 0; k < NS; ++k) bs[(tm.rank >> 5) * NS + k] = s[k];
      bm[tm.rank >> 5] = m;
      bf[tm.rank >> 5] = f;
    }
    tm.sync();
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      V a = bs[k];
#pragma unroll
      for (int w = 1; w < NW; ++w) a += bs[w * NS + k];
      s[k] = a;
    }
    m = bm[0];
    unsigned any = bf[0];
#pragma unroll
    for (int w = 1; w < NW; ++w) {
      m = max(m, bm[w]);
      any |= bf[w];
    }
    f = any != 0;
  }
}

// team_sum_ff of e and team_sum of x in one pass (one cross-warp exchange):
// each value gets exactly the operations, in the order, of its own reduction
template <int T>
__device__ __forceinline__ void team_sum_ff_f(const Team<T>& tm, ff& e, float& x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const ff w{shfl_xor(e.hi, o), shfl_xor(e.lo, o)};
    x += shfl_xor(x, o);
    e = ff_add(e, w);
  }
  if constexpr (T > 32) {
    constexpr int NW = T / 32;
    float* buf = reinterpret_cast<float*>(tm.scratch());
    if ((tm.rank & 31) == 0) {
      buf[3 * (tm.rank >> 5)] = e.hi;
      buf[3 * (tm.rank >> 5) + 1] = e.lo;
      buf[3 * (tm.rank >> 5) + 2] = x;
    }
    tm.sync();
    ff s{buf[0], buf[1]};
    float t = buf[2];
#pragma unroll
    for (int w = 1; w < NW; ++w) {
      s = ff_add(s, ff{buf[3 * w], buf[3 * w + 1]});
      t += buf[3 * w + 2];
    }
    e = s;
    x = t;
  }
}

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11), from the published round
// function and key schedule, and the 53-bit uniform built from two words.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r > 0) {
      k.x += 0x9E3779B9u;
      k.y += 0xBB67AE85u;
    }
    const uint32_t hi0 = __umulhi(0xD2511F53u, c.x);
    const uint32_t lo0 = 0xD2511F53u * c.x;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z);
    const uint32_t lo1 = 0xCD9E8D57u * c.z;
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
  }
  return c;
}

__device__ __forceinline__ double u01_53(uint32_t a, uint32_t b) {
  const double hi = (double)(a >> 5);
  const double lo = (double)(b >> 6);
  return __dmul_rn(__dadd_rn(__dmul_rn(hi, 67108864.0), lo), 1.0 / 9007199254740992.0);
}

// uniform number `draw` of stream `tag` at counter (k, s, w)
__device__ __forceinline__ double stream_u01(uint64_t seed, uint32_t tag, uint32_t draw,
                                             uint32_t k, uint32_t s, uint32_t w) {
  const uint2 key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32) ^ tag);
  const uint4 r = philox4x32_10(make_uint4(draw >> 1, k, s, w), key);
  return (draw & 1u) ? u01_53(r.z, r.w) : u01_53(r.x, r.y);
}

// ---------------------------------------------------------------------------
// Pair loops of Eq. (1).  One-sided form: the thread owning atom i sums over
// every j != i, so no two threads write the same gradient entry and the
// result is deterministic.  Per owned atom it returns
//   acc_i = sum_j s2 s6 (2 s6 - 1) (x_i - x_j),  e_i = sum_j s6 (s6 - 1)
// with s2 = sigma^2 / r^2, s6 = s2^3; then grad_i = -(24 eps / sigma^2) acc_i
// and E = 2 eps sum_i e_i (every unordered pair is visited twice).
// ---------------------------------------------------------------------------
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

__device__ __forceinline__ float rsqrt_approx(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float ex2_approx(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// 1 / a in FP64, correctly rounded: the hardware's estimate r (PTX
// rcp.approx.ftz.f64, ~2^-20 relative), one third-order Householder step,
// y = r (1 + e + e^2) with e = 1 - a r formed by one FMA (truncation error
// e^3 < 2^-58: within an ulp), and Markstein's correction y + y (1 - a y)
// (IBM J. Res. Dev. 34, 1990), whose residual is exact and whose own error is far
// below the distance of any 1 / a from a rounding boundary, but for the
// significand of all ones.  Five FP64 instructions, about nine of __drcp_rn
// (65,536 x LJ38: 2.23 ms; 2.07 without the correction, which leaves a few results
// in a thousand an ulp off).  None on the FP64 pipe for the ends of the range: an
// estimate of 0 or infinity (a = 0, infinite or so small that its inverse overflows)
// is returned as it is, chosen by its exponent bits on the integer pipe.
__device__ __forceinline__ bool f64_end(double r) {   // 0, subnormal, infinite or NaN
  const int ex = __double2hiint(r) & 0x7ff00000;
  return ex == 0 || ex == 0x7ff00000;
}
__device__ __forceinline__ double rcp_f64(double a, double one = 1.0) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(a));
  const double e = fma(-a, r, one);
  double y = fma(r, fma(e, e, e), r);
  y = fma(y, fma(-a, y, one), y);
  return f64_end(r) ? r : y;
}

struct alignas(16) PosF { float x, y, z, w; };
struct alignas(16) PosD { double x, y, z, w; };

template <typename X> struct PosOf;
template <> struct PosOf<float> { using type = PosF; };
template <> struct PosOf<double> { using type = PosD; };

// ---------------------------------------------------------------------------
// FP32 pair rows on packed float pairs (sm_100+ FADD2 / FMUL2 / FFMA2: two
// IEEE single operations per instruction, each rounded exactly like its
// scalar form).  Positions are staged two atoms per 32-byte record, atoms
// 2m and 2m+1 in record m (unscaled: differences of the given coordinates
// are the exact-as-possible inputs of r2, and sigma enters as one product
// sigma^2 / r2 where sigma != 1); an odd cluster
// pads its last record with kFarAtom, whose terms underflow to exactly zero
// (r2 ~ 4e36 keeps 1/r2 normal, (1/r2)^2 rounds to 0), so every record holds
// two live lanes and no lane needs a bounds test.  One instruction then
// serves two pair terms, which halves the issue slots of the FP32 row: the
// row is bound by the FMA pipe instead of by instruction issue.
// ---------------------------------------------------------------------------
struct alignas(16) PosF2 {
  float x[2], y[2], z[2], w[2];
};
constexpr float kFarAtom = 0x1p60f;

__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }

// stage atom i into its record; the owner of the last atom of an odd
// cluster also writes the padding lane
__device__ __forceinline__ void stage_f32x2(PosF2* pos, int n, int i, float x, float y, float z) {
  PosF2& r = pos[i >> 1];
  const int l = i & 1;
  r.x[l] = x; r.y[l] = y; r.z[l] = z;
  if (i == n - 1 && l == 0) {
    r.x[1] = kFarAtom; r.y[1] = kFarAtom; r.z[1] = kFarAtom;
  }
}

// One-sided row of atom i (position px, py, pz) against the n atoms of
// `pos`: b = sum_j c_ij (x_j - x_i) with c = s2 s6 (2 s6 - 1), s2 = sigma^2
// / r^2 (SIG: sigma != 1, sig2 = sigma^2), and e += sum_j s6 (s6 - 1), the
// self term excluded.  Energy: per lane, blocks of 4 terms summed in FP32,
// the two lanes' block sums added and folded into the float-float `e`.
template <bool SIG>
__device__ __forceinline__ void pair_row_f32x2(int n, int i, float px, float py, float pz,
                                               const PosF2* __restrict__ pos, float sig2,
                                               float& bx, float& by, float& bz, ff& e) {
  const int M = (n + 1) >> 1;
  const float2 npx = f2(-px), npy = f2(-py), npz = f2(-pz), m1 = f2(-1.f);
  const int sx = (i & 1) ? -1 : (i >> 1);     // record whose lane 0 is atom i
  const int sy = (i & 1) ? (i >> 1) : -1;     // record whose lane 1 is atom i
  float2 ax = f2(0.f), ay = f2(0.f), az = f2(0.f);
  auto term = [&](int m, float2& eb) {
    const float4 xy = *reinterpret_cast<const float4*>(&pos[m].x[0]);
    const float2 zz = *reinterpret_cast<const float2*>(&pos[m].z[0]);
    const float2 dx = __fadd2_rn(make_float2(xy.x, xy.y), npx);
    const float2 dy = __fadd2_rn(make_float2(xy.z, xy.w), npy);
    const float2 dz = __fadd2_rn(zz, npz);
    const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
    float2 s2;
    s2.x = (m == sx) ? 0.f : rcp_approx(r2.x);
    s2.y = (m == sy) ? 0.f : rcp_approx(r2.y);
    if constexpr (SIG) s2 = __fmul2_rn(s2, f2(sig2));
    const float2 s6 = __fmul2_rn(__fmul2_rn(s2, s2), s2);
    const float2 t = __fadd2_rn(s6, m1);
    eb = __ffma2_rn(s6, t, eb);
    const float2 c = __fmul2_rn(__fmul2_rn(s2, s6), __fadd2_rn(s6, t));
    ax = __ffma2_rn(c, dx, ax);
    ay = __ffma2_rn(c, dy, ay);
    az = __ffma2_rn(c, dz, az);
  };
  int m = 0;
  for (; m + 4 <= M; m += 4) {
    float2 eb = f2(0.f);
#pragma unroll
    for (int u = 0; u < 4; ++u) term(m + u, eb);
    e = ff_add_f(e, __fadd_rn(eb.x, eb.y));
  }
  if (m < M) {
    float2 eb = f2(0.f);
    for (; m < M; ++m) term(m, eb);
    e = ff_add_f(e, __fadd_rn(eb.x, eb.y));
  }
  bx = __fadd_rn(ax.x, ax.y);
  by = __fadd_rn(ay.x, ay.y);
  bz = __fadd_rn(az.x, az.y);
}

// One-sided Morse row of atom i on the same packed records (unscaled
// coordinates): with r from r^2 and a reciprocal square root, e = exp(rho -
// rr r) (rr = rho / re; FP32 __expf), b = sum_j e (e - 1) (x_j - x_i) / r and
// e_row += sum_j e (e - 2), the self term excluded; the padding atom's terms
// vanish (its exponential underflows to 0).  Energy blocks as in
// pair_row_f32x2 (float-float).
__device__ __forceinline__ void morse_row_f32x2(int n, int i, float px, float py, float pz,
                                                const PosF2* __restrict__ pos, float rho,
                                                float rr, float& bx, float& by, float& bz,
                                                ff& e) {
  const int M = (n + 1) >> 1;
  const float2 npx = f2(-px), npy = f2(-py), npz = f2(-pz);
  const float2 nrr = f2(-rr), rho2 = f2(rho), m1 = f2(-1.f), m2 = f2(-2.f);
  const int sx = (i & 1) ? -1 : (i >> 1);     // record whose lane 0 is atom i
  const int sy = (i & 1) ? (i >> 1) : -1;     // record whose lane 1 is atom i
  float2 ax = f2(0.f), ay = f2(0.f), az = f2(0.f);
  auto term = [&](int m, float2& eb) {
    const float4 xy = *reinterpret_cast<const float4*>(&pos[m].x[0]);
    const float2 zz = *reinterpret_cast<const float2*>(&pos[m].z[0]);
    const float2 dx = __fadd2_rn(make_float2(xy.x, xy.y), npx);
    const float2 dy = __fadd2_rn(make_float2(xy.z, xy.w), npy);
    const float2 dz = __fadd2_rn(zz, npz);
    const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
    float2 ir = make_float2(rsqrtf(r2.x), rsqrtf(r2.y));
    if (m == sx) ir.x = 0.f;                   // the self term: r = 0 instead of 0 * inf
    if (m == sy) ir.y = 0.f;
    const float2 x = __ffma2_rn(nrr, __fmul2_rn(r2, ir), rho2);      // rho (1 - r / re)
    float2 ex = make_float2(__expf(x.x), __expf(x.y));
    if (m == sx) ex.x = 0.f;
    if (m == sy) ex.y = 0.f;
    eb = __ffma2_rn(ex, __fadd2_rn(ex, m2), eb);
    const float2 c = __fmul2_rn(__fmul2_rn(ex, __fadd2_rn(ex, m1)), ir);
    ax = __ffma2_rn(c, dx, ax);
    ay = __ffma2_rn(c, dy, ay);
    az = __ffma2_rn(c, dz, az);
  };
  int m = 0;
  for (; m + 4 <= M; m += 4) {
    float2 eb = f2(0.f);
#pragma unroll
    for (int u = 0; u < 4; ++u) term(m + u, eb);
    e = ff_add_f(e, __fadd_rn(eb.x, eb.y));
  }
  if (m < M) {
    float2 eb = f2(0.f);
    for (; m < M; ++m) term(m, eb);
    e = ff_add_f(e, __fadd_rn(eb.x, eb.y));
  }
  bx = __fadd_rn(ax.x, ax.y);
  by = __fadd_rn(ay.x, ay.y);
  bz = __fadd_rn(az.x, az.y);
}

struct dd {
  double hi, lo;
};
// s += v for a running double-double sum (Sum2, as df_acc).  TwoSum with the
// operands ordered by magnitude on the integer pipe: three FP64 additions
// (Dekker's FastTwoSum) instead of six; a warp's FP64 instruction takes its
// SM sub-partition's unit for 67 cycles.
__device__ __forceinline__ void dd_acc(dd& s, dd v) {
  const bool sw = (__double2hiint(s.hi) & 0x7fffffff) < (__double2hiint(v.hi) & 0x7fffffff);
  const double a = sw ? v.hi : s.hi, b = sw ? s.hi : v.hi;
  s.hi = __dadd_rn(a, b);
  s.lo = __dadd_rn(__dsub_rn(b, __dsub_rn(s.hi, a)), __dadd_rn(s.lo, v.lo));
}
__device__ __forceinline__ void dd_acc(dd& s, double v) {
  const bool sw = (__double2hiint(s.hi) & 0x7fffffff) < (__double2hiint(v) & 0x7fffffff);
  const double a = sw ? v : s.hi, b = sw ? s.hi : v;
  s.hi = __dadd_rn(a, b);
  s.lo = __dadd_rn(__dsub_rn(b, __dsub_rn(s.hi, a)), s.lo);
}

template <int T>
__device__ __forceinline__ double team_sum_dd(const Team<T>& tm, dd v) {
  // the error of a sum is the same number whichever operand FastTwoSum takes
  // first, so both partners of a butterfly step hold the same bits
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) dd_acc(v, dd{shfl_xor(v.hi, o), shfl_xor(v.lo, o)});
  if constexpr (T > 32) {
    constexpr int NW = T / 32;
    double* buf = tm.scratch();
    if ((tm.rank & 31) == 0) {
      buf[2 * (tm.rank >> 5)] = v.hi;
      buf[2 * (tm.rank >> 5) + 1] = v.lo;
    }
    tm.sync();
    dd s{buf[0], buf[1]};
#pragma unroll
    for (int w = 1; w < NW; ++w) dd_acc(s, dd{buf[2 * w], buf[2 * w + 1]});
    v = s;
  }
  return __dadd_rn(v.hi, v.lo);
}

// FP64: the energy is summed in
// 4-term blocks folded into a compensated (double-double) accumulator, so
// that near a minimum its rounding noise stays below the decreases the
// line search must resolve (|E| ~ 170 for LJ38, decreases ~1e-12).
__device__ __forceinline__ void pair_row_f64(int n, int i, double px, double py, double pz,
                                             const PosD* __restrict__ pos, double sig2,
                                             double& ax, double& ay, double& az, dd& e) {
  ax = 0.0; ay = 0.0; az = 0.0;
  int j = 0;
  for (; j + 4 <= n; j += 4) {
    double eb = 0.0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const PosD q = pos[j + u];
      const double dx = px - q.x, dy = py - q.y, dz = pz - q.z;
      const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
      const double ir2 = (j + u == i) ? 0.0 : rcp_f64(r2);
      const double s2 = sig2 * ir2;
      const double s6 = s2 * s2 * s2;
      const double t = s6 - 1.0;
      eb = fma(s6, t, eb);
      const double c = (s2 * s6) * (s6 + t);
      ax = fma(c, dx, ax);
      ay = fma(c, dy, ay);
      az = fma(c, dz, az);
    }
    dd_acc(e, eb);
  }
  double eb = 0.0;
  for (; j < n; ++j) {
    const PosD q = pos[j];
    const double dx = px - q.x, dy = py - q.y, dz = pz - q.z;
    const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
    const double ir2 = (j == i) ? 0.0 : rcp_f64(r2);
    const double s2 = sig2 * ir2;
    const double s6 = s2 * s2 * s2;
    const double t = s6 - 1.0;
    eb = fma(s6, t, eb);
    const double c = (s2 * s6) * (s6 + t);
    ax = fma(c, dx, ax);
    ay = fma(c, dy, ay);
    az = fma(c, dz, az);
  }
  dd_acc(e, eb);
}

// ---------------------------------------------------------------------------
// Double-float ("df") arithmetic: a value is hi + lo with two FP32 words
// (~48-bit significand), built from error-free transformations on the FP32
// pipes (TwoSum, and TwoProd via FMA; Dekker 1971, Knuth TAOCP 4.2.2).  The
// mixed path evaluates its polish phase with these: on GB300 one FP64
// instruction issues at ~1/62 the FP32 rate, so ~200 FP32 operations per pair
// cost several times less than ~27 FP64 ones while giving ~1e-14 relative
// accuracy.  Products whose rounded value enters an error term use the _rn
// intrinsics so that no multiply is contracted into a later add.
// ---------------------------------------------------------------------------
struct alignas(16) PosDF { float xh, yh, zh, wh, xl, yl, zl, wl; };

__device__ __forceinline__ ff df_fast_two_sum(float a, float b) {   // |a| >= |b| or a == 0
  const float s = __fadd_rn(a, b);
  return ff{s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ ff df_two_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return ff{p, fmaf(a, b, -p)};
}
__device__ __forceinline__ ff df_add(ff a, ff b) {
  const ff s = ff_two_sum(a.hi, b.hi);
  return df_fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ ff df_sub(ff a, ff b) {
  const ff s = ff_two_sum(a.hi, -b.hi);
  return df_fast_two_sum(s.hi, __fadd_rn(s.lo, __fsub_rn(a.lo, b.lo)));
}
// a b without the last renormalisation, for products that are only summed (df_acc):
// 4 operations instead of 7.  Differences of coordinates are renormalised
// before they are multiplied: without that, lo is an ulp of the coordinates and
// not of their difference, and the lo * lo and the roundings that a product drops
// made pair terms 1.2 (small clusters) to 1.8 times (12 sigma across) less exact.
__device__ __forceinline__ ff df_mul_raw(ff a, ff b) {
  const ff p = df_two_prod(a.hi, b.hi);
  return ff{p.hi, fmaf(a.lo, b.hi, fmaf(a.hi, b.lo, p.lo))};
}
__device__ __forceinline__ ff df_add_f(ff a, float b) {
  const ff s = ff_two_sum(a.hi, b);
  return df_fast_two_sum(s.hi, __fadd_rn(s.lo, a.lo));
}
__device__ __forceinline__ ff df_mul(ff a, ff b) {
  const ff p = df_two_prod(a.hi, b.hi);
  const float e = fmaf(a.lo, b.hi, fmaf(a.hi, b.lo, p.lo));
  return df_fast_two_sum(p.hi, e);
}
__device__ __forceinline__ ff df_sqr(ff a) {
  const ff p = df_two_prod(a.hi, a.hi);
  return df_fast_two_sum(p.hi, fmaf(__fmul_rn(2.f, a.hi), a.lo, p.lo));
}
// 1 / a: FP32 reciprocal estimate refined by one Newton step in df,
// w = r + r (1 - a r); relative error ~ (rel. error of r)^2 + 2^-47
__device__ __forceinline__ ff df_rcp(ff a) {
  const float r = rcp_approx(a.hi);
  const ff p = df_two_prod(a.hi, r);
  float t = __fsub_rn(__fsub_rn(1.f, p.hi), p.lo);
  t = fmaf(-a.lo, r, t);
  return df_fast_two_sum(r, __fmul_rn(r, t));
}
__device__ __forceinline__ ff df_from_double(double x) {
  const float h = (float)x;
  return ff{h, (float)(x - (double)h)};
}

// |d|^2 of a double-float vector with one renormalisation: the high squares
// exactly (TwoProd by FMA), summed by two TwoSums, and every low-order part
// (their rounding errors, (2 hi + lo) lo, the TwoProd errors) gathered in one FP32
// word, whose roundings are ~2^-47 of the result.
__device__ __forceinline__ ff df_norm2(ff x, ff y, ff z) {
  const float px = __fmul_rn(x.hi, x.hi), py = __fmul_rn(y.hi, y.hi), pz = __fmul_rn(z.hi, z.hi);
  const float ex = fmaf(x.hi, x.hi, -px), ey = fmaf(y.hi, y.hi, -py), ez = fmaf(z.hi, z.hi, -pz);
  const ff s1 = ff_two_sum(px, py);
  const ff s2 = ff_two_sum(s1.hi, pz);
  float lo = __fadd_rn(__fadd_rn(s1.lo, s2.lo), __fadd_rn(__fadd_rn(ex, ey), ez));
  lo = fmaf(fmaf(2.f, x.hi, x.lo), x.lo, lo);
  lo = fmaf(fmaf(2.f, y.hi, y.lo), y.lo, lo);
  lo = fmaf(fmaf(2.f, z.hi, z.lo), z.lo, lo);
  return df_fast_two_sum(s2.hi, lo);
}

// sqrt(a) in double-float (Karp and Markstein, ACM TOMS 1997): y ~ 1/sqrt(a)
// in FP32, s = a y, and one correction s + y (a - s^2) / 2 with a - s^2
// formed exactly (TwoProd); ~2^-46 relative.  a = 0 gives 0.
__device__ __forceinline__ ff df_sqrt(ff a) {
  if (!(a.hi > 0.f)) return ff{0.f, 0.f};
  const float y = rsqrtf(a.hi);
  const float s = __fmul_rn(a.hi, y);
  const ff p = df_two_prod(s, s);
  const float res = __fadd_rn(__fsub_rn(__fsub_rn(a.hi, p.hi), p.lo), a.lo);
  return df_fast_two_sum(s, __fmul_rn(__fmul_rn(res, y), 0.5f));
}

// e^x in double-float.  Argument reduction x = k ln 2 + r, k = rint(x / ln 2),
// with ln 2 split into three FP32 words of which the first has 16 bits (so
// k ln2_1 is exact for |k| < 256); then e^r = (e^(r/32))^32, e^(r/32) by its
// Taylor series to degree 7 in double-float Horner form (|r/32| <= 0.0109:
// the first dropped term is below 2^-58), five squarings (which multiply the
// relative error by 32: ~2^-42 in all), and the exact scaling of both words by
// 2^k.  For x < -87.3 (e^x below FP32's normal range) the result is 0.
constexpr double kLn2 = 0.69314718055994530942;
constexpr float kLn2_1 = (float)((double)(long long)(kLn2 * 65536.0) / 65536.0);
constexpr float kLn2_2 = (float)(kLn2 - (double)kLn2_1);
constexpr float kLn2_3 = (float)(kLn2 - (double)kLn2_1 - (double)kLn2_2);
// 1/k! as double-float words (high: the FP32 rounding, low: the FP32
// rounding of the rest), formed at compile time
constexpr float df_hi(double c) { return (float)c; }
constexpr float df_lo(double c) { return (float)(c - (double)(float)c); }
constexpr float kF3h = df_hi(1.0 / 6), kF3l = df_lo(1.0 / 6);
constexpr float kF4h = df_hi(1.0 / 24), kF4l = df_lo(1.0 / 24);
constexpr float kF5h = df_hi(1.0 / 120), kF5l = df_lo(1.0 / 120);
constexpr float kF6h = df_hi(1.0 / 720), kF6l = df_lo(1.0 / 720);
constexpr float kF7h = df_hi(1.0 / 5040), kF7l = df_lo(1.0 / 5040);
__device__ __forceinline__ ff df_exp(ff x) {
  if (x.hi < -87.3f) return ff{0.f, 0.f};
  const float k = rintf(__fmul_rn(x.hi, 1.44269504f));
  ff r = df_add_f(x, -__fmul_rn(k, kLn2_1));            // k ln2_1 exact
  r = df_sub(r, df_two_prod(k, kLn2_2));
  r = df_add_f(r, -__fmul_rn(k, kLn2_3));
  r.hi *= 0.03125f;                                      // r / 32, exact
  r.lo *= 0.03125f;
  ff p{kF7h, kF7l};
  p = df_add(df_mul(p, r), ff{kF6h, kF6l});
  p = df_add(df_mul(p, r), ff{kF5h, kF5l});
  p = df_add(df_mul(p, r), ff{kF4h, kF4l});
  p = df_add(df_mul(p, r), ff{kF3h, kF3l});
  p = df_add(df_mul(p, r), ff{0.5f, 0.f});
  p = df_add_f(df_mul(p, r), 1.f);
  p = df_add_f(df_mul(p, r), 1.f);
#pragma unroll
  for (int i = 0; i < 5; ++i) p = df_sqr(p);
  const float sc = __int_as_float(((int)k + 127) << 23);   // 2^k, k in [-126, 127]
  return ff{p.hi * sc, p.lo * sc};
}

// Morse pair term in double-float on coordinates scaled by 1/re: with
// e = exp(rho (1 - r)), v = e (e - 1) (x_i - x_j) / r and e_pair = e (e - 2)
// (+inf for coincident atoms).  rho is the double-float range parameter.
__device__ __forceinline__ void pair_term_morse_df(const PosDF& a, const PosDF& b, ff rho,
                                                   ff& vx, ff& vy, ff& vz, ff& e) {
  const ff dx = df_sub(ff{a.xh, a.xl}, ff{b.xh, b.xl});
  const ff dy = df_sub(ff{a.yh, a.yl}, ff{b.yh, b.yl});
  const ff dz = df_sub(ff{a.zh, a.zl}, ff{b.zh, b.zl});
  const ff r2 = df_norm2(dx, dy, dz);
  const ff r = df_sqrt(r2);
  const ff ex = df_exp(df_sub(rho, df_mul(rho, r)));
  e = r2.hi > 0.f ? df_mul(ex, df_add_f(ex, -2.f)) : ff{__int_as_float(0x7f800000), 0.f};
  const ff c = df_mul(df_mul(ex, df_add_f(ex, -1.f)), df_rcp(r));
  vx = df_mul_raw(c, dx); vy = df_mul_raw(c, dy); vz = df_mul_raw(c, dz);
}

// One row of the pair sum in df arithmetic, coordinates pre-scaled by
// 1/sigma (so s2 = 1/r^2).  Accumulates acc_i = sum_j s2 s6 (2 s6 - 1) d_ij
// and e_i = sum_j s6 (s6 - 1), both as df.
__device__ __forceinline__ void pair_row_df(int n, int i, ff px, ff py, ff pz,
                                            const PosDF* __restrict__ pos,
                                            ff& ax, ff& ay, ff& az, ff& e) {
  ax = ff{0.f, 0.f}; ay = ff{0.f, 0.f}; az = ff{0.f, 0.f};
#pragma unroll 2
  for (int j = 0; j < n; ++j) {
    const PosDF q = pos[j];
    const ff dx = df_sub(px, ff{q.xh, q.xl});
    const ff dy = df_sub(py, ff{q.yh, q.yl});
    const ff dz = df_sub(pz, ff{q.zh, q.zl});
    const ff r2 = df_norm2(dx, dy, dz);
    ff s2 = df_rcp(r2);
    if (j == i) s2 = ff{0.f, 0.f};
    const ff s6 = df_mul(df_sqr(s2), s2);
    const ff t = df_add_f(s6, -1.f);
    df_acc(e, df_mul(s6, t));
    const ff c = df_mul(df_mul(s2, s6), df_add(s6, t));
    df_acc(ax, df_mul(c, dx));
    df_acc(ay, df_mul(c, dy));
    df_acc(az, df_mul(c, dz));
  }
}

// ---------------------------------------------------------------------------
// Half-pair evaluation (FP64 and double-float, clusters of up to 64 atoms): each
// unordered pair once.  Thread p mod T evaluates pair p and writes its vector
// v_p = c_ij (x_i - x_j) to a shared buffer; after a barrier the sum of an atom
// and axis takes +v of the pairs that start at the atom and -v of those that
// end there.  Every pair costs one evaluation instead of two and the work
// splits evenly over the team whatever N is.  Fixed pair order, fixed sum order.
//
// Mixed precision (double-float and its FP64 tier): the order of a ring.  Pair p is atom i = p mod n with
// j = (i + k) mod n, k = 1 + p / n (for even n the shift n/2 holds the n/2 pairs
// i < n/2), so that an atom's pairs are at ((k-1) n + atom) and
// ((k-1) n + (atom - k) mod n): consecutive lanes at consecutive words, no bank
// conflicts, one index and one comparison a term.
//
// FP64 path: row-major order of the upper triangle, i < j, and row sums over j = 0 ..
// n-1 in four interleaved parts.  Which order is taken shows in results: at the
// default gtol of 1e-6 the decrease that a last line search has to resolve
// (~1e-15 for LJ13) is below an ulp of E, so whether a trial ends as CONVERGED
// or as LINESEARCH_FAIL is decided by the last bit of a sum, and a Basin Hopping
// trace records it.  The ring's order with a flat history and a reciprocal within
// an ulp is faster (50 steps of LJ13: 37 against 46 ms) but gives other traces.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int n_pairs(int n) { return n * (n - 1) / 2; }

// pair (i, j) of index p in the ring's order, advanced by a fixed step
struct PairWalk {
  int i, k;
  __device__ __forceinline__ PairWalk(int n, int p) : i(p % n), k(1 + p / n) {}
  __device__ __forceinline__ int j(int n) const {
    const int t = i + k;
    return t >= n ? t - n : t;
  }
  // step = dk n + di, 0 <= di < n
  __device__ __forceinline__ void advance(int n, int dk, int di) {
    i += di;
    k += dk;
    if (i >= n) { i -= n; ++k; }
  }
};

// two pairs in flight a thread (the second clamped to pair (0, 1) past the end
// and discarded); term(i, j, vx, vy, vz, e) evaluates one, add(e) takes its
// energy
template <int T, typename F, typename Term, typename Add>
__device__ __forceinline__ void half_pairs(int rank, int n, F* vb, Term&& term, Add&& add) {
  const int np = n_pairs(n);
  const int dk = 2 * T / n, di = 2 * T - dk * n;
  PairWalk w1(n, rank), w2(n, rank + T);
  for (int q = rank; q < np; q += 2 * T) {
    const bool two = q + T < np;
    F ax, ay, az, ae, bx, by, bz, be;
    term(w1.i, w1.j(n), ax, ay, az, ae);
    term(two ? w2.i : 0, two ? w2.j(n) : 1, bx, by, bz, be);
    vb[q] = ax; vb[np + q] = ay; vb[2 * np + q] = az;
    add(ae);
    if (two) {
      vb[q + T] = bx; vb[np + q + T] = by; vb[2 * np + q + T] = bz;
      add(be);
    }
    w1.advance(n, dk, di);
    w2.advance(n, dk, di);
  }
}

__device__ __forceinline__ void half_plus(ff& s, ff v) { df_acc(s, v); }
__device__ __forceinline__ void half_minus(ff& s, ff v) { df_acc(s, ff{-v.hi, -v.lo}); }
__device__ __forceinline__ float half_total(ff a, ff b, ff c, ff d) {
  df_acc(a, c); df_acc(b, d); df_acc(a, b);
  return __fadd_rn(a.hi, a.lo);
}
__device__ __forceinline__ void half_plus(double& s, double v) { s += v; }
__device__ __forceinline__ void half_minus(double& s, double v) { s -= v; }
__device__ __forceinline__ double half_total(double a, double b, double c, double d) {
  return (a + c) + (b + d);              // the pairs that start, then those that end
}

// sums[3 atom + axis] = scale * sum, one (axis, atom) a thread, four
// independent sums each
template <int T, typename F, typename G>
__device__ __forceinline__ void half_rows(int rank, int n, const F* vb, G scale, G* sums) {
  const int np = n_pairs(n), H = (n - 1) >> 1;
  for (int q3 = rank; q3 < 3 * n; q3 += T) {
    const int axis = q3 >= 2 * n ? 2 : q3 >= n ? 1 : 0;
    const int ii = q3 - axis * n;
    const F* vc = vb + axis * np;
    const F* vp = vc + ii;                 // pairs that start at the atom
    int e = ii;                            // (atom - k) mod n
    F s0{}, s1{}, s2{}, s3{};
    int k = 0;
    for (; k + 2 <= H; k += 2) {
      const int e1 = e > 0 ? e - 1 : n - 1;
      const int e2 = e1 > 0 ? e1 - 1 : n - 1;
      const F a = vp[0], b = vc[e1], c = vp[n], d = vc[n + e2];
      half_plus(s0, a);
      half_minus(s1, b);
      half_plus(s2, c);
      half_minus(s3, d);
      e = e2;
      vp += 2 * n;
      vc += 2 * n;
    }
    if (k < H) {
      half_plus(s0, vp[0]);
      half_minus(s1, vc[e > 0 ? e - 1 : n - 1]);
      vp += n;
      vc += n;
    }
    if (!(n & 1)) {                        // the half shift of an even n
      if (ii < n / 2) half_plus(s2, vp[0]);
      else half_minus(s3, vc[ii - n / 2]);
    }
    sums[3 * ii + axis] = scale * half_total(s0, s1, s2, s3);
  }
}

// pair (i, j) of index p, i < j, in the row-major upper triangle; j = -1 if none
struct TriWalk {
  int i, j;
  __device__ __forceinline__ TriWalk(int n, int p) : i(0) {
    int row = n - 1;
    while (row > 0 && p >= row) { p -= row; ++i; --row; }
    j = row > 0 ? i + 1 + p : -1;
  }
  __device__ __forceinline__ void advance(int n, int step) {
    j += step;
    while (i < n - 1 && j >= n) {
      j -= n;         // j - n = offset past the row end
      ++i;
      j += i + 1;     // first column of the next row is i+1
    }
  }
};
// pair (j, i), j < i, sits at tri_base(n, j) + i and pair (i, j), j > i, at
// tri_base(n, i) + j; tri_base(n, j + 1) = tri_base(n, j) + n - j - 2,
// tri_base(n, 0) = -1
__device__ __forceinline__ int tri_base(int n, int i) {
  return i * (2 * n - i - 1) / 2 - i - 1;
}

// two pairs in flight a thread, as half_pairs; the energies of the two are
// added in FP64, then to the double-double sum
template <int T, typename Term>
__device__ __forceinline__ void tri_pairs(int rank, int n, double* vb, Term&& term, dd& e) {
  const int np = n_pairs(n);
  TriWalk w1(n, rank), w2 = w1;
  w2.advance(n, T);
  for (int q = rank; q < np; q += 2 * T) {
    const bool two = q + T < np;
    double ax, ay, az, ae, bx, by, bz, be;
    term(w1.i, w1.j, ax, ay, az, ae);
    term(two ? w2.i : 0, two ? w2.j : 1, bx, by, bz, be);
    vb[q] = ax; vb[np + q] = ay; vb[2 * np + q] = az;
    double eb = ae;
    if (two) {
      vb[q + T] = bx; vb[np + q + T] = by; vb[2 * np + q + T] = bz;
      eb += be;
    }
    dd_acc(e, eb);
    w1.advance(n, 2 * T);
    w2.advance(n, 2 * T);
  }
}

// sums[3 atom + axis] = -gs * sum, one (atom, axis) a thread; all lanes walk j
// together, +v over j > atom, -v over j < atom
template <int T>
__device__ __forceinline__ void tri_rows(int rank, int n, const double* vb, double gs,
                                              double* sums) {
  const int np = n_pairs(n);
  for (int q3 = rank; q3 < 3 * n; q3 += T) {
    const int ii = q3 / 3;
    const double* vc = vb + (q3 - 3 * ii) * np;
    const int ri = tri_base(n, ii);
    int rj = -1;                           // tri_base(n, j)
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    for (int j0 = 0; j0 < n; j0 += 4) {
      double v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int j = j0 + u;
        const int q = j < ii ? rj + ii : ri + j;
        v[u] = 0.0;
        if (j < n && j != ii) v[u] = vc[q];
        if (j < ii) v[u] = -v[u];
        rj += n - j - 2;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) s[u] += v[u];
    }
    sums[q3] = -gs * ((s[0] + s[1]) + (s[2] + s[3]));
  }
}

// pair term in FP64: v = c (x_i - x_j) with c = s2 s6 (2 s6 - 1), e = s6 (s6 - 1)
__device__ __forceinline__ void pair_term_f64(const PosD& a, const PosD& b, double sig2,
                                              double& vx, double& vy, double& vz, double& e) {
  const double dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z;
  const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
  const double s2 = sig2 * rcp_f64(r2);
  const double s6 = s2 * s2 * s2;
  const double t = s6 - 1.0;
  e = s6 * t;
  const double c = (s2 * s6) * (s6 + t);
  vx = c * dx; vy = c * dy; vz = c * dz;
}

// pair term in double-float on coordinates scaled by 1/sigma.  v and e are not
// renormalised (they are summed by df_acc).
__device__ __forceinline__ void pair_term_df(const PosDF& a, const PosDF& b, ff& vx, ff& vy,
                                             ff& vz, ff& e) {
  const ff dx = df_sub(ff{a.xh, a.xl}, ff{b.xh, b.xl});
  const ff dy = df_sub(ff{a.yh, a.yl}, ff{b.yh, b.yl});
  const ff dz = df_sub(ff{a.zh, a.zl}, ff{b.zh, b.zl});
  const ff r2 = df_norm2(dx, dy, dz);
  const ff s2 = df_rcp(r2);
  const ff s6 = df_mul(df_sqr(s2), s2);
  const ff t = df_add_f(s6, -1.f);
  e = df_mul_raw(s6, t);
  const ff c = df_mul(df_mul(s2, s6), df_add(s6, t));
  vx = df_mul_raw(c, dx); vy = df_mul_raw(c, dy); vz = df_mul_raw(c, dz);
}

// ---------------------------------------------------------------------------
// Ring evaluation (FP64 and double-float, clusters of 65 to 256 atoms): every
// unordered pair once, by the thread of atom i at shift k with j = (i + k) mod
// n, k = 1 .. n/2 (at k = n/2 of an even n, i < n/2 only).  The thread adds
// v = c (x_i - x_j) to its own atom in registers and leaves it for j in the
// buffer (KS shifts of n entries, one writer each); after a barrier the owners
// subtract, in the order of the shifts.  Two pairs in flight a thread.
// ---------------------------------------------------------------------------
template <int T, int A, typename F, typename Term, typename Add>
__device__ __forceinline__ void ring_pairs(const Team<T>& tm, int n, int KS, F* buf, Term&& term,
                                           Add&& add, F (&acc)[A][3]) {
  const int full = (n - 1) >> 1;           // shifts that every atom takes
  const int last = n >> 1;                 // > full: the half shift
#pragma unroll
  for (int a = 0; a < A; ++a)
#pragma unroll
    for (int c = 0; c < 3; ++c) acc[a][c] = F{};
  auto one = [&](int a, int i, int k, F* b) {
    int j = i + k;
    if (j >= n) j -= n;
    F vx, vy, vz, e;
    term(i, j, vx, vy, vz, e);
    half_plus(acc[a][0], vx);
    half_plus(acc[a][1], vy);
    half_plus(acc[a][2], vz);
    add(e);
    b[j] = vx; b[n + j] = vy; b[2 * n + j] = vz;
  };
  for (int k0 = 1; k0 <= last; k0 += KS) {
    const int ks = min(KS, last - k0 + 1);
    if (k0 > 1) tm.sync();                 // the last chunk's readers are done
    const int nf = min(ks, full - k0 + 1);
#pragma unroll
    for (int a = 0; a < A; ++a) {
      const int i = tm.rank + a * T;
      if (i < n) {
        int s = 0;
        for (; s + 2 <= nf; s += 2) {
          one(a, i, k0 + s, buf + 3 * n * s);
          one(a, i, k0 + s + 1, buf + 3 * n * (s + 1));
        }
        if (s < nf) one(a, i, k0 + s, buf + 3 * n * s);
        if (nf < ks && i < last) one(a, i, last, buf + 3 * n * nf);
      }
    }
    tm.sync();
#pragma unroll
    for (int a = 0; a < A; ++a) {
      const int i = tm.rank + a * T;
      if (i < n) {
        const int ns = nf < ks && i >= last ? ks : nf;
        for (int s = 0; s < ns; ++s)
#pragma unroll
          for (int c = 0; c < 3; ++c) half_minus(acc[a][c], buf[3 * n * s + c * n + i]);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Double-float evaluation of clusters above the half-pair size: each
// unordered pair once, in tiles of 32 x 32 atom blocks (block b = atoms
// 32b .. 32b+31).  Blocks are paired by the circle method -- round r pairs
// block NB-1 with r and (r+t) mod (NB-1) with (r-t) mod (NB-1), NB even
// (a missing block when the count is odd) -- so that within a round every
// block is in exactly one tile.  A warp takes a tile (I, J): lane l keeps
// atom 32I+l, and atom 32J+l's position and reaction rotate one lane per
// step, so after 32 steps every lane has met every atom of J and holds its
// own J atom's reaction again.  Both sides are then added into per-atom
// double-float accumulators acc[c * n + atom] in shared memory: within a
// round no atom is in two tiles and rounds are separated by a barrier, so
// there are no conflicts and the order is fixed.  A last round takes the
// diagonal tiles (pairs inside a block, each once).  Positions are scaled by
// 1/sigma; v = c (x_i - x_j) as in pair_term_df; e accumulates this lane's
// pair energies s6 (s6 - 1).
// ---------------------------------------------------------------------------
__device__ __forceinline__ PosDF shfl_pos(const PosDF& q, int src) {
  PosDF r;
  r.xh = __shfl_sync(kFull, q.xh, src); r.yh = __shfl_sync(kFull, q.yh, src);
  r.zh = __shfl_sync(kFull, q.zh, src); r.wh = 0.f;
  r.xl = __shfl_sync(kFull, q.xl, src); r.yl = __shfl_sync(kFull, q.yl, src);
  r.zl = __shfl_sync(kFull, q.zl, src); r.wl = 0.f;
  return r;
}
__device__ __forceinline__ ff shfl_ff(ff v, int src) {
  return ff{__shfl_sync(kFull, v.hi, src), __shfl_sync(kFull, v.lo, src)};
}

template <int T>
__device__ void df_tile_eval(const Team<T>& tm, int n, const PosDF* __restrict__ pos, ff* acc,
                             ff& e) {
  constexpr int W = T / 32;
  const int lane = tm.rank & 31, warp = tm.rank >> 5;
  for (int i = tm.rank; i < 3 * n; i += T) acc[i] = ff{0.f, 0.f};
  tm.sync();
  const int nb = (n + 31) >> 5;
  const int nbe = nb + (nb & 1);
  const PosDF far{0x1p60f, 0x1p60f, 0x1p60f, 0.f, 0.f, 0.f, 0.f, 0.f};
  auto tile = [&](int I, int J) {
    const bool diag = I == J;
    const int i = 32 * I + lane;
    const bool vi = i < n;
    const PosDF pi = vi ? pos[i] : far;
    int jl = 32 * J + lane;
    PosDF pj = jl < n ? pos[jl] : far;
    ff fx{0.f, 0.f}, fy{0.f, 0.f}, fz{0.f, 0.f};
    ff hx{0.f, 0.f}, hy{0.f, 0.f}, hz{0.f, 0.f};   // reaction of the rotating J atom
    const int src = (lane + 1) & 31;
    for (int k = 0; k < 32; ++k) {
      const int jk = 32 * J + ((lane + k) & 31);
      bool act = vi && jk < n;
      if (diag) act = act && k >= 1 && (k < 16 || (k == 16 && lane < 16));
      if (__any_sync(kFull, act)) {
        ff vx, vy, vz, ep;
        pair_term_df(pi, pj, vx, vy, vz, ep);
        if (act) {   // cascaded TwoSum (Sum2): one add on each high word's chain
          df_acc(fx, vx); df_acc(fy, vy); df_acc(fz, vz);
          df_acc(hx, ff{-vx.hi, -vx.lo}); df_acc(hy, ff{-vy.hi, -vy.lo});
          df_acc(hz, ff{-vz.hi, -vz.lo});
          df_acc(e, ep);
        }
      }
      pj = shfl_pos(pj, src);
      hx = shfl_ff(hx, src); hy = shfl_ff(hy, src); hz = shfl_ff(hz, src);
    }
    if (diag) {
      fx = df_add(fx, hx); fy = df_add(fy, hy); fz = df_add(fz, hz);
    } else if (jl < n) {
      acc[jl] = df_add(acc[jl], hx);
      acc[n + jl] = df_add(acc[n + jl], hy);
      acc[2 * n + jl] = df_add(acc[2 * n + jl], hz);
    }
    if (vi) {
      acc[i] = df_add(acc[i], fx);
      acc[n + i] = df_add(acc[n + i], fy);
      acc[2 * n + i] = df_add(acc[2 * n + i], fz);
    }
  };
  for (int r = 0; r < nbe - 1; ++r) {
    for (int t = warp; t < nbe / 2; t += W) {
      const int I = t == 0 ? nbe - 1 : (r + t) % (nbe - 1);
      const int J = t == 0 ? r : (r - t + nbe - 1) % (nbe - 1);
      if (I < nb && J < nb) tile(I, J);
    }
    tm.sync();
  }
  for (int b = warp; b < nb; b += W) tile(b, b);
  tm.sync();
}

// FP64 twin of df_tile_eval (clusters above 256 atoms, same circle-method
// rounds of 32 x 32 tiles): pair terms by pair_term_f64 on unscaled
// coordinates, per-atom FP64 accumulators acc[c * n + atom] in the same
// 24-byte-per-atom slot; a lane's pair energies are summed over its tile,
// then added into e with TwoSum.  Each pair once: the FP64 pipe, which bounds
// these evaluations, does ~40% fewer operations than for two one-sided terms.
__device__ __forceinline__ void shfl_posd(PosD& q, int src) {
  q.x = __shfl_sync(kFull, q.x, src);
  q.y = __shfl_sync(kFull, q.y, src);
  q.z = __shfl_sync(kFull, q.z, src);
}

template <int T>
__device__ void d_tile_eval(const Team<T>& tm, int n, const PosD* __restrict__ pos, double sig2,
                            double* acc, dd& e) {
  constexpr int W = T / 32;
  const int lane = tm.rank & 31, warp = tm.rank >> 5;
  for (int i = tm.rank; i < 3 * n; i += T) acc[i] = 0.0;
  tm.sync();
  const int nb = (n + 31) >> 5;
  const int nbe = nb + (nb & 1);
  const PosD far{0x1p300, 0x1p300, 0x1p300, 0.0};
  auto tile = [&](int I, int J) {
    const bool diag = I == J;
    const int i = 32 * I + lane;
    const bool vi = i < n;
    const PosD pi = vi ? pos[i] : far;
    const int jl = 32 * J + lane;
    PosD pj = jl < n ? pos[jl] : far;
    double fx = 0.0, fy = 0.0, fz = 0.0;
    double hx = 0.0, hy = 0.0, hz = 0.0;   // reaction of the rotating J atom
    double eb = 0.0;
    const int src = (lane + 1) & 31;
    for (int k = 0; k < 32; ++k) {
      const int jk = 32 * J + ((lane + k) & 31);
      bool act = vi && jk < n;
      if (diag) act = act && k >= 1 && (k < 16 || (k == 16 && lane < 16));
      if (__any_sync(kFull, act)) {
        double vx, vy, vz, ep;
        pair_term_f64(pi, pj, sig2, vx, vy, vz, ep);
        if (act) {
          fx += vx; fy += vy; fz += vz;
          hx -= vx; hy -= vy; hz -= vz;
          eb += ep;
        }
      }
      shfl_posd(pj, src);
      hx = __shfl_sync(kFull, hx, src);
      hy = __shfl_sync(kFull, hy, src);
      hz = __shfl_sync(kFull, hz, src);
    }
    dd_acc(e, eb);
    if (diag) {
      fx += hx; fy += hy; fz += hz;
    } else if (jl < n) {
      acc[jl] += hx;
      acc[n + jl] += hy;
      acc[2 * n + jl] += hz;
    }
    if (vi) {
      acc[i] += fx;
      acc[n + i] += fy;
      acc[2 * n + i] += fz;
    }
  };
  for (int r = 0; r < nbe - 1; ++r) {
    for (int t = warp; t < nbe / 2; t += W) {
      const int I = t == 0 ? nbe - 1 : (r + t) % (nbe - 1);
      const int J = t == 0 ? r : (r - t + nbe - 1) % (nbe - 1);
      if (I < nb && J < nb) tile(I, J);
    }
    tm.sync();
  }
  for (int b = warp; b < nb; b += W) tile(b, b);
  tm.sync();
}

}  // namespace ljd
