// lj_ring.cuh -- the "ring" layout of lj_energy_grad_batched: every unordered
// pair of a cluster once, any cluster size, any batch.
//
// The atoms of a candidate are taken in groups of G (FP32: four or eight; FP64:
// two to four), NG = ceil(N / G) groups; the missing atoms of the last
// group sit at distinct far positions (2^60 or 2^300 times 1, 2, ...) whose pair
// terms underflow to exactly zero.  Pairs inside a group are taken by its
// thread.  Pairs between groups follow a ring: at shift k = 1 .. H,
// H = floor(NG / 2), group g meets group (g + k) mod NG.  For even NG the
// groups g and g + H would meet twice at shift H, so there the lower one
// takes the lower half of its atoms with all of the partner's and the upper
// one all of its own with the upper half of its partner's.
//
// A candidate has P * NG threads in each of S CTAs (a thread-block cluster):
// thread (p, g) of CTA s takes the shifts k = 1 + j S P + s P + p of group g,
// j = 0, 1, ...  It keeps the force on its own atoms in registers and hands a
// shift's reaction on the partner group to shared memory, one writer per slot;
// after KS shifts and a barrier it subtracts the reactions that were handed to
// its group, in the order of the shifts.  At the end the parts are added in
// the order of p, then of s.  C candidates share a CTA where one would leave
// most of it idle.  Fixed pairs, fixed order, no atomics.
//
// The host's rule (ring_plan in lj_eval.cu) sets C, P and S from N and the
// number of candidates: a large batch runs C candidates a CTA with P = S = 1,
// a small one spreads each candidate over more threads and CTAs.
#pragma once
#include <cooperative_groups.h>

#include "lj_internal.h"
#include "lj_minimize.cuh"
#include "lj_teams.cuh"

namespace ljr {

using namespace ljd;
namespace cg = cooperative_groups;

struct RingPlan {
  int C;       // candidates per CTA (uniform and packed uneven batches; other uneven ones: 1)
  int P;       // parts of a candidate in a CTA (uneven: as many as fit, per candidate)
  int S;       // CTAs per candidate (cluster size)
  int KS;      // shifts between two barriers
  int vec;     // 4-byte words by which every atom group's address is aligned (1, 2 or 4)
};

// FP32: a group's slot (forces) and position record; the latter holds every coordinate twice, as
// the packed operations take it ((x, x, y, y) of each atom, (z, z) of two), and
// is padded so that eight consecutive records start in eight different quarters
// of the banks
template <int G> struct alignas(16) SlotF { float x[G], y[G], z[G]; };
template <int G> struct alignas(16) PosRing { float4 xy[G], zz[G / 2], pad; };
template <int G> struct alignas(16) PosDG { double x[G], y[G], z[G]; };

// shared bytes of a CTA of B threads: positions, reactions, parts, energies
// (16 bytes a thread), one energy per candidate for the cluster
__host__ __device__ constexpr size_t ring_smem(int B, const RingPlan& pl, bool fp32, int G) {
  const size_t slot = fp32 ? 12 * (size_t)G : 24 * (size_t)((G + 1) / 2 * 2);
  const size_t pos = fp32 ? 24 * (size_t)G + 16 : slot;
  return (size_t)B * (pos + slot * (pl.KS + (pl.P > 1 || pl.S > 1 ? 1 : 0))) + (size_t)B * 16 +
         (size_t)pl.C * 16;
}
static_assert(sizeof(PosDG<2>) == 48 && sizeof(PosDG<4>) == 96 && sizeof(SlotF<4>) == 48 &&
                  sizeof(SlotF<8>) == 96 && sizeof(PosRing<4>) == 112 && sizeof(PosRing<8>) == 208,
              "slots of ring_smem");

// ---------------------------------------------------------------------------
// energies: cnt values of each of C candidates (consecutive in `es`), added by
// the first warp in a fixed order: L lanes a candidate, strided, then a tree
// ---------------------------------------------------------------------------
__device__ __forceinline__ void acc_pair(ff& s, ff v) { df_acc(s, v); }
__device__ __forceinline__ void acc_pair(dd& s, dd v) { dd_acc(s, v); }
__device__ __forceinline__ double total(ff s) { return (double)s.hi + (double)s.lo; }
__device__ __forceinline__ double total(dd s) { return __dadd_rn(s.hi, s.lo); }

template <typename E, typename F>
__device__ __forceinline__ void sum_energies(const E* es, int C, int cnt, F&& store) {
  int L = 32;
  while (L > 1 && (L * C > 32 || L >= 2 * cnt)) L >>= 1;
  const int lane = threadIdx.x & 31, sub = lane & (L - 1), per = 32 / L;
  for (int c0 = 0; c0 < C; c0 += per) {
    const int c = c0 + lane / L;
    E s{0, 0};
    if (c < C)
      for (int q = sub; q < cnt; q += L) acc_pair(s, es[c * cnt + q]);
    for (int o = L >> 1; o > 0; o >>= 1)
      acc_pair(s, E{__shfl_xor_sync(kFull, s.hi, o), __shfl_xor_sync(kFull, s.lo, o)});
    if (c < C && sub == 0) store(c, s);
  }
}

// ---------------------------------------------------------------------------
// FP32: packed operations on pairs of pairs
// ---------------------------------------------------------------------------
struct V2 {
  float2 x, y, z;
};

// a thread's energy: in each of the two lanes a running double-float sum (Sum2, as
// df_acc).  Seven packed operations a block of terms, and the lanes stay apart
// to the end: adding them first, in FP32, took nine scalar ones and was the largest
// rounding of a block (65,536 x LJ38: energies off by 6.19e-8 in 57.4 us, 6.06e-8 in
// 59.4 so; 6.08e-8 with blocks of eight pairs in the first ring kernel, 65.5 us).
struct E2 {
  float2 hi, lo;
};
__device__ __forceinline__ float2 sub2(const float2& a, const float2& b) {
  return __ffma2_rn(b, f2(-1.f), a);       // exact product: one rounding
}
__device__ __forceinline__ void e2_acc(E2& e, const float2& v) {
  const float2 s = __fadd2_rn(e.hi, v);
  const float2 bb = sub2(s, e.hi);
  const float2 err = __fadd2_rn(sub2(e.hi, sub2(s, bb)), sub2(v, bb));
  e.hi = s;
  e.lo = __fadd2_rn(e.lo, err);
}
__device__ __forceinline__ ff e2_total(const E2& e) {
  const ff t = ff_two_sum(e.hi.x, e.hi.y);
  return ff{t.hi, __fadd_rn(t.lo, __fadd_rn(e.lo.x, e.lo.y))};
}
__device__ __forceinline__ V2 v2_zero() { return V2{f2(0.f), f2(0.f), f2(0.f)}; }
__device__ __forceinline__ void v2_add(V2& a, const V2& b) {
  a.x = __fadd2_rn(a.x, b.x); a.y = __fadd2_rn(a.y, b.y); a.z = __fadd2_rn(a.z, b.z);
}

// constants of a pair term.  Eq. (1): a = sigma^2.  Morse: a = -re and b + c =
// -(rho / re) log2 e, b its FP32 rounding
struct RingK {
  float a, b, c;
};

// One packed operation: the two pairs (X.lane0, Y.lane0) and (X.lane1,
// Y.lane1), given NX = -X (negation is exact, so y + (-x) rounds like y - x):
// d = y - x, the factor c of the force term c d on x (in units of the
// potential's gradient factor, sign of sum_j c (x_j - x_i); its reaction on y
// is subtracted), and eb += e.
// Eq. (1): s2 = sigma^2 / r^2, c = s2 s6 (2 s6 - 1), e = s6 (s6 - 1).
// Morse: the exponential is 2^((b + c)(r - re)); r - re is one FMA from r^2 and
// 1 / r, so it carries no rounding of r itself.  The slope takes two words: its
// rounding is the same for every pair and would not average out (rho = 6: energies
// of 500 atoms off by 2.4e-8, 0.75e-8 before the ring layout); c = m (m - 1) / r,
// e = m (m - 2).
// With the force and the reaction 19 FP32 lane operations a pair and one
// (Morse: 20 and two) on the MUFU.
template <int POT, bool SIG>
__device__ __forceinline__ void ring_op(const V2& NX, const V2& Y, const RingK& k, V2& d,
                                        float2& c, float2& eb) {
  d.x = __fadd2_rn(Y.x, NX.x);
  d.y = __fadd2_rn(Y.y, NX.y);
  d.z = __fadd2_rn(Y.z, NX.z);
  const float2 r2 = __ffma2_rn(d.x, d.x, __ffma2_rn(d.y, d.y, __fmul2_rn(d.z, d.z)));
  if constexpr (POT == LJ_POT_LJ) {
    float2 s2 = make_float2(rcp_approx(r2.x), rcp_approx(r2.y));
    if constexpr (SIG) s2 = __fmul2_rn(s2, f2(k.a));
    const float2 s6 = __fmul2_rn(__fmul2_rn(s2, s2), s2);
    const float2 t = __fadd2_rn(s6, f2(-1.f));
    eb = __ffma2_rn(s6, t, eb);
    c = __fmul2_rn(__fmul2_rn(s2, s6), __fadd2_rn(s6, t));
  } else {
    const float2 ir = make_float2(rsqrt_approx(r2.x), rsqrt_approx(r2.y));
    const float2 u = __ffma2_rn(r2, ir, f2(k.a));
    const float2 x = __ffma2_rn(u, f2(k.b), __fmul2_rn(u, f2(k.c)));
    const float2 m = make_float2(ex2_approx(x.x), ex2_approx(x.y));
    eb = __ffma2_rn(m, __fadd2_rn(m, f2(-2.f)), eb);
    c = __fmul2_rn(__fmul2_rn(m, __fadd2_rn(m, f2(-1.f))), ir);
  }
}
__device__ __forceinline__ V2 v2_scale(const float2& c, const V2& d) {
  return V2{__fmul2_rn(c, d.x), __fmul2_rn(c, d.y), __fmul2_rn(c, d.z)};
}
__device__ __forceinline__ void v2_fma(V2& f, const float2& c, const V2& d) {
  f.x = __ffma2_rn(c, d.x, f.x);
  f.y = __ffma2_rn(c, d.y, f.y);
  f.z = __ffma2_rn(c, d.z, f.z);
}

// the 3 G coordinates of group g of a cluster of n atoms at x (vec: words by
// which a group's address is aligned); far positions for missing atoms
template <int G, typename IO>
__device__ __forceinline__ void load_group(const IO* __restrict__ x, int n, int g, int vec,
                                           float (&q)[3 * G]) {
  const IO* p = x + 3 * G * g;
  if (sizeof(IO) == 4 && vec == 4 && G * g + G <= n) {
#pragma unroll
    for (int v = 0; v < 3 * G / 4; ++v) {
      const float4 w = reinterpret_cast<const float4*>(p)[v];
      q[4 * v] = w.x; q[4 * v + 1] = w.y; q[4 * v + 2] = w.z; q[4 * v + 3] = w.w;
    }
  } else if (sizeof(IO) == 4 && vec >= 2 && G * g + G <= n) {
#pragma unroll
    for (int v = 0; v < 3 * G / 2; ++v) {
      const float2 w = reinterpret_cast<const float2*>(p)[v];
      q[2 * v] = w.x; q[2 * v + 1] = w.y;
    }
  } else {
#pragma unroll
    for (int a = 0; a < G; ++a) {
      const int i = G * g + a;
      if (i < n) {
        q[3 * a] = (float)p[3 * a];
        q[3 * a + 1] = (float)p[3 * a + 1];
        q[3 * a + 2] = (float)p[3 * a + 2];
      } else {
        const float f = kFarAtom * (float)(1 + (i - n));
        q[3 * a] = f; q[3 * a + 1] = f; q[3 * a + 2] = f;
      }
    }
  }
}

template <int G, typename IO>
__device__ __forceinline__ void store_group(IO* __restrict__ x, int n, int g, int vec,
                                            const float (&q)[3 * G]) {
  IO* p = x + 3 * G * g;
  if (sizeof(IO) == 4 && vec == 4 && G * g + G <= n) {
#pragma unroll
    for (int v = 0; v < 3 * G / 4; ++v)
      reinterpret_cast<float4*>(p)[v] = make_float4(q[4 * v], q[4 * v + 1], q[4 * v + 2],
                                                    q[4 * v + 3]);
  } else if (sizeof(IO) == 4 && vec >= 2 && G * g + G <= n) {
#pragma unroll
    for (int v = 0; v < 3 * G / 2; ++v)
      reinterpret_cast<float2*>(p)[v] = make_float2(q[2 * v], q[2 * v + 1]);
  } else {
#pragma unroll
    for (int a = 0; a < G; ++a) {
      if (G * g + a < n) {
        p[3 * a] = (IO)q[3 * a];
        p[3 * a + 1] = (IO)q[3 * a + 1];
        p[3 * a + 2] = (IO)q[3 * a + 2];
      }
    }
  }
}

// the own group: atoms 2h and 2h + 1 in the two lanes of operand h, so that no
// coordinate or force of the own atoms is held twice; the partner's atoms come
// from shared memory in both lanes
template <int G>
struct Own {
  V2 f[G / 2];
};
template <int G>
__device__ __forceinline__ void own_zero(Own<G>& o) {
#pragma unroll
  for (int h = 0; h < G / 2; ++h) o.f[h] = v2_zero();
}
template <bool ADD, int G>
__device__ __forceinline__ void own_add(Own<G>& o, const Own<G>& r) {
  // f + s r by one FMA: exact product
#pragma unroll
  for (int h = 0; h < G / 2; ++h) v2_fma(o.f[h], f2(ADD ? 1.f : -1.f), r.f[h]);
}
template <int G>
__device__ __forceinline__ void own_slot(Own<G>& o, const SlotF<G>& r) {
#pragma unroll
  for (int v = 0; v < G / 4; ++v) {
    const float4 x = reinterpret_cast<const float4*>(r.x)[v];
    const float4 y = reinterpret_cast<const float4*>(r.y)[v];
    const float4 z = reinterpret_cast<const float4*>(r.z)[v];
    v2_add(o.f[2 * v], V2{make_float2(x.x, x.y), make_float2(y.x, y.y), make_float2(z.x, z.y)});
    v2_add(o.f[2 * v + 1],
           V2{make_float2(x.z, x.w), make_float2(y.z, y.w), make_float2(z.z, z.w)});
  }
}
template <int G>
__device__ __forceinline__ void own_write(const Own<G>& o, SlotF<G>& w) {
#pragma unroll
  for (int v = 0; v < G / 4; ++v) {
    const V2 &a = o.f[2 * v], &b = o.f[2 * v + 1];
    reinterpret_cast<float4*>(w.x)[v] = make_float4(a.x.x, a.x.y, b.x.x, b.x.y);
    reinterpret_cast<float4*>(w.y)[v] = make_float4(a.y.x, a.y.y, b.y.x, b.y.y);
    reinterpret_cast<float4*>(w.z)[v] = make_float4(a.z.x, a.z.y, b.z.x, b.z.y);
  }
}
template <int G>
__device__ __forceinline__ void own_scaled(const Own<G>& o, float gs, float (&w)[3 * G]) {
#pragma unroll
  for (int h = 0; h < G / 2; ++h) {
    w[6 * h] = gs * o.f[h].x.x; w[6 * h + 1] = gs * o.f[h].y.x; w[6 * h + 2] = gs * o.f[h].z.x;
    w[6 * h + 3] = gs * o.f[h].x.y; w[6 * h + 4] = gs * o.f[h].y.y; w[6 * h + 5] = gs * o.f[h].z.y;
  }
}
template <int G>
__device__ __forceinline__ void put_pos(PosRing<G>& r, const float (&q)[3 * G]) {
#pragma unroll
  for (int j = 0; j < G; ++j)
    r.xy[j] = make_float4(q[3 * j], q[3 * j], q[3 * j + 1], q[3 * j + 1]);
#pragma unroll
  for (int j = 0; j < G; j += 2)
    r.zz[j / 2] = make_float4(q[3 * j + 2], q[3 * j + 2], q[3 * j + 5], q[3 * j + 5]);
}
template <int G>
__device__ __forceinline__ void get_pos(const PosRing<G>& r, float (&q)[3 * G]) {
#pragma unroll
  for (int j = 0; j < G; ++j) {
    q[3 * j] = r.xy[j].x;
    q[3 * j + 1] = r.xy[j].z;
    q[3 * j + 2] = j & 1 ? r.zz[j / 2].z : r.zz[j / 2].x;
  }
}
// atom j of a record, in both lanes
template <int G>
__device__ __forceinline__ V2 partner(const PosRing<G>& rb, int j, const float4& zz) {
  const float4 xy = rb.xy[j];
  return V2{make_float2(xy.x, xy.y), make_float2(xy.z, xy.w),
            j & 1 ? make_float2(zz.z, zz.w) : make_float2(zz.x, zz.y)};
}

// the pairs inside a group: operand h with the atoms above 2h + 1 (from the own
// record), and the pairs (2h, 2h + 1) of two operands at a time
template <int G, int POT, bool SIG>
__device__ __forceinline__ void intra(const V2 (&N)[G / 2], const PosRing<G>& own, const RingK& k,
                                      Own<G>& o, E2& e) {
  float2 eb[2] = {f2(0.f), f2(0.f)};
#pragma unroll
  for (int j = 2; j < G; ++j) {
    const V2 b = partner(own, j, own.zz[j / 2]);
    V2 r;
#pragma unroll
    for (int h = 0; h < j / 2; ++h) {
      V2 d;
      float2 c;
      ring_op<POT, SIG>(N[h], b, k, d, c, eb[G > 4 ? j & 1 : 0]);
      if (h == 0) r = v2_scale(c, d);
      else v2_fma(r, c, d);
      v2_fma(o.f[h], c, d);
    }
    V2& f = o.f[j / 2];
    if (j & 1) {
      f.x.y -= r.x.x + r.x.y; f.y.y -= r.y.x + r.y.y; f.z.y -= r.z.x + r.z.y;
    } else {
      f.x.x -= r.x.x + r.x.y; f.y.x -= r.y.x + r.y.y; f.z.x -= r.z.x + r.z.y;
    }
  }
#pragma unroll
  for (int h = 0; h < G / 2; h += 2) {
    const V2 &A = N[h], &B = N[h + 1];
    V2 d;
    float2 c;
    ring_op<POT, SIG>(V2{make_float2(A.x.x, B.x.x), make_float2(A.y.x, B.y.x),
                         make_float2(A.z.x, B.z.x)},
                      V2{make_float2(-A.x.y, -B.x.y), make_float2(-A.y.y, -B.y.y),
                         make_float2(-A.z.y, -B.z.y)},
                      k, d, c, eb[G > 4 ? h / 2 & 1 : 0]);
    const V2 r = v2_scale(c, d);
    v2_add(o.f[h], V2{make_float2(r.x.x, -r.x.x), make_float2(r.y.x, -r.y.x),
                      make_float2(r.z.x, -r.z.x)});
    v2_add(o.f[h + 1], V2{make_float2(r.x.y, -r.x.y), make_float2(r.y.y, -r.y.y),
                          make_float2(r.z.y, -r.z.y)});
  }
  e2_acc(e, G > 4 ? __fadd2_rn(eb[0], eb[1]) : eb[0]);
}

// one shift: the G^2 pairs (a split shift: half of them) of the own group,
// negated in N, with the partner's record; its reaction goes to w.  Energies
// are summed in FP32 over four (G = 8: eight) pairs a lane, two such sums at a
// time, then in double-float.
template <int G, int POT, bool SIG>
__device__ __forceinline__ void shift(const V2 (&N)[G / 2], const PosRing<G>& rb, bool split,
                                      bool lower, const RingK& k, Own<G>& o, E2& e,
                                      SlotF<G>& w) {
  float px[4], py[4], pz[4];               // reactions on four of the partner's atoms
  auto fold = [&](int j, const V2& r) {
    px[j & 3] = __fadd_rn(r.x.x, r.x.y);
    py[j & 3] = __fadd_rn(r.y.x, r.y.y);
    pz[j & 3] = __fadd_rn(r.z.x, r.z.y);
  };
  auto put = [&](int v) {
    reinterpret_cast<float4*>(w.x)[v] = make_float4(px[0], px[1], px[2], px[3]);
    reinterpret_cast<float4*>(w.y)[v] = make_float4(py[0], py[1], py[2], py[3]);
    reinterpret_cast<float4*>(w.z)[v] = make_float4(pz[0], pz[1], pz[2], pz[3]);
  };
  if (!split) {
    float4 zz;
    float2 eb[2] = {f2(0.f), f2(0.f)};
#pragma unroll
    for (int j = 0; j < G; ++j) {
      if (!(j & 1)) zz = rb.zz[j / 2];
      const V2 b = partner(rb, j, zz);
      V2 r;
#pragma unroll
      for (int h = 0; h < G / 2; ++h) {
        V2 d;
        float2 c;
        ring_op<POT, SIG>(N[h], b, k, d, c, eb[h & 1]);
        if (h == 0) r = v2_scale(c, d);
        else v2_fma(r, c, d);
        v2_fma(o.f[h], c, d);
      }
      fold(j, r);
      if ((j & 3) == 3) {
        put(j / 4);
        e2_acc(e, __fadd2_rn(eb[0], eb[1]));
        eb[0] = eb[1] = f2(0.f);
      }
    }
  } else if constexpr (G == 4) {
    // lower thread a0, a1 with b0 .. b3, upper thread a0 .. a3 with b2, b3
    V2 r[4];
    float2 eb = f2(0.f);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = lower ? u : 2 + (u >> 1);
      const float4 zz = rb.zz[j >> 1];
      const V2 b = partner(rb, j, zz);
      V2 d;
      float2 c;
      ring_op<POT, SIG>(lower || !(u & 1) ? N[0] : N[1], b, k, d, c, eb);
      r[u] = v2_scale(c, d);
    }
    v2_add(o.f[0], r[0]);
    v2_add(o.f[0], r[2]);
    if (lower) {
      v2_add(o.f[0], r[1]);
      v2_add(o.f[0], r[3]);
#pragma unroll
      for (int u = 0; u < 4; ++u) fold(u, r[u]);
    } else {
      v2_add(o.f[1], r[1]);
      v2_add(o.f[1], r[3]);
      fold(0, v2_zero());
      fold(1, v2_zero());
      v2_add(r[0], r[1]);
      fold(2, r[0]);
      v2_add(r[2], r[3]);
      fold(3, r[2]);
    }
    put(0);
    e2_acc(e, eb);
  } else {
    // lower thread the lower half of its atoms with all of b, upper thread all
    // of its atoms with the upper half of b
    const int j0 = lower ? 0 : G / 2;
    if (!lower) {
#pragma unroll
      for (int j = 0; j < 4; ++j) fold(j, v2_zero());
#pragma unroll
      for (int v = 0; v < G / 8; ++v) put(v);
    }
#pragma unroll 1
    for (int j = j0; j < G; j += 4) {
      float2 eb[2] = {f2(0.f), f2(0.f)};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const V2 b = partner(rb, j + u, rb.zz[(j + u) / 2]);
        V2 r = v2_zero();
#pragma unroll
        for (int h = 0; h < G / 2; ++h) {
          if (lower && h >= G / 4) continue;
          V2 d;
          float2 c;
          ring_op<POT, SIG>(N[h], b, k, d, c, eb[h & 1]);
          v2_fma(r, c, d);
          v2_fma(o.f[h], c, d);
        }
        fold(u, r);
      }
      put(j / 4);
      e2_acc(e, __fadd2_rn(eb[0], eb[1]));
    }
  }
}

// ---------------------------------------------------------------------------
// FP64: scalar operations, G atoms a group.  The FP64 unit of an SM
// sub-partition takes a warp's instruction every 67 cycles if its operands are
// registers and every 80 if one is a constant (measured), whatever its active
// lanes: `one` is 1.0 kept in a register.
// ---------------------------------------------------------------------------
// pair (x, y): f += c (y - x) on x, p += c (y - x) to be subtracted on y, e +=
// the pair's energy (units and signs as in ring_op); LJ: k0 = sigma^2;
// Morse: k0 = rho, k1 = rho / re
template <int POT, bool SIG>
__device__ __forceinline__ void ringd_op(double ax, double ay, double az, double bx, double by,
                                         double bz, double one, double k0, double k1, double& fx,
                                         double& fy, double& fz, double& px, double& py,
                                         double& pz, double& e) {
  const double dx = bx - ax, dy = by - ay, dz = bz - az;
  const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
  double c;
  if constexpr (POT == LJ_POT_LJ) {
    double s2 = rcp_f64(r2, one);
    if constexpr (SIG) s2 *= k0;
    const double s6 = s2 * s2 * s2;
    const double t = s6 - one;
    e = fma(s6, t, e);
    c = (s2 * s6) * (s6 + t);
  } else {
    // an ulp of r is rho ulps of m: r is the correctly rounded root.  A reciprocal
    // root within an ulp for both r and 1 / r made gradients 1.5 times less exact
    const double r = sqrt(r2);
    const double m = exp(fma(-k1, r, k0));
    const double term = m * (m - 2.0);
    e += r2 > 0.0 ? term : __longlong_as_double(0x7ff0000000000000LL);
    c = m * (m - 1.0) / r;
  }
  fx = fma(c, dx, fx); fy = fma(c, dy, fy); fz = fma(c, dz, fz);
  px = fma(c, dx, px); py = fma(c, dy, py); pz = fma(c, dz, pz);
}

template <int G>
struct GroupD {
  double x[G], y[G], z[G];
};
template <int G>
__device__ __forceinline__ void group_zero(GroupD<G>& q) {
#pragma unroll
  for (int a = 0; a < G; ++a) { q.x[a] = 0.0; q.y[a] = 0.0; q.z[a] = 0.0; }
}

template <int G, typename IO>
__device__ __forceinline__ void load_group_d(const IO* __restrict__ x, int n, int g, GroupD<G>& q) {
#pragma unroll
  for (int a = 0; a < G; ++a) {
    const int i = G * g + a;
    if (i < n) {
      q.x[a] = (double)x[3 * i]; q.y[a] = (double)x[3 * i + 1]; q.z[a] = (double)x[3 * i + 2];
    } else {
      const double f = 0x1p300 * (double)(1 + (i - n));   // far: terms underflow to 0
      q.x[a] = f; q.y[a] = f; q.z[a] = f;
    }
  }
}

// Energies: four pairs at most in FP64, then double-double; Morse, whose exponential
// makes the rest cheap, pair by pair.
template <int POT>
__device__ __forceinline__ void fold_d(dd& e, double& eb, bool block) {
  if (POT != LJ_POT_LJ || block) {
    dd_acc(e, eb);
    eb = 0.0;
  }
}

template <int G, int POT, bool SIG>
__device__ __forceinline__ void intra_d(const GroupD<G>& q, double one, double k0, double k1,
                                        GroupD<G>& f, dd& e) {
  double eb = 0.0;
#pragma unroll
  for (int i = 0; i < G; ++i)
#pragma unroll
    for (int j = i + 1; j < G; ++j) {
      double px = 0, py = 0, pz = 0;
      ringd_op<POT, SIG>(q.x[i], q.y[i], q.z[i], q.x[j], q.y[j], q.z[j], one, k0, k1, f.x[i],
                         f.y[i], f.z[i], px, py, pz, eb);
      fold_d<POT>(e, eb, j == G - 1 && (G > 3 && i == 0 || i == G - 2));
      f.x[j] -= px; f.y[j] -= py; f.z[j] -= pz;
    }
}

template <int G, int POT, bool SIG>
__device__ __forceinline__ void shift_d(const GroupD<G>& q, const PosDG<G>& rb, bool split,
                                        bool lower, double one, double k0, double k1, GroupD<G>& f,
                                        dd& e, PosDG<G>& w) {
  GroupD<G> p;
  group_zero(p);
  double eb = 0.0;
  if (!split) {
#pragma unroll
    for (int j = 0; j < G; ++j)
#pragma unroll
      for (int i = 0; i < G; ++i) {
        ringd_op<POT, SIG>(q.x[i], q.y[i], q.z[i], rb.x[j], rb.y[j], rb.z[j], one, k0, k1, f.x[i],
                           f.y[i], f.z[i], p.x[j], p.y[j], p.z[j], eb);
        fold_d<POT>(e, eb, i == G - 1 && (G > 2 || j == G - 1));
      }
  } else {
    // lower thread the lower half of its atoms with all of b, upper thread
    // all of its atoms with the upper half of b
#pragma unroll
    for (int j = 0; j < G; ++j)
#pragma unroll
      for (int i = 0; i < G; ++i)
        if (lower ? i < G / 2 : j >= G / 2) {
          ringd_op<POT, SIG>(q.x[i], q.y[i], q.z[i], rb.x[j], rb.y[j], rb.z[j], one, k0, k1,
                             f.x[i], f.y[i], f.z[i], p.x[j], p.y[j], p.z[j], eb);
          fold_d<POT>(e, eb, i == (lower ? G / 2 : G) - 1 && (G > 2 || j == G - 1));
        }
  }
#pragma unroll
  for (int j = 0; j < G; ++j) { w.x[j] = p.x[j]; w.y[j] = p.y[j]; w.z[j] = p.z[j]; }
}

}  // namespace ljr
