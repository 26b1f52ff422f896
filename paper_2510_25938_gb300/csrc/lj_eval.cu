// lj_eval.cu -- lj_energy_grad_batched: batched energy + gradient of Eq. (1)
// and of the Morse pair potential, in the ring layout of lj_ring.cuh (every
// unordered pair once) for every batch shape.
#include <algorithm>

#include "lj_internal.h"
#include "lj_ring.cuh"

namespace {

using namespace ljd;
using namespace ljr;

// ---- FP32 --------------------------------------------------------------------
// PACKED: C candidates a CTA, one part each, all H shifts before one barrier
// (large uniform batches of small clusters).  PACKED_UNEVEN: the same, every
// candidate with the threads of the largest; a variant of its own, since its
// sizes and bounds cost PACKED 6% (65,536 x LJ38: 61.1 against 57.4 us).
// MULTI_PART: any batch.
enum RingMode { PACKED, PACKED_UNEVEN, MULTI_PART };
template <int G, typename IO, int POT, bool SIG, int MODE>
__global__ void __launch_bounds__(256, 2) eval_ring_f32_kernel(ljh::EvalArgs a, RingPlan pl) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr bool MULTI = MODE == MULTI_PART, UNEVEN = MODE == PACKED_UNEVEN;
  const int B = blockDim.x, tid = threadIdx.x;
  const int S = MULTI ? pl.S : 1, KS = pl.KS;
  PosRing<G>* pos = reinterpret_cast<PosRing<G>*>(smem);
  SlotF<G>* react = reinterpret_cast<SlotF<G>*>(pos + B);
  SlotF<G>* own = react + (size_t)KS * B;
  const bool parts_buf = MULTI && (pl.P > 1 || S > 1);
  ff* es = reinterpret_cast<ff*>(own + (parts_buf ? B : 0));
  ff* ecl = reinterpret_cast<ff*>(reinterpret_cast<unsigned char*>(es) + (size_t)B * 16);
  const RingK k = POT == LJ_POT_LJ ? RingK{a.k.sig2_f, 0.f, 0.f}
                                   : RingK{-a.k.re_f, -a.k.m_slope2_f, -a.k.m_slope2_lo};
  const float gs = POT == LJ_POT_LJ ? a.k.gscale_f : a.k.m_g_f;
  const double ef = POT == LJ_POT_LJ ? a.k.e4 : a.k.eps;
  const IO* __restrict__ xin = static_cast<const IO*>(a.x);
  IO* __restrict__ gout = static_cast<IO*>(a.grad);
  const int srank = MULTI && S > 1 ? (int)(blockIdx.x % S) : 0;
  const long long stride = (long long)(gridDim.x / S) * pl.C;

  int n = a.uniform_n;
  int NG = (n + G - 1) / G, H = NG >> 1, P = 1, lc = 0, p = 0, g = 0;
  auto place = [&]() {                 // this thread's candidate of the tile, part and group
    const int per = NG * P;
    lc = per > 0 ? tid / per : pl.C;
    const int rem = tid - lc * per;
    p = P > 1 ? rem / NG : 0;
    g = rem - p * NG;
  };
  const int NS = UNEVEN ? (a.max_n + G - 1) / G : NG;   // packed: threads of a candidate
  if (UNEVEN) {
    lc = tid / NS;
    g = tid - lc * NS;
  } else if (a.uniform_n > 0) {
    P = MULTI ? pl.P : 1;
    place();
  }
  for (long long c0 = (long long)(blockIdx.x / S) * pl.C; c0 < a.n_cand; c0 += stride) {
    long long a0;
    bool bad = false;
    if (MODE == PACKED || (MULTI && a.uniform_n > 0)) {
      a0 = (c0 + lc) * n;
    } else if (UNEVEN) {
      n = 0;
      a0 = 0;
      if (lc < pl.C && c0 + lc < a.n_cand) {
        a0 = a.off[c0 + lc];
        const long long na = a.off[c0 + lc + 1] - a0;
        bad = na > a.max_n || na < 0;
        n = bad ? 0 : (int)na;
      }
      NG = (n + G - 1) / G;
      H = NG >> 1;
    } else {
      a0 = a.off[c0];
      n = (int)(a.off[c0 + 1] - a0);
      if (n > a.max_n || n < 0) {
        if (tid == 0 && srank == 0) a.energy[c0] = __longlong_as_double(0x7ff8000000000000LL);
        continue;
      }
      NG = (n + G - 1) / G;
      H = NG >> 1;
      P = NG > 0 ? max(1, min(B / NG, (H + S - 1) / S + 1)) : 1;
      place();
    }
    const bool here = lc < pl.C && c0 + lc < a.n_cand;
    const bool live = here && (!UNEVEN || g < NG);
    const int slot = UNEVEN ? lc * NS : (lc * P + p) * NG;  // first slot of this candidate's part
    const int pslot = UNEVEN ? slot : lc * NG;              // its first position record
    V2 N[G / 2];                             // own atoms, negated
    {
      float q[3 * G];
      if (live && p == 0) {
        load_group<G>(xin + 3 * a0, n, g, pl.vec, q);
        put_pos(pos[pslot + g], q);
      }
      __syncthreads();
      if (MULTI && live && p > 0) get_pos(pos[pslot + g], q);
#pragma unroll
      for (int h = 0; h < G / 2; ++h)
        N[h] = V2{make_float2(-q[6 * h], -q[6 * h + 3]), make_float2(-q[6 * h + 1], -q[6 * h + 4]),
                  make_float2(-q[6 * h + 2], -q[6 * h + 5])};
    }
    E2 e{f2(0.f), f2(0.f)};
    Own<G> o, tot;
    own_zero(o);
    own_zero(tot);
    const int GP = MULTI ? S * P : 1, gp = MULTI ? srank * P + p : 0;
    // the pairs inside the groups go to the last part, which has no more
    // shifts than any other
    if (live && gp == GP - 1) intra<G, POT, SIG>(N, pos[pslot + g], k, o, e);
    const bool even = (NG & 1) == 0;
    for (int kc = 0; kc * GP < H || kc == 0; kc += KS) {
      if (kc > 0) __syncthreads();           // the last chunk's readers are done
      if (live) {
        for (int s = 0; s < KS; ++s) {
          const int sh = 1 + (kc + s) * GP + gp;
          if (sh > H) break;
          int t = g + sh;
          if (t >= NG) t -= NG;
          shift<G, POT, SIG>(N, pos[pslot + t], even && sh == H, g < H, k, o, e,
                             react[s * B + slot + t]);
        }
        if (!UNEVEN) es[tid] = e2_total(e);
      }
      // zeros from a candidate's idle threads, NaN for a bad size
      if (UNEVEN && here) es[tid] = bad && g == 0 ? ff{__int_as_float(0x7fc00000), 0.f} : e2_total(e);
      __syncthreads();
      // forces are summed in parts -- the reactions by themselves, then (several
      // chunks) chunk by chunk -- and not in one FP32 sum over all atoms, whose error
      // grows with their number (1,024 x 500 atoms: 5.5e-7 of the gradient so, 4.2e-7 in
      // parts; 111 and 115 us with the energies' blocks)
      if (live && (MULTI || gout)) {
        Own<G> r;
        own_zero(r);
        for (int s = 0; s < KS; ++s) {
          if (1 + (kc + s) * GP + gp > H) break;
          own_slot(r, react[s * B + slot + g]);
        }
        own_add<false>(o, r);
      }
      if (!MULTI) break;
      own_add<true>(tot, o);
      own_zero(o);
    }
    if (MULTI) o = tot;
    if (MULTI && P > 1) {                    // parts in the order of p
      if (live && p > 0) own_write(o, own[slot + g]);
      __syncthreads();
      if (live && p == 0)
        for (int pp = 1; pp < P; ++pp) own_slot(o, own[slot + pp * NG + g]);
    }
    if (tid < 32)
      sum_energies(es, pl.C, UNEVEN ? NS : NG * P, [&](int c, ff s) {
        if (MULTI && S > 1) ecl[c] = s;
        else if (c0 + c < a.n_cand) a.energy[c0 + c] = total(s) * ef;
      });
    if (MULTI && S > 1) {                    // CTAs of the cluster in the order of s
      cg::cluster_group cl = cg::this_cluster();
      if (live && p == 0) own_write(o, own[slot + g]);
      cl.sync();
      own_zero(o);
      if (live && p == 0 && g % S == srank)
        for (int s = 0; s < S; ++s) own_slot(o, *cl.map_shared_rank(&own[slot + g], s));
      if (srank == 0 && tid < pl.C && c0 + tid < a.n_cand) {
        ff s = ecl[tid];
        for (int r = 1; r < S; ++r) acc_pair(s, *cl.map_shared_rank(&ecl[tid], r));
        a.energy[c0 + tid] = total(s) * ef;
      }
      cl.sync();
    }
    if (live && gout && p == 0 && (!MULTI || S == 1 || g % S == srank)) {
      float w[3 * G];
      own_scaled(o, gs, w);
      store_group<G>(gout + 3 * a0, n, g, pl.vec, w);
    }
    // the next tile writes `es`, `react` and `own` after its first barrier
  }
}

// ---- FP64 --------------------------------------------------------------------
template <int G, typename IO, int POT, bool SIG>
__global__ void __launch_bounds__(256, POT == LJ_POT_LJ ? 2 : 1) eval_ring_f64_kernel(ljh::EvalArgs a, RingPlan pl) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int B = blockDim.x, tid = threadIdx.x;
  const int S = pl.S, KS = pl.KS;
  PosDG<G>* pos = reinterpret_cast<PosDG<G>*>(smem);
  PosDG<G>* react = pos + B;
  PosDG<G>* own = react + (size_t)KS * B;
  dd* es = reinterpret_cast<dd*>(own + (pl.P > 1 || S > 1 ? B : 0));
  dd* ecl = es + B;
  const double k0 = POT == LJ_POT_LJ ? a.k.sig2 : a.k.rho;
  const double k1 = POT == LJ_POT_LJ ? 0.0 : a.k.rho_re;
  double one = 1.0;
  asm volatile("" : "+d"(one));              // a register, not a constant
  const double gs = POT == LJ_POT_LJ ? a.k.gscale : a.k.m_g;
  const double ef = POT == LJ_POT_LJ ? a.k.e4 : a.k.eps;
  const IO* __restrict__ xin = static_cast<const IO*>(a.x);
  IO* __restrict__ gout = static_cast<IO*>(a.grad);
  const int srank = S > 1 ? (int)(blockIdx.x % S) : 0;
  const long long stride = (long long)(gridDim.x / S) * pl.C;

  int n = a.uniform_n;
  int NG = (n + G - 1) / G, H = NG >> 1, P = pl.P, lc = 0, p = 0, g = 0;
  auto place = [&]() {
    const int per = NG * P;
    lc = per > 0 ? tid / per : pl.C;
    const int rem = tid - lc * per;
    p = P > 1 ? rem / NG : 0;
    g = rem - p * NG;
  };
  if (a.uniform_n > 0) place();
  for (long long c0 = (long long)(blockIdx.x / S) * pl.C; c0 < a.n_cand; c0 += stride) {
    long long a0;
    if (a.uniform_n > 0) {
      a0 = (c0 + lc) * n;
    } else {
      a0 = a.off[c0];
      n = (int)(a.off[c0 + 1] - a0);
      if (n > a.max_n || n < 0) {
        if (tid == 0 && srank == 0) a.energy[c0] = __longlong_as_double(0x7ff8000000000000LL);
        continue;
      }
      NG = (n + G - 1) / G;
      H = NG >> 1;
      P = NG > 0 ? max(1, min(B / NG, (H + S - 1) / S + 1)) : 1;
      place();
    }
    const bool live = lc < pl.C && c0 + lc < a.n_cand;
    const int slot = (lc * P + p) * NG;
    const int pslot = lc * NG;
    GroupD<G> q, f;
    group_zero(q);
    group_zero(f);
    if (live && p == 0) {
      load_group_d(xin + 3 * a0, n, g, q);
      PosDG<G>& r = pos[pslot + g];
#pragma unroll
      for (int j = 0; j < G; ++j) { r.x[j] = q.x[j]; r.y[j] = q.y[j]; r.z[j] = q.z[j]; }
    }
    __syncthreads();
    if (live && p > 0) {
      const PosDG<G>& r = pos[pslot + g];
#pragma unroll
      for (int j = 0; j < G; ++j) { q.x[j] = r.x[j]; q.y[j] = r.y[j]; q.z[j] = r.z[j]; }
    }
    dd e{0.0, 0.0};
    const int GP = S * P, gp = srank * P + p;
    if (live && gp == GP - 1) intra_d<G, POT, SIG>(q, one, k0, k1, f, e);
    const bool even = (NG & 1) == 0;
    for (int kc = 0; kc * GP < H || kc == 0; kc += KS) {
      if (kc > 0) __syncthreads();
      if (live) {
        for (int s = 0; s < KS; ++s) {
          const int k = 1 + (kc + s) * GP + gp;
          if (k > H) break;
          int t = g + k;
          if (t >= NG) t -= NG;
          shift_d<G, POT, SIG>(q, pos[pslot + t], even && k == H, g < H, one, k0, k1, f, e,
                               react[s * B + slot + t]);
        }
        es[tid] = e;
      }
      __syncthreads();
      if (live) {
        for (int s = 0; s < KS; ++s) {
          if (1 + (kc + s) * GP + gp > H) break;
          const PosDG<G>& r = react[s * B + slot + g];
#pragma unroll
          for (int j = 0; j < G; ++j) { f.x[j] -= r.x[j]; f.y[j] -= r.y[j]; f.z[j] -= r.z[j]; }
        }
      }
    }
    if (P == 1 && S == 1) {
      if (live && gout) {
        IO* go = gout + 3 * a0;
#pragma unroll
        for (int j = 0; j < G; ++j) {
          const int i = G * g + j;
          if (i < n) {
            go[3 * i] = (IO)(gs * f.x[j]);
            go[3 * i + 1] = (IO)(gs * f.y[j]);
            go[3 * i + 2] = (IO)(gs * f.z[j]);
          }
        }
      }
      if (tid < 32)
        sum_energies(es, pl.C, NG, [&](int c, dd s) {
          if (c0 + c < a.n_cand) a.energy[c0 + c] = total(s) * ef;
        });
      continue;
    }
    // parts in the order of p, then CTAs in the order of s, one coordinate a
    // thread (C = 1 here); the energies by the last warp meanwhile
    if (live) {
      PosDG<G>& w = own[slot + g];
#pragma unroll
      for (int j = 0; j < G; ++j) { w.x[j] = f.x[j]; w.y[j] = f.y[j]; w.z[j] = f.z[j]; }
    }
    __syncthreads();
    constexpr int D = sizeof(PosDG<G>) / sizeof(double);   // doubles a slot, 3 G used
    double* od = reinterpret_cast<double*>(own);
    const long long first = a.uniform_n > 0 ? c0 * n : a0;   // of any thread, live or not
    auto out = [&](int o, double v) {        // coordinate o: group, axis, atom of the group
      const int i = G * (o / (3 * G)) + o % G, ax = o % (3 * G) / G;
      if (gout && i < n) gout[3 * (first + i) + ax] = (IO)(gs * v);
    };
    for (int o = tid; o < 3 * G * NG; o += B) {
      double* q0 = od + (o / (3 * G)) * D + o % (3 * G);
      double v = *q0;
      for (int pp = 1; pp < P; ++pp) v += q0[(size_t)pp * NG * D];
      if (S == 1) out(o, v);
      else *q0 = v;
    }
    if (tid >= B - 32)
      sum_energies(es, 1, NG * P, [&](int, dd s) {
        if (S > 1) ecl[0] = s;
        else a.energy[c0] = total(s) * ef;
      });
    if (S > 1) {
      cg::cluster_group cl = cg::this_cluster();
      cl.sync();
      for (int o = tid; o < 3 * G * NG; o += B) {
        if (o / (3 * G) % S != srank) continue;
        double* q0 = od + (o / (3 * G)) * D + o % (3 * G);
        double v = 0.0;
        for (int s = 0; s < S; ++s) v += *cl.map_shared_rank(q0, s);
        out(o, v);
      }
      if (srank == 0 && tid == 0) {
        dd s = ecl[0];
        for (int r = 1; r < S; ++r) acc_pair(s, *cl.map_shared_rank(&ecl[0], r));
        a.energy[c0] = total(s) * ef;
      }
      cl.sync();
    }
  }
}

// ---- launch ------------------------------------------------------------------
constexpr int kRingMaxB = 256;                // largest CTA of both kernels
constexpr size_t kRingSmem = 104 * 1024;      // shared memory that lets two CTAs share an SM
constexpr int kUnevenPackedH = 8;             // most shifts of a packed uneven cluster (68 atoms)

struct RingLaunch {
  RingPlan pl;
  int G;           // atoms a group
  int B;           // threads per CTA
  bool multi;      // FP32: the general kernel
};

// FP32: shifts whose reactions fit in 444 bytes a thread (227 KB for 512
// threads), after the position record, the energy and the parts' slot
constexpr int ring_most_ks(int G, bool parts) {
  return (444 - 16 - (24 * G + 16)) / (12 * G) - (parts ? 1 : 0);
}
static_assert(ring_most_ks(8, false) == 2 && ring_most_ks(4, true) == 5, "shifts per chunk");

// Relative time of a uniform batch of n_cand clusters of n atoms on `sms` SMs:
// operations of one thread times the warps that a scheduler gets, which is
// never less than `floor` (a single warp waits for its own chain) and ends in an
// uneven tail.  An SM gets whole CTAs, so their number is rounded up: 75 large CTAs on
// 152 SMs take as long as 152 would.  The weights are fitted to 118 shapes (2 to
// 1,000 atoms, 1 to 65,536 clusters), each in up to 80 layouts: the layout of the
// least modelled time takes 2% more than the best measured one in the geometric
// mean, 14% at most.  (A fixed threshold between packed and split batches left up to
// half of the SMs or 31 of 32 lanes idle beside it: 5,000 x 4 atoms FP64 47 us, now 9;
// 30,000 x 2 FP32 33, 6; 150 x 300 FP64 734, 365.)
double ring_time(bool fp32, int n, long long n_cand, int sms, const RingLaunch& r) {
  const int G = r.G, NG = (n + G - 1) / G, H = NG / 2, parts = r.pl.P * r.pl.S;
  const bool one = parts == 1;
  const int k = (H + parts - 1) / parts;               // shifts of a thread
  double ops;
  if (fp32) {                                          // packed instructions
    const double half = one && H > 0 && !(NG & 1) && G == 4 ? 0.5 : 0.0;   // the split shift
    ops = (k - half) * (9.5 * G * G + 7.0 * G + 12) + (one ? 4.75 * G * G : 0.0) + 36.0 * G + 90;
    if (r.multi) ops = 1.1 * ops + 300;
    ops += (r.pl.P > 1 ? 200 : 0) + (r.pl.S > 1 ? 500 + 200 * r.pl.S : 0);
  } else {                                             // FP64 instructions
    ops = k * (25.0 * G * G + 20.0 * G) + 50 + (one ? 12.5 * G * (G - 1) : 0.0);
    ops = ops * (G == 2 ? 1.0 : G == 3 ? 1.15 : 1.25) + (one ? 0 : 100) + (r.pl.S > 1 ? 200 : 0);
  }
  const long long ctas = (n_cand + r.pl.C - 1) / r.pl.C * r.pl.S;
  const double warps = (double)((ctas + sms - 1) / sms) * r.B / 128;   // of a scheduler
  return ops * (fp32 ? std::max(3.0, warps) + 0.6 : std::max(1.0, warps) + 0.2);
}

RingLaunch ring_plan(const ljh::EvalArgs& a, int sms) {
  RingLaunch r;
  const int n = a.uniform_n > 0 ? a.uniform_n : a.max_n;
  const bool fp32 = a.prec != LJ_PREC_FP64;
  r.pl = RingPlan{1, 1, 1, 1, 1};
  RingPlan& pl = r.pl;
  r.multi = true;
  // the smallest group that fits a CTA; large batches may take a larger one
  r.G = fp32 ? 4 : n <= 2 * kRingMaxB ? 2 : n <= 3 * kRingMaxB ? 3 : 4;
  int NG = (n + r.G - 1) / r.G;
  if (a.uniform_n > 0) {
    RingLaunch best = r;
    double least = 0.0;
    auto consider = [&](int G, int C, int P, int S, int B, bool multi) {
      RingLaunch o = r;
      o.G = G;
      o.B = B;
      o.multi = multi;
      o.pl.C = C;
      o.pl.P = P;
      o.pl.S = S;
      const double t = ring_time(fp32, n, a.n_cand, sms, o);
      if (least == 0.0 || t < least || (t == least && B < best.B)) {
        least = t;
        best = o;
      }
    };
    // one part, several candidates a CTA (FP32: of 64 threads; larger ones were never
    // more than 1% faster, and up to 9% slower where they leave fewer threads idle)
    for (int G = r.G; G <= (fp32 ? 8 : 4); G += fp32 ? 4 : 1) {
      const int ng = (n + G - 1) / G;
      if (fp32 && ng / 2 > ring_most_ks(G, false)) continue;
      for (int B = fp32 ? 64 : 32; B <= (fp32 ? 64 : 128); B += 32)
        if (B >= ng) consider(G, B / ng, 1, 1, B, !fp32);
    }
    // a candidate in parts, over one CTA or several
    for (int G = r.G; G <= 4; G += std::max(1, 4 - G)) {
      const int ng = (n + G - 1) / G, h = ng / 2;
      for (int P : {1, 2, 3, 4, 5, 6, 8, 10}) {
        if ((P > 1 && P > h + 1) || ng * P > kRingMaxB) break;
        for (int fill : {64, 128}) {
          const int C = fp32 ? std::max(1, fill / (ng * P)) : 1;
          const int B = (ng * P * C + 31) / 32 * 32;
          for (int S = 1; S <= 8 && (S == 1 || (C == 1 && h >= S * P)); S *= 2)
            consider(G, C, P, S, B, true);
          if (C == 1) break;
        }
      }
    }
    r = best;
    NG = (n + r.G - 1) / r.G;
  } else if (fp32 && NG / 2 <= kUnevenPackedH && a.n_cand * NG > 64LL * sms) {
    // large uneven batch of small clusters: packed like a uniform one, every
    // candidate with the threads of the largest (33,563 of 4..9 atoms: 22 us a
    // call, 55 with a CTA each; 20,000 of 15..60: 35, 70)
    r.B = 64;
    pl.C = r.B / NG;
    r.multi = false;
  } else {
    // uneven: one candidate a CTA, its parts set by the kernel from its own
    // size; small candidates cannot use many threads (6,583 of 8..47 atoms, FP32
    // Morse: 25 us a call with one warp, 44 us with 128 threads; 4,096 of 13..150
    // atoms, FP32: 44 us with 128 threads, 45 with 64, 57 with 32)
    r.B = NG <= 13 ? 32 : NG <= 26 ? 64 : std::max(128, (NG + 31) / 32 * 32);
    pl.P = 2;                                // (reserves the parts' buffer)
  }
  const int H = NG / 2;
  // uneven, few candidates: several CTAs each, while there are fewer than four per SM to
  // share out and each keeps eight shifts a part
  if (a.uniform_n <= 0 && r.multi)
    while (pl.S < 8 && a.n_cand * pl.S < 4LL * sms && H >= 16 * pl.S * (r.B / NG)) pl.S *= 2;
  // shifts between barriers, in equal chunks: FP32 as many as leave shared
  // memory for 16 warps an SM, FP64 up to five for two CTAs an SM; packed ones
  // take all at once
  const int per = pl.P * pl.S, all = std::max(1, (H + per - 1) / per);
  pl.KS = all;
  for (int most = fp32 ? ring_most_ks(r.G, per > 1) : 5; r.multi && most >= 1; --most) {
    const int chunks = (all + most - 1) / most;
    pl.KS = (all + chunks - 1) / chunks;
    if (fp32 || ring_smem(r.B, pl, false, r.G) <= kRingSmem) break;
  }
  if (fp32 && a.uniform_n > 0 && a.xtype == LJ_F32) {
    const uintptr_t al = reinterpret_cast<uintptr_t>(a.x) | reinterpret_cast<uintptr_t>(a.grad);
    pl.vec = n % 4 == 0 && al % 16 == 0 ? 4 : n % 2 == 0 && al % 8 == 0 ? 2 : 1;
  }
  return r;
}

template <typename K>
cudaError_t launch_ring(K k, const ljh::EvalArgs& a, const RingLaunch& r, cudaStream_t s) {
  const size_t smem = ring_smem(r.B, r.pl, a.prec != LJ_PREC_FP64, r.G);
  // The limit belongs to the kernel and not to the launch, and one kernel serves many
  // shapes (53 KB for 1,024 x 500 atoms, 107 KB for 256 x 1,024): it is always
  // the most there is, so that no thread lowers it between another's two calls.
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
    if (e != cudaSuccess) return e;
  }
  const long long need = (a.n_cand + r.pl.C - 1) / r.pl.C;
  // a CTA per tile: the hardware shares out candidates of different sizes
  const long long tiles = std::min(need, 1LL << 27);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(tiles * r.pl.S), 1, 1);
  cfg.blockDim = dim3((unsigned)r.B, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)r.pl.S;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = r.pl.S > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, a, r.pl);
}

template <typename IO, int POT, bool SIG>
cudaError_t launch_typed(const ljh::EvalArgs& a, int sms, cudaStream_t s) {
  const RingLaunch r = ring_plan(a, sms);
  if (a.prec == LJ_PREC_FP64) {
    if (r.G == 2) return launch_ring(eval_ring_f64_kernel<2, IO, POT, SIG>, a, r, s);
    if (r.G == 3) return launch_ring(eval_ring_f64_kernel<3, IO, POT, SIG>, a, r, s);
    return launch_ring(eval_ring_f64_kernel<4, IO, POT, SIG>, a, r, s);
  }
  if (r.multi) return launch_ring(eval_ring_f32_kernel<4, IO, POT, SIG, MULTI_PART>, a, r, s);
  if (a.uniform_n <= 0)
    return launch_ring(eval_ring_f32_kernel<4, IO, POT, SIG, PACKED_UNEVEN>, a, r, s);
  return r.G == 8 ? launch_ring(eval_ring_f32_kernel<8, IO, POT, SIG, PACKED>, a, r, s)
                  : launch_ring(eval_ring_f32_kernel<4, IO, POT, SIG, PACKED>, a, r, s);
}

template <typename IO>
cudaError_t launch_io(const ljh::EvalArgs& a, int sms, cudaStream_t s) {
  if (a.k.pot == LJ_POT_MORSE) return launch_typed<IO, LJ_POT_MORSE, false>(a, sms, s);
  return a.k.sigma == 1.0 ? launch_typed<IO, LJ_POT_LJ, false>(a, sms, s)
                          : launch_typed<IO, LJ_POT_LJ, true>(a, sms, s);
}

}  // namespace

namespace ljh {

cudaError_t eval_launch(const EvalArgs& a, cudaStream_t s) {
  return a.xtype == LJ_F32 ? launch_io<float>(a, a.sms, s) : launch_io<double>(a, a.sms, s);
}

}  // namespace ljh
