// legpair.cu -- associated-Legendre synthesis and analysis in the parity-pair
// basis, with the recurrence restarted from a table of checkpoints.
//
// F and G hold the two rings of a pair side by side, [m][pair][north, south]: the
// lanes of a warp (one pair each) read and write whole lines, and the ring kernels
// touch one (north, south) element per m.  The equator (the last pair) has no south
// ring.
//
// Basis (Ishioka 2018, J. Meteor. Soc. Japan 96, "A new recurrence formula for
// efficient computation of spherical harmonic transform").  With
// eps_l = sqrt((l^2 - m^2) / (4 l^2 - 1)), z lam_l = eps_{l+1} lam_{l+1} +
// eps_l lam_{l-1}, let Q_j = lam_{m+2j+1} / z (an even function of z, as the
// lam of even l - m are).  Then
//   lam_{m+2j+1} = z Q_j,   lam_{m+2j} = eps_{m+2j+1} Q_j + eps_{m+2j} Q_{j-1},
// so one function serves an even and an odd l, and Q_j steps by two l at once:
//   eps_{l+1} eps_{l+2} Q_{j+1} = (z^2 - eps_{l+1}^2 - eps_l^2) Q_j
//                                 - eps_l eps_{l-1} Q_{j-1},   l = m + 2 j + 1.
// Scaled and sign-folded, Q_j = h_j s_j with h_0 = h_1 = 1 and
//   s_j = (A_j w + B_j) s_{j-1} + s_{j-2}
// (tables indexed by the j they produce) with w = z^2 - w0 and B_j taken at w0:
// three equal forms, w0 = 1, 1/2 and 0, for the pairs below kform[0] (near the
// pole, where -sin^2 theta keeps the small angle that z^2 rounds away), below
// kform[1], and the others.  Each keeps |B| at or below the size of the sum, so
// that rounding B does not add to the phase; 32 pairs take the form of their middle one.
//
// Per (m, ring pair) and j this costs 2 multiply-adds for the recurrence and 4
// for the two complex sums, 3 per (l, m, pair) term; the one-step recurrence in
// lam_l needs a multiply and 3 multiply-adds (in FP32, with z in two parts, a
// multiply and 4).
//
// Near the equator Q_j grows like lam / z while neighbouring Q_j cancel in
// lam_{m+2j}, so rounding in s_j is amplified by up to 1/z there (measured in
// FP64 at Nside 1024: 1.1e-13 of the map's rms on the rings next to the equator,
// 1.5e-15 with the one-step recurrence; in FP32 7e-5 at Nside 256 and 4e-4 at
// Nside 1024, 4e-7 and 1e-6 with it).  The ring pairs k >= keq (|z| < 1/6 and what makes
// whole warps, where lam_mm itself is the seed for every m: equatorial_pair) therefore
// take the one-step recurrence lam_l <- z lam_{l-1}, lam_{l-2}, two l per j, at 8
// multiply-adds instead of 6 (FP32: 10, z in two parts).  In the synthesis they get warps,
// and in FP64 CTAs, of their own, so no number of pairs per thread and no Nside mixes the
// two kinds.  In the analysis a block's sums over them are separate ones, of even and odd
// l instead of E and O: a map that is zero but on nine rings around the equator comes out
// to 1.6e-7 in FP32 at Nside 512 (1.3e-4 without it) and to 6.5e-16 in FP64 (1.8e-13).
//
// Bound: the FP64 unit, 2 multiply-adds per clock and SM (98 and 92 % busy at Nside 512).
// At Nside 1024, lmax 2048 (3.14e9 terms) the synthesis takes 16.6 ms (21.4 ms with the
// one-step recurrence for all pairs) and the analysis 17.7 ms (29.0 ms), against 15.6 ms
// for 3 multiply-adds per term, 4 for the equatorial eighth, at the unit's measured 1.25
// TFLOP/s; at Nside 150, lmax 311, 0.104 and 0.137 ms (0.233 and 0.276 ms).  FP32: the
// FMA pipe takes 6 clocks per warp and step (equatorial 10), 0.28 ms at Nside 1024;
// measured 0.487 ms (synthesis, from 0.645) and 0.656 ms (analysis, from 0.891), at Nside
// 256 17.9 and 31.5 us: what is left is the reductions, the loads between the blocks (1.0
// GB of DRAM at Nside 1024, most of it checkpoints: 0.15 ms) and, on small maps, the
// largest m's chain.  Double-float (93 FP32 operations per step, 110 equatorial, against
// 116 for two l of the one-step recurrence; a multiply-add counts as two): Nside 512
// synthesis 0.61 ms (0.76), analysis 1.05 ms (0.97 and a combine pass of 0.04), Nside 1024
// 4.4 and 7.6 ms, bound by the FP32 pipe's dependent chains at 16 warps per SM.
//
// Checkpoints: ck[(block b of 16 j of m)][pair] holds (s_{16b-1}, s_{16b-2}), so any 16
// j can be computed on their own: a warp of the analysis owns 16 j of one m, keeps
// their 64 sums per lane in registers over all ring pairs, and reduces them across the
// lanes once.  The terms start at the first |Q_j| >= 2^-100 (j = js); in the block that
// holds js the checkpoint is, where the state before the block is out of the
// arithmetic's range, the seeds (s_js, s_js+1) instead, which enter at j = js (jin).
// FP64 always has that state; FP32 where it is above 2^-120.
#include <limits.h>
#include <math.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "wf_internal.cuh"

namespace wf {

namespace {

// ------------------------------------------------------------- indexing
// blocks of 16 j of one m: (L - m) / 32 + 1
__host__ __device__ __forceinline__ long tri_b(long n) {
  const long q = (n + 1) / 32, r = (n + 1) % 32;  // t = 0 .. n: sum of t / 32 + 1
  return n + 1 + 16 * q * (q - 1) + q * r;
}
__host__ __device__ __forceinline__ long block_base(int lmax, int m) {
  return tri_b(lmax) - tri_b(lmax - m);
}
__device__ __forceinline__ long alm_base(int lmax, int m) {  // index of (m, m)
  return (long)m * (2 * lmax + 1 - m) / 2 + m;
}

// ------------------------------------------------------------- arithmetic
template <typename V> struct Cx;  // complex element of F, G and the alm input
template <> struct Cx<double> { typedef double2 type; };
template <> struct Cx<float> { typedef float2 type; };
template <> struct Cx<dd> { typedef PairVec<dd>::type type; };
template <typename V> struct alignas(16) Quad { V a, b, c, d; };
template <typename V> struct alignas(2 * sizeof(V)) Pair { V a, b; };

__device__ __forceinline__ double fmav(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ void accv(double &acc, double s, double x) { acc = fma(s, x, acc); }

__device__ __forceinline__ float fmav(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ void accv(float &acc, float s, float x) { acc = fmaf(s, x, acc); }
// (dx, dy) = (ax, ay) (bx, by) + (cx, cy): one packed instruction (f32x2), each half
// rounded as the scalar one
__device__ __forceinline__ void fma2(float &dx, float &dy, float ax, float ay, float bx, float by,
                                     float cx, float cy) {
  asm("{\n .reg .b64 ra, rb, rc, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n"
      " mov.b64 rc, {%6, %7};\n fma.rn.f32x2 rd, ra, rb, rc;\n mov.b64 {%0, %1}, rd;\n}"
      : "=f"(dx), "=f"(dy)
      : "f"(ax), "f"(ay), "f"(bx), "f"(by), "f"(cx), "f"(cy));
}

// ------------------------------------------------------------- double-float
// dd: an unevaluated sum hi + lo of two floats (~48-bit significand), products by the
// FMA two-product, sums by two-sum (Dekker, Knuth); explicit _rn intrinsics, so nothing
// is contracted or reassociated.  The anchors of the mixed solver need the FP64
// iteration map to ~1e-10, not to FP64's last bit, and this part's FP64 unit runs at
// ~1/64 of its FP32 rate.
__device__ __forceinline__ dd dd_of(double x) {
  const float h = (float)x;
  return {h, (float)(x - (double)h)};
}
__device__ __forceinline__ double dd_val(dd a) { return (double)a.hi + (double)a.lo; }
// (s, e) with |s| >= |e| -> normalised pair
__device__ __forceinline__ dd dd_quick(float s, float e) {
  const float h = __fadd_rn(s, e);
  return {h, __fsub_rn(e, __fsub_rn(h, s))};
}
// a b and the rounding error of the float product
__device__ __forceinline__ void dd_prod(dd a, dd b, float &p, float &e) {
  p = __fmul_rn(a.hi, b.hi);
  e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, e));
}
__device__ __forceinline__ float two_sum(float a, float b, float &err) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return s;
}
__device__ __forceinline__ dd operator+(dd a, dd b) {
  float err;
  const float s = two_sum(a.hi, b.hi, err);
  return dd_quick(s, __fadd_rn(err, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ dd operator-(dd a, dd b) { return a + dd{-b.hi, -b.lo}; }
__device__ __forceinline__ dd operator*(dd a, dd b) {
  float p, e;
  dd_prod(a, b, p, e);
  return dd_quick(p, e);
}
__device__ __forceinline__ dd fmav(dd a, dd b, dd c) {
  float p, e, err;
  dd_prod(a, b, p, e);
  const float s = two_sum(p, c.hi, err);
  return dd_quick(s, __fadd_rn(__fadd_rn(e, c.lo), err));
}
// a b + c without the last normalisation: the factor of the next product
__device__ __forceinline__ dd coefv(dd a, dd b, dd c) {
  float p, e, err;
  dd_prod(a, b, p, e);
  const float s = two_sum(p, c.hi, err);
  return {s, __fadd_rn(__fadd_rn(e, c.lo), err)};
}
// acc += s x, acc kept unnormalised (hi the running sum, lo the rounding errors)
__device__ __forceinline__ void accv(dd &acc, dd s, dd x) {
  float p, e, err;
  dd_prod(s, x, p, e);
  acc.hi = two_sum(acc.hi, p, err);
  acc.lo = __fadd_rn(acc.lo, __fadd_rn(err, e));
}
// c z f + acc, the step of the one-step recurrence (equator); FP32 carries z in two
// parts and rounds c f: c nears 2 along l, and a rounded c z would add up its error
__device__ __forceinline__ double eqv(double c, double z, double, double f, double acc) {
  return fma(c * z, f, acc);
}
__device__ __forceinline__ float eqv(float c, float z, float zl, float f, float acc) {
  const float x = c * f;
  return fmaf(x, z, fmaf(x, zl, acc));
}
__device__ __forceinline__ dd eqv(dd c, dd z, dd, dd f, dd acc) {
  dd x;
  dd_prod(c, z, x.hi, x.lo);
  return fmav(x, f, acc);
}
// the same for two pairs, each half rounded as the scalar one
__device__ __forceinline__ void eqv2(float c, float z0, float z1, float l0, float l1, float f0,
                                     float f1, float &a0, float &a1) {
  float t0, t1;
  const float x0 = c * f0, x1 = c * f1;
  fma2(t0, t1, x0, x1, l0, l1, a0, a1);
  fma2(a0, a1, x0, x1, z0, z1, t0, t1);
}
__device__ __forceinline__ double coefv(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float coefv(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double shfx(double v, int s) { return __shfl_xor_sync(0xffffffffu, v, s); }
__device__ __forceinline__ float shfx(float v, int s) { return __shfl_xor_sync(0xffffffffu, v, s); }
__device__ __forceinline__ dd shfx(dd v, int s) { return {shfx(v.hi, s), shfx(v.lo, s)}; }
// a checkpoint in the kernel's arithmetic (the dd kernels read the FP64 ones)
template <typename V, typename W>
__device__ __forceinline__ typename Cx<V>::type state_as(W v) {
  if constexpr (std::is_same<V, dd>::value)
    return {dd_of(v.x), dd_of(v.y)};
  else
    return v;
}

__device__ __forceinline__ int wmin(int v) { return __reduce_min_sync(0xffffffffu, v); }
__device__ __forceinline__ int wmax(int v) { return __reduce_max_sync(0xffffffffu, v); }

// v[0..31] per lane -> lane i returns the sum over the lanes of v[i]
template <typename V>
__device__ __forceinline__ V lane_sums(V *v, int lane) {
#pragma unroll
  for (int s = 16; s >= 1; s >>= 1) {
    const bool upper = (lane & s) != 0;
#pragma unroll
    for (int j = 0; j < s; ++j) {
      const V send = upper ? v[j] : v[j + s];
      const V keep = upper ? v[j + s] : v[j];
      v[j] = keep + shfx(send, s);
    }
  }
  return v[0];
}

}  // namespace

// ------------------------------------------------------------- synthesis
// One thread per NP ring pairs of one m (grid: tiles of pairs x m), a
// warp-uniform loop over j.  FP32 with NP even runs two pairs per packed instruction
// (f32x2); its shared-memory inputs hold every value twice, so that a packed operand
// is one load.  The CTA stages the m's coefficients in shared
// memory, combined to the pair basis on the way:
//   E_j = se_j a_{m+2j} + sn_j a_{m+2j+2},   O_j = so_j a_{m+2j+1}.
// F_north = sum_j s_j (E_j + z O_j), F_south the difference.
constexpr int PSYN_THREADS = 64;     // FP64
constexpr int PSYN_THREADS32 = 256;  // FP32, at most

template <typename V>
__host__ __device__ constexpr int synth_forms(int np) {  // forms staged by a CTA
  return std::is_same<V, float>::value || (std::is_same<V, double>::value && np > 1) ? 3 : 1;
}
template <typename V, int NP>
__global__ void __launch_bounds__(PSYN_THREADS32)
    k_pair_synth(const PairTab<V> t, int npairs, int lmax,
                 const typename Cx<V>::type *__restrict__ x,
                 typename Cx<V>::type *__restrict__ F, const SolverState *__restrict__ st,
                 int lstatic, int nlow, int eq_ofs) {
  typedef typename Cx<V>::type C;
  const int m = blockIdx.y;
  int L = lstatic;
  if (st) {
    if (st->done) return;
    L = st->lcur;
  }
  if (m > L) return;  // the ring step ignores m above the band
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr bool PK = std::is_same<V, float>::value && NP % 2 == 0;
  const int J = (L - m) / 2 + 1;
  // per j a quad (E_re, E_im, O_re, O_im), or, PK, two: (E_re, E_re, E_im, E_im),
  // (O_re, O_re, O_im, O_im); then the forms' (A, B), [NF][J]
  constexpr int QJ = PK ? 2 : 1;
  constexpr int NE = PK ? NP : 1;  // equatorial pairs per thread
  Quad<V> *sx = reinterpret_cast<Quad<V> *>(smraw);
  Pair<V> *srec = reinterpret_cast<Pair<V> *>(sx + QJ * J);
  // the same for the equatorial warps, where the CTA has both kinds behind the others
  Quad<V> *sxe = reinterpret_cast<Quad<V> *>(smraw + eq_ofs);
  Pair<V> *sre = reinterpret_cast<Pair<V> *>(sxe + QJ * J);
  // the first nlow warps of a row take the pairs below keq, the others the equatorial ones
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int warp0 = blockIdx.x * nw;
  const bool equator = warp0 + warp >= nlow;
  const int pair0 = equator ? t.keq + (warp0 + warp - nlow) * 32 * NE
                            : (warp0 + warp) * 32 * NP;
  const int kend = equator ? npairs : t.keq;
  // where a CTA spans several forms all three are staged and every 32 pairs take their
  // own (one form of the CTA's or the warp's for all of them: FP64 with four pairs per
  // thread, Nside 512, 2.8e-14 of the rms at z = 2/3 instead of 3e-15).  FP64 CTAs with a
  // pair per thread hold 64 pairs, double-float ones 64, or 128 of 1024 and more: one
  constexpr int NF = synth_forms<V>(NP);
  int form[NP];
  V w[NP];
  int js[NP];
#pragma unroll
  for (int i = 0; i < NP; ++i) {  // in flight while the coefficients are staged
    const int k = pair0 + lane + 32 * i;
    form[i] = t.form(NF == 1 ? warp0 * 32 * NP + (int)blockDim.x * NP / 2 - 1 : pair0 + 32 * i + 15);
    w[i] = V(0);
    js[i] = INT_MAX / 2;
    if (!equator && k < kend) {
      w[i] = t.w[form[i] * t.stride + k];
      js[i] = t.js[(long)m * t.stride + k];
    }
  }
  {
    const long q0 = pair_base(lmax, m), a0 = alm_base(lmax, m);
    auto put = [](Quad<V> *q, int j, V er, V ei, V orr, V oi) {
      if constexpr (PK) {
        q[2 * j] = {er, er, ei, ei};
        q[2 * j + 1] = {orr, orr, oi, oi};
      } else {
        q[j] = {er, ei, orr, oi};
      }
    };
    for (int j = threadIdx.x; j < J; j += blockDim.x) {
      const int l = m + 2 * j;
      const C c0 = x[a0 + 2 * j];
      C c1 = {}, c2 = {};
      if (l + 1 <= L) c1 = x[a0 + 2 * j + 1];
      if (l + 2 <= L) c2 = x[a0 + 2 * j + 2];
      if (warp0 + nw > nlow) {
        const V ge = t.ge[q0 + j], go = t.go[q0 + j];
        put(sxe, j, ge * c0.x, ge * c0.y, go * c1.x, go * c1.y);
        sre[j] = reinterpret_cast<const Pair<V> *>(t.rec_e)[q0 + j];
      }
      if (warp0 < nlow) {
        const V se = t.se[q0 + j], sn = t.sn[q0 + j], so = t.so[q0 + j];
        put(sx, j, fmav(se, c0.x, sn * c2.x), fmav(se, c0.y, sn * c2.y), so * c1.x, so * c1.y);
        if constexpr (NF == 1) {
          srec[j] = reinterpret_cast<const Pair<V> *>(t.rec[form[0]])[q0 + j];
        } else {
#pragma unroll
          for (int f = 0; f < NF; ++f)
            srec[f * J + j] = reinterpret_cast<const Pair<V> *>(t.rec[f])[q0 + j];
        }
      }
    }
  }
  __syncthreads();
  if (pair0 >= kend) return;

  Quad<V> *out = reinterpret_cast<Quad<V> *>(F) + (long)m * npairs;
  if (equator) {
    V z[NE], zl[NE], u[NE], o[NE], er[NE], ei[NE], orr[NE], oi[NE];
#pragma unroll
    for (int i = 0; i < NE; ++i) {
      const int k = pair0 + lane + 32 * i;
      z[i] = zl[i] = u[i] = o[i] = er[i] = ei[i] = orr[i] = oi[i] = V(0);
      if (k < kend) {
        z[i] = t.z[k];
        if constexpr (std::is_same<V, float>::value) zl[i] = t.zl[k];
        u[i] = state_as<V>(t.ck_e[block_base(lmax, m) * t.estride + k - t.keq / 64 * 64]).x;
      }
    }
#pragma unroll 4
    for (int j = 0; j < J; ++j) {
      const Pair<V> r = sre[j];
      if constexpr (PK) {
        const Quad<V> xe = sxe[2 * j], xo = sxe[2 * j + 1];
#pragma unroll
        for (int i = 0; i < NE; i += 2) {
          eqv2(r.a, z[i], z[i + 1], zl[i], zl[i + 1], o[i], o[i + 1], u[i], u[i + 1]);
          fma2(er[i], er[i + 1], u[i], u[i + 1], xe.a, xe.b, er[i], er[i + 1]);
          fma2(ei[i], ei[i + 1], u[i], u[i + 1], xe.c, xe.d, ei[i], ei[i + 1]);
          eqv2(r.b, z[i], z[i + 1], zl[i], zl[i + 1], u[i], u[i + 1], o[i], o[i + 1]);
          fma2(orr[i], orr[i + 1], o[i], o[i + 1], xo.a, xo.b, orr[i], orr[i + 1]);
          fma2(oi[i], oi[i + 1], o[i], o[i + 1], xo.c, xo.d, oi[i], oi[i + 1]);
        }
      } else {
        const Quad<V> q = sxe[j];
#pragma unroll
        for (int i = 0; i < NE; ++i) {
          u[i] = eqv(r.a, z[i], zl[i], o[i], u[i]);
          accv(er[i], u[i], q.a);
          accv(ei[i], u[i], q.b);
          o[i] = eqv(r.b, z[i], zl[i], u[i], o[i]);
          accv(orr[i], o[i], q.c);
          accv(oi[i], o[i], q.d);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < NE; ++i) {
      const int k = pair0 + lane + 32 * i;
      if (k < kend) out[k] = {er[i] + orr[i], ei[i] + oi[i], er[i] - orr[i], ei[i] - oi[i]};
    }
    return;
  }

  const Pair<V> *sr[NP];
  bool mixed = false;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    sr[i] = srec + (NF == 1 ? 0 : form[i] * J);
    mixed |= NF > 1 && form[i] != form[0];
  }
  V s1[NP], s2[NP], d0[NP], d1[NP], er[NP], ei[NP], orr[NP], oi[NP];
  int jmin = INT_MAX, jinj = -1;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    const int k = pair0 + lane + 32 * i;
    s1[i] = s2[i] = d0[i] = d1[i] = er[i] = ei[i] = orr[i] = oi[i] = V(0);
    if (js[i] < J) {
      const C s = state_as<V>(t.seed[(long)m * t.stride + k]);
      d0[i] = s.x;
      d1[i] = s.y;
      jmin = min(jmin, js[i]);
      jinj = max(jinj, js[i] + 1);
    }
  }
  jmin = wmin(jmin);
  jinj = min(wmax(jinj), J - 1);
  // INJ: seeds may still enter; MIXED: the pairs' forms differ
  auto step = [&](int jj, auto INJ, auto MIXED) {
    Pair<V> r[NP];
    r[0] = sr[0][jj];
#pragma unroll
    for (int i = 1; i < NP; ++i) r[i] = MIXED ? sr[i][jj] : r[0];
    V s[NP];
#pragma unroll
    for (int i = 0; i < NP; i += PK ? 2 : 1) {
      if constexpr (PK) {
        V c0, c1;
        fma2(c0, c1, r[i].a, r[i + 1].a, w[i], w[i + 1], r[i].b, r[i + 1].b);
        fma2(s[i], s[i + 1], c0, c1, s1[i], s1[i + 1], s2[i], s2[i + 1]);
      } else {
        s[i] = fmav(coefv(r[i].a, w[i], r[i].b), s1[i], s2[i]);
      }
    }
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      if (INJ) {
        s[i] = jj == js[i] ? d0[i] : s[i];
        s[i] = jj == js[i] + 1 ? d1[i] : s[i];
      }
      s2[i] = s1[i];
      s1[i] = s[i];
    }
    if constexpr (PK) {
      const Quad<V> xe = sx[2 * jj], xo = sx[2 * jj + 1];
#pragma unroll
      for (int i = 0; i < NP; i += 2) {
        fma2(er[i], er[i + 1], s[i], s[i + 1], xe.a, xe.b, er[i], er[i + 1]);
        fma2(ei[i], ei[i + 1], s[i], s[i + 1], xe.c, xe.d, ei[i], ei[i + 1]);
        fma2(orr[i], orr[i + 1], s[i], s[i + 1], xo.a, xo.b, orr[i], orr[i + 1]);
        fma2(oi[i], oi[i + 1], s[i], s[i + 1], xo.c, xo.d, oi[i], oi[i + 1]);
      }
    } else {
      const Quad<V> q = sx[jj];
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        accv(er[i], s[i], q.a);
        accv(ei[i], s[i], q.b);
        accv(orr[i], s[i], q.c);
        accv(oi[i], s[i], q.d);
      }
    }
  };
  const std::true_type yes;
  const std::false_type no;
  int j = jmin;
  if (NF > 1 && NP > 1 && mixed) {
    for (; j <= jinj; ++j) step(j, yes, yes);
#pragma unroll 4
    for (; j < J; ++j) step(j, no, yes);
  } else {
    for (; j <= jinj; ++j) step(j, yes, no);
#pragma unroll 4
    for (; j < J; ++j) step(j, no, no);
  }
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    const int k = pair0 + lane + 32 * i;
    if (k >= kend) continue;
    const V z = t.z[k], zr = z * orr[i], zi = z * oi[i];
    out[k] = {er[i] + zr, ei[i] + zi, er[i] - zr, ei[i] - zi};
  }
}

// ------------------------------------------------------------- analysis
// One CTA per m.  The m's ring sums P_k = (G_N + G_S, z (G_N - G_S)) are staged
// in shared memory, in tiles of PANA_TILE pairs; each warp takes blocks of 16 j,
// holds the block's 64 sums per lane in registers, walks the tile's pairs 32 at a
// time (one per lane, the recurrence restarted from the checkpoints) and reduces
// across the lanes into D.  The epilogue goes back to l,
//   a_{m+2j} = Omega (se_j De_j + sn_{j-1} De_{j-1}),  a_{m+2j+1} = Omega so_j Do_j,
// with the solver's filter, source term and Cauchy sums fused.
constexpr int PANA_TILE = 2048;
constexpr int PAIR_SMEM = 220 * 1024;  // dynamic shared memory limit of these kernels
constexpr int PANA_MAXWARPS = 16;
constexpr int CKJ = 16;

// 16 steps of R pairs (one lane's): the recurrence and the four sums of each j; in
// FP32 the real and the imaginary sum of one parity are one packed accumulator.
// INJ: a pair's seeds c may enter, at step `rel` and the next (else c is the state
// before the block), and the pairs may differ in their form (table sr[i]).
// NJ steps from step `skip` on (dd's second halves: the steps before it run in a loop, one
// copy of the unrolled ones serves both halves -- with a copy for each, this kernel's
// warps wait for instructions).
template <typename V, int R, bool INJ, int NJ>
__device__ __forceinline__ void pair_block(V (&v)[4 * NJ], const Pair<V> *const (&sr)[R],
                                           const V (&w)[R], const typename Cx<V>::type (&c)[R],
                                           const Quad<V> (&p)[R], const int (&rel)[R], int skip) {
  V s1[R], s2[R];
  int at[R];  // the seeds' step, counted on from the current one
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const bool inj = INJ && (unsigned)rel[i] < (unsigned)CKJ;
    s1[i] = inj ? V(0) : c[i].x;
    s2[i] = inj ? V(0) : c[i].y;
    at[i] = inj ? rel[i] : -100;
  }
  const Pair<V> *r0 = sr[0];
  if constexpr (NJ < CKJ) {
    static_assert(R == 1 && INJ, "halves: one pair per lane");
#pragma unroll 4
    for (int jj = 0; jj < skip; ++jj) {
      const Pair<V> r = *r0++;
      V s = fmav(coefv(r.a, w[0], r.b), s1[0], s2[0]);
      s = at[0] == 0 ? c[0].x : s;
      s = at[0] == -1 ? c[0].y : s;
      s2[0] = s1[0];
      s1[0] = s;
      --at[0];
    }
  }
#pragma unroll
  for (int jj = 0; jj < NJ; ++jj) {
    Pair<V> r = r0[jj];
#pragma unroll
    for (int i = 0; i < R; ++i) {
      if (INJ && i > 0) r = sr[i][jj];
      V s = fmav(coefv(r.a, w[i], r.b), s1[i], s2[i]);
      if (INJ) {
        s = jj == at[i] ? c[i].x : s;
        if (jj > 0 || NJ < CKJ) s = jj == at[i] + 1 ? c[i].y : s;
      }
      s2[i] = s1[i];
      s1[i] = s;
      V *x = v + 4 * jj;
      if constexpr (std::is_same<V, float>::value) {
        fma2(x[0], x[1], s, s, p[i].a, p[i].b, x[0], x[1]);
        fma2(x[2], x[3], s, s, p[i].c, p[i].d, x[2], x[3]);
      } else {
        accv(x[0], s, p[i].a);
        accv(x[1], s, p[i].b);
        accv(x[2], s, p[i].c);
        accv(x[3], s, p[i].d);
      }
    }
  }
}

// The same for equatorial pairs: c is (lam_{m+2j-2}, lam_{m+2j-1}), scaled and folded,
// before the block; the sums are those of even and of odd l - m, from step `skip` on
// (dd's second halves).  FP32 steps its two pairs packed.
template <typename V, int R, int NJ>
__device__ __forceinline__ void eq_block(V (&v)[4 * NJ], const Pair<V> *sr, const V (&z)[R],
                                         const V (&zl)[R], const typename Cx<V>::type (&c)[R],
                                         const Quad<V> (&p)[R], int skip) {
  V u[R], o[R];
#pragma unroll
  for (int i = 0; i < R; ++i) {
    u[i] = c[i].x;
    o[i] = c[i].y;
  }
  auto next = [&](Pair<V> r) {
    if constexpr (R == 2) {
      eqv2(r.a, z[0], z[1], zl[0], zl[1], o[0], o[1], u[0], u[1]);
      eqv2(r.b, z[0], z[1], zl[0], zl[1], u[0], u[1], o[0], o[1]);
    } else {
      u[0] = eqv(r.a, z[0], zl[0], o[0], u[0]);
      o[0] = eqv(r.b, z[0], zl[0], u[0], o[0]);
    }
  };
  if constexpr (NJ < CKJ) {
#pragma unroll 1
    for (int jj = 0; jj < skip; ++jj) next(sr[jj]);
    sr += skip;
  }
#pragma unroll
  for (int jj = 0; jj < NJ; ++jj) {
    next(sr[jj]);
    asm volatile("" ::: "memory");  // keeps later table loads, and their registers, below
    V *x = v + 4 * jj;
#pragma unroll
    for (int i = 0; i < R; ++i) {
      accv(x[0], u[i], p[i].a);
      accv(x[1], u[i], p[i].b);
      accv(x[2], o[i], p[i].c);
      accv(x[3], o[i], p[i].d);
    }
  }
}

// Epilogue of one coefficient (FP64): a = Omega (sr, si), then in ANA_FILTER mode
// the source term of an anchored stage, the filter f_l = Sbar / (Sbar + xi Omega),
// Sbar = max(C_l - mu Omega, 0) (Eq. 15, App. B) and the Cauchy partial sums
// (weight wm = 1 for m = 0, 2 else); writes x.
__device__ __forceinline__ void pair_finish(long i, int l, double ar, double ai, double wm,
                                            int mode, const double *__restrict__ cl,
                                            double omega, double xi, double mu,
                                            const double2 *__restrict__ src,
                                            const double2 *__restrict__ xa,
                                            double2 *__restrict__ x, double &num, double &den,
                                            double &dx) {
  if (mode == ANA_FILTER) {
    const double sbar = fmax(cl[l] - mu * omega, 0.0);
    const double f = sbar / (sbar + xi * omega);
    if (src) {  // harmonic source term of a correction solve
      ar += xi * omega * src[i].x;
      ai += xi * omega * src[i].y;
    }
    ar *= f;
    ai *= f;
    const double2 old = x[i];
    const double dr = ar - old.x, di = ai - old.y;
    num += wm * (dr * dr + di * di);
    den += wm * (ar * ar + ai * ai);
    if (xa) {  // anchored stage: ||x_a + delta||^2
      const double2 b = xa[i];
      const double tr = ar + b.x, ti = ai + b.y;
      dx += wm * (tr * tr + ti * ti);
    }
  }
  x[i] = make_double2(ar, ai);
}

// The same in FP32 (this part's FP64 unit runs at 1/64 of the FP32 rate): the filter
// from the FP32 C_l, om = Omega, xio = xi Omega, muo = mu Omega.  Only the Cauchy
// differences against the FP64 iterate stay in FP64 (unweighted: the caller
// multiplies by wm once).  xs (optional): the coefficient in FP32, the next
// synthesis' input.
__device__ __forceinline__ void pair_finish32(long i, int l, float sr, float si, int mode,
                                              const float *__restrict__ cl, float om, float xio,
                                              float muo, const double2 *__restrict__ src,
                                              const double2 *__restrict__ xa,
                                              double2 *__restrict__ x, float2 *__restrict__ xs,
                                              double &num, double &den, double &dx) {
  float ar = om * sr, ai = om * si;
  if (mode == ANA_FILTER) {
    const float sbar = fmaxf(cl[l] - muo, 0.f);
    const float f = sbar > 0.f ? sbar / (sbar + xio) : 0.f;
    if (src) {  // harmonic source term of a correction solve
      const double2 sv = src[i];
      ar = fmaf(xio, (float)sv.x, ar);
      ai = fmaf(xio, (float)sv.y, ai);
    }
    ar *= f;
    ai *= f;
    const double2 old = x[i];
    const double ard = ar, aid = ai;
    const double dr = ard - old.x, di = aid - old.y;
    num = fma(dr, dr, fma(di, di, num));
    den = fma(ard, ard, fma(aid, aid, den));
    if (xa) {  // anchored stage: ||x_a + delta||^2
      const double2 b = xa[i];
      const double tr = ard + b.x, ti = aid + b.y;
      dx = fma(tr, tr, fma(ti, ti, dx));
    }
  }
  x[i] = make_double2(ar, ai);
  if (xs) xs[i] = make_float2(ar, ai);
}

// block sums of the Cauchy partials -> partials[2m], [2m + 1] and (anchored
// stages) [2 (lmax + 1) + m], in a fixed order
__device__ __forceinline__ void pair_partials(double num, double den, double dx, int m, int lmax,
                                              double *__restrict__ partials) {
  __shared__ double ws[3][PANA_MAXWARPS];
  for (int o = 16; o > 0; o >>= 1) {
    num += __shfl_xor_sync(0xffffffffu, num, o);
    den += __shfl_xor_sync(0xffffffffu, den, o);
    dx += __shfl_xor_sync(0xffffffffu, dx, o);
  }
  const int warp = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    ws[0][warp] = num;
    ws[1][warp] = den;
    ws[2][warp] = dx;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0, c = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      a += ws[0][w];
      b += ws[1][w];
      c += ws[2][w];
    }
    partials[2 * m] = a;
    partials[2 * m + 1] = b;
    partials[2 * (lmax + 1) + m] = c;
  }
}

// the epilogue's tables and sums: the kernel's own arithmetic, or (dd) FP64
template <typename E>
__device__ __forceinline__ const E *epi(const E *own, const double *) { return own; }
template <typename E>
__device__ __forceinline__ const E *epi(const dd *, const double *f64) { return f64; }
template <typename E> __device__ __forceinline__ E epi_val(E v) { return v; }
template <typename E> __device__ __forceinline__ double epi_val(dd v) { return dd_val(v); }

template <typename V>
__global__ void __launch_bounds__(std::is_same<V, dd>::value ? 32 * PANA_MAXWARPS : 256,
                                  std::is_same<V, float>::value ? 2 : 1)
    k_pair_anal(const PairTab<V> t, int npairs, int lmax,
                const double *__restrict__ cl, double omega,
                const typename Cx<V>::type *__restrict__ G, double2 *__restrict__ x,
                double *__restrict__ partials, const double2 *__restrict__ src,
                typename Cx<V>::type *__restrict__ xs, const float *__restrict__ cl32,
                const double *__restrict__ se64, const double *__restrict__ sn64,
                const double *__restrict__ so64, const double *__restrict__ ge64,
                const double *__restrict__ go64, const SolverState *__restrict__ st, int mode,
                int lstatic, int tile_max) {
  typedef typename Cx<V>::type C;
  typedef typename CkVec<V>::type Ck;
  constexpr int R = std::is_same<V, float>::value ? 2 : 1;  // pairs in flight per lane
  // where seeds may enter: FP32 the blocks in jin; dd the block of js, from the seed
  // table (the FP64 state before it may be below FP32's range); FP64 none
  constexpr bool DD = std::is_same<V, dd>::value, SEEDS = R == 2 || DD;
  // FP32: one item does both kinds of pairs, its pair-basis sums brought to those of
  // even and odd l before the equatorial ones are added, which saves a lane reduction
  // (FP64 and dd: the arithmetic of that costs as much as the reduction)
  constexpr bool ONE = R == 2;
  // j per warp item: dd halves a block (32 double-float sums leave room for 16 warps
  // per SM, 64 for 8: 1.01 ms at Nside 512), the second half repeating the first's
  // recurrence
  constexpr int NJ = DD ? CKJ / 2 : CKJ, HALVES = CKJ / NJ;
  const int m = blockIdx.x;
  int L = lstatic;
  double xi = 0.0, mu = 0.0;
  const double2 *xa = nullptr;  // anchored stage: the anchor iterate x_a
  if (st) {
    if (st->done) return;
    L = st->lcur;
    xi = st->xi;
    mu = filter_mu(*st, st->mu);
    xa = st->xa;
  }
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nwarps = blockDim.x >> 5;
  const long a0 = alm_base(lmax, m);
  const double wm = (m == 0) ? 1.0 : 2.0;
  double num = 0.0, den = 0.0, dx = 0.0;

  if (m <= L) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int J = (L - m) / 2 + 1, nb = (J + CKJ - 1) / CKJ, J16 = nb * CKJ;
    const int tile = min((npairs + 63) / 64 * 64, tile_max);
    Quad<V> *sp = reinterpret_cast<Quad<V> *>(smraw);                 // [tile]
    Quad<V> *sd = sp + tile;                                          // [J16]
    Quad<V> *se = sd + J16;  // [J16]: equatorial sums; ONE: the change of basis
    Pair<V> *srec = reinterpret_cast<Pair<V> *>(se + J16);            // [4][J16]
    Pair<V> *scar = srec + 4 * J16;  // ONE, [nb + 1]: even sum of the last j of a block
    const long q0 = pair_base(lmax, m), cb = block_base(lmax, m);
    for (int j = tid; j < J16; j += blockDim.x) {
      sd[j] = se[j] = {V(0), V(0), V(0), V(0)};
      if constexpr (ONE) {
        if (j <= nb) scar[j] = {V(0), V(0)};
        if (j < J) {
          const V ge = V(1) / t.ge[q0 + j];
          se[j] = {t.se[q0 + j] * ge, j % CKJ ? t.sn[q0 + j - 1] * ge : V(0),
                   t.so[q0 + j] / t.go[q0 + j], V(0)};
        }
      }
    }
    for (int f = 0; f < 4; ++f) {
      const Pair<V> *rec = reinterpret_cast<const Pair<V> *>(f < 3 ? t.rec[f] : t.rec_e);
      for (int j = tid; j < J16; j += blockDim.x) {
        const Pair<V> zero = {V(0), V(0)};
        srec[f * J16 + j] = j < J ? rec[q0 + j] : zero;
      }
    }
    for (int t0 = 0; t0 < npairs; t0 += tile_max) {
      const int nt = min(tile_max, npairs - t0);
      __syncthreads();  // the previous tile's reads are done
      for (int k = tid; k < (nt + 63) / 64 * 64; k += blockDim.x) {
        Quad<V> q = {V(0), V(0), V(0), V(0)};
        if (k < nt) q = reinterpret_cast<const Quad<V> *>(G)[(long)m * npairs + t0 + k];
        if (t0 + k == npairs - 1) q.c = q.d = V(0);  // the equator
        const V z = t0 + k < t.keq ? t.z[t0 + k] : V(1);
        sp[k] = {q.a + q.c, q.b + q.d, z * (q.a - q.c), z * (q.b - q.d)};
      }
      __syncthreads();
      // the tile's pairs below keq are nlow; a block's sums over those and over the
      // equatorial ones are items of their own
      const int nlow = max(0, min(nt, t.keq - t0));
      const int items_low = nlow > 0 || ONE ? HALVES * nb : 0;
      const int items = items_low + (nlow < nt && !ONE ? HALVES * nb : 0);
      // js, the checkpoints, w and z are loaded one step (32 R pairs) ahead
      const int *jrow = (DD ? t.js : t.jin) + (long)m * t.stride + t0 + lane;
      const Ck *srow = t.seed + (long)m * t.stride + t0 + lane;
      for (int item = warp; item < items; item += nwarps) {
        const bool eq = item >= items_low;
        const int bh = eq ? item - items_low : item;
        const int b = bh / HALVES, j0 = b * CKJ;
        V v[4 * NJ];
#pragma unroll
        for (int i = 0; i < 4 * NJ; ++i) v[i] = V(0);
        if (ONE || !eq) {
          const Ck *crow = t.ck + (cb + b) * t.cstride + t0 + lane;
          int rel[R], form[R];
          Ck c[R];
          V w[R];
          auto load = [&](int g) {
#pragma unroll
            for (int i = 0; i < R; ++i) {
              const int k = g + 32 * i;
              form[i] = t.form(t0 + k);
              rel[i] = SEEDS ? jrow[k] - j0 : -1;
              c[i] = crow[k];
              if constexpr (DD) {
                const Ck sd0 = srow[k];
                if ((unsigned)rel[i] < (unsigned)CKJ) c[i] = sd0;
              }
              w[i] = t.w[form[i] * t.stride + t0 + lane + k];
            }
          };
          // below its first warp of pairs a block is zero
          int g = max(0, t.gfirst[cb + b] - t0) / (32 * R) * (32 * R);
          if (g < nlow) load(g);
          for (; g < nlow; g += 32 * R) {
            const Pair<V> *sr[R];
            V wc[R];
            C d[R];
            Quad<V> p[R];
            int rl[R];
            bool slow = R == 2 && form[0] != form[R - 1];
#pragma unroll
            for (int i = 0; i < R; ++i) {
              sr[i] = srec + form[i] * J16 + j0;
              wc[i] = w[i];
              d[i] = state_as<V>(c[i]);
              rl[i] = rel[i];
              p[i] = sp[g + 32 * i + lane];
              slow |= (unsigned)rel[i] < (unsigned)CKJ;
            }
            if (g + 32 * R < nlow) load(g + 32 * R);
            if (DD || (R == 2 && __any_sync(0xffffffffu, slow)))
              pair_block<V, R, SEEDS, NJ>(v, sr, wc, d, p, rl, DD ? (bh & 1) * NJ : 0);
            else if constexpr (!DD)
              pair_block<V, R, false, NJ>(v, sr, wc, d, p, rl, 0);
          }
        }
        if constexpr (ONE) {
          // even: De_j and De_{j-1} make up l = m + 2 j; the block's last De_j also
          // belongs to the first l of the next block
          if (nlow > 0) {
            V ca = v[4 * NJ - 4], cc = v[4 * NJ - 3];
            for (int o = 16; o > 0; o >>= 1) {
              ca = ca + shfx(ca, o);
              cc = cc + shfx(cc, o);
            }
            if (lane == 0) scar[b + 1] = {scar[b + 1].a + ca, scar[b + 1].b + cc};
#pragma unroll
            for (int jj = NJ - 1; jj >= 0; --jj) {
              const Quad<V> f = se[j0 + jj];
              V *x = v + 4 * jj;
              x[0] = f.a * x[0];
              x[1] = f.a * x[1];
              if (jj > 0) {
                x[0] = fmav(f.b, x[-4], x[0]);
                x[1] = fmav(f.b, x[-3], x[1]);
              }
              x[2] = f.c * x[2];
              x[3] = f.c * x[3];
            }
          }
        }
        if (ONE || eq) {
          // the rows start at a multiple of 64, zero below keq
          const Ck *crow = t.ck_e + (cb + b) * t.estride + (t0 - t.keq / 64 * 64) + lane;
          for (int g = nlow / (32 * R) * (32 * R); g < nt; g += 32 * R) {
            V z[R], zl[R];
            C c[R];
            Quad<V> p[R];
#pragma unroll
            for (int i = 0; i < R; ++i) {
              const int k = g + 32 * i;
              c[i] = state_as<V>(crow[k]);
              z[i] = t.z[t0 + lane + k];
              zl[i] = V(0);
              if constexpr (std::is_same<V, float>::value) zl[i] = t.zl[t0 + lane + k];
              p[i] = sp[k + lane];
            }
            eq_block<V, R, NJ>(v, srec + 3 * J16 + j0, z, zl, c, p, DD ? (bh & 1) * NJ : 0);
          }
        }
        V *out = reinterpret_cast<V *>(eq ? se : sd) + 4 * (j0 + (bh % HALVES) * NJ) + lane;
        const V lo = lane_sums(v, lane);
        out[0] = out[0] + lo;
        if constexpr (!DD) {
          const V hi = lane_sums(v + 32, lane);
          out[32] = out[32] + hi;
        }
      }
    }
    __syncthreads();
    for (int i = tid; i <= L - m; i += blockDim.x) {
      const int j = i >> 1;
      // dd: back to l in FP64
      typedef typename std::conditional<DD, double, V>::type E;
      const E *fo = epi<E>(t.so, so64), *fe = epi<E>(t.se, se64), *fn = epi<E>(t.sn, sn64);
      E sr, si;
      if constexpr (ONE) {
        const E g = (i & 1 ? t.go : t.ge)[q0 + j];
        const Quad<V> q = sd[j];
        sr = g * (i & 1 ? q.c : q.a);
        si = g * (i & 1 ? q.d : q.b);
        if (j > 0 && i % (2 * CKJ) == 0) {
          const Pair<V> c = scar[j / CKJ];
          sr = fmav(t.sn[q0 + j - 1], c.a, sr);
          si = fmav(t.sn[q0 + j - 1], c.b, si);
        }
      } else if (i & 1) {
        const Quad<V> qe = se[j];
        const E f = fo[q0 + j], g = epi<E>(t.go, go64)[q0 + j];
        sr = fmav(g, epi_val<E>(qe.c), f * epi_val<E>(sd[j].c));
        si = fmav(g, epi_val<E>(qe.d), f * epi_val<E>(sd[j].d));
      } else {
        const Quad<V> qe = se[j];
        const E f = fe[q0 + j], ge = epi<E>(t.ge, ge64)[q0 + j];
        sr = fmav(ge, epi_val<E>(qe.a), f * epi_val<E>(sd[j].a));
        si = fmav(ge, epi_val<E>(qe.b), f * epi_val<E>(sd[j].b));
        if (j > 0) {
          const E g = fn[q0 + j - 1];
          sr = fmav(g, epi_val<E>(sd[j - 1].a), sr);
          si = fmav(g, epi_val<E>(sd[j - 1].b), si);
        }
      }
      if constexpr (std::is_same<V, float>::value)
        pair_finish32(a0 + i, m + i, sr, si, mode, cl32, (float)omega, (float)(xi * omega),
                      (float)(mu * omega), src, xa, x, xs, num, den, dx);
      else
        pair_finish(a0 + i, m + i, omega * sr, omega * si, wm, mode, cl, omega, xi, mu, src, xa,
                    x, num, den, dx);
    }
    if constexpr (std::is_same<V, float>::value) {
      num *= wm;
      den *= wm;
      dx *= wm;
    }
  }
  // coefficients of this m above the band are zero
  for (int l = max(m, L + 1) + tid; l <= lmax; l += blockDim.x) {
    const long i = a0 + (l - m);
    if (mode == ANA_FILTER) {
      const double2 old = x[i];
      num += wm * (old.x * old.x + old.y * old.y);
    }
    x[i] = make_double2(0.0, 0.0);
    if constexpr (std::is_same<V, float>::value) {
      if (xs) xs[i] = make_float2(0.f, 0.f);
    }
  }
  if (mode == ANA_FILTER) pair_partials(num, den, dx, m, lmax, partials);
}

// ------------------------------------------------------------- launch
// The synthesis' warps: nlow of 32 np pairs each below keq, then the equatorial ones; mix:
// in the same CTAs, else the equatorial ones in CTAs of their own.  Shared memory per j: a
// quad (packed FP32: two) and the pairs of nf forms, equatorial a quad or two and a pair.
struct SynthGrid {
  unsigned ctas;
  int nlow, eq_ofs;
  size_t smem;
  SynthGrid(size_t v, int npairs, int keq, int lmax, int threads, int np, int nf, bool packed,
            bool mix) {
    const int nw = threads / 32, j = lmax / 2 + 1, ne = packed ? np : 1;
    const size_t quads = packed ? 8 : 4, low = (quads + 2 * nf) * v * j,
                 eq = (quads + 2) * v * j;
    nlow = (keq + 32 * np - 1) / (32 * np);
    if (!mix) nlow = (nlow + nw - 1) / nw * nw;
    ctas = (unsigned)((nlow + (npairs - keq + 32 * ne - 1) / (32 * ne) + nw - 1) / nw);
    eq_ofs = mix ? (int)((low + 15) / 16 * 16) : 0;
    smem = mix ? eq_ofs + eq : low;
  }
};
static size_t anal_smem(size_t v, int npairs, int lmax, int tile) {
  const size_t j16 = (size_t)(lmax / 32 + 1) * CKJ;
  return 4 * v * std::min((npairs + 63) / 64 * 64, tile) + 16 * v * j16 +
         2 * v * (j16 / CKJ + 1);
}
// half a tile where a whole one leaves too little shared memory (FP64 above lmax ~ 2500)
static int anal_tile(size_t v, int npairs, int lmax) {
  return anal_smem(v, npairs, lmax, PANA_TILE) <= PAIR_SMEM ? PANA_TILE : PANA_TILE / 2;
}
// a warp per item of the CTA of m = 0 (FP64, dd: twice its blocks), at most 8; dd 16 where
// one CTA fills an SM's shared memory (Nside 1024: 8 warps 9.9 ms, 16 7.6 ms)
static int anal_threads(size_t v, int lmax, size_t dd_smem = 0) {
  const int nb = lmax / 32 + 1, most = dd_smem > PAIR_SMEM / 2 ? PANA_MAXWARPS : 8;
  return 32 * std::max(2, std::min(most, v == 4 ? nb : 2 * nb));
}

static wf_status ready(const void *ck) {
  if (ck) return WF_OK;
  set_error("transform: Nside is too large for the ring FFTs of this precision");
  return WF_ERR_CUDA;
}

template <int NP>
static void synth64(const Plan &P, const double2 *x, double2 *F, const SolverState *st,
                    int lstatic, int threads) {
  const SynthGrid g(8, P.npairs, P.pt64.keq, P.lmax, threads, NP, synth_forms<double>(NP), false,
                    false);
  k_pair_synth<double, NP><<<dim3(g.ctas, P.lmax + 1), threads, g.smem, P.stream>>>(
      P.pt64, P.npairs, P.lmax, x, F, st, lstatic, g.nlow, g.eq_ofs);
}

template <>
wf_status launch_legendre_synth<double2>(const Plan &P, const double2 *x, double2 *F,
                                         const SolverState *st, int lstatic) {
  WF_TRY(ready(P.pt64.ck));
  ++P.nlaunch;
  // one or two warps per CTA: an SM's FP64 unit (2 lanes per clock) is full with a
  // few warps, and small CTAs spread small maps over the SMs
  const int threads = (long)P.npairs * (P.lmax + 1) <= 64L * 4 * P.num_sms ? 32 : PSYN_THREADS;
  switch (P.syn_np[0]) {
    case 2: synth64<2>(P, x, F, st, lstatic, threads); break;
    case 4: synth64<4>(P, x, F, st, lstatic, threads); break;
    default: synth64<1>(P, x, F, st, lstatic, threads); break;
  }
  WF_CUDA(cudaGetLastError());
  return WF_OK;
}

template <>
wf_status launch_legendre_anal<double2>(const Plan &P, const double2 *G, double2 *x,
                                        const SolverState *st, int mode, int lstatic,
                                        const double2 *src, double2 *) {
  WF_TRY(ready(P.pt64.ck));
  ++P.nlaunch;
  const int tile = anal_tile(8, P.npairs, P.lmax);
  k_pair_anal<double><<<P.lmax + 1, anal_threads(8, P.lmax), anal_smem(8, P.npairs, P.lmax, tile),
                     P.stream>>>(
      P.pt64, P.npairs, P.lmax, P.cl_d, P.omega, G, x, P.partials, src, nullptr, nullptr,
      nullptr, nullptr, nullptr, nullptr, nullptr, st, mode, lstatic, tile);
  WF_CUDA(cudaGetLastError());
  return WF_OK;
}

template <int NP>
static void synth32(const Plan &P, const float2 *x, float2 *F, const SolverState *st,
                    int lstatic) {
  // both kinds of pairs in a CTA while two fit an SM, so that few of its warps idle, and 8
  // warps on large maps.  4 warps with CTAs of their own for the equatorial pairs: 0.574 ms
  // at Nside 1024 (a fifth of the warps idle), 0.487 ms with 8 in common ones; transform
  // at Nside 512 201 and 194 us; at Nside 256 the kernel takes 17.9 us with 4 warps, 19.2
  // with 8
  const int np = P.npairs, keq = P.pt32.keq, nf = synth_forms<float>(NP);
  const int threads = np < 1024 ? PSYN_THREADS32 / 2 : PSYN_THREADS32;
  constexpr bool packed = NP % 2 == 0;
  SynthGrid g(4, np, keq, P.lmax, threads, NP, nf, packed, true);
  if (g.smem > PAIR_SMEM / 2) g = SynthGrid(4, np, keq, P.lmax, threads, NP, nf, packed, false);
  k_pair_synth<float, NP><<<dim3(g.ctas, P.lmax + 1), threads, g.smem, P.stream>>>(
      P.pt32, P.npairs, P.lmax, x, F, st, lstatic, g.nlow, g.eq_ofs);
}

template <>
wf_status launch_legendre_synth<float2>(const Plan &P, const float2 *xs, float2 *F,
                                        const SolverState *st, int lstatic) {
  WF_TRY(ready(P.pt32.ck));
  ++P.nlaunch;
  switch (P.syn_np[1]) {
    case 1: synth32<1>(P, xs, F, st, lstatic); break;
    case 4: synth32<4>(P, xs, F, st, lstatic); break;
    default: synth32<2>(P, xs, F, st, lstatic); break;
  }
  WF_CUDA(cudaGetLastError());
  return WF_OK;
}

template <>
wf_status launch_legendre_anal<float2>(const Plan &P, const float2 *G, double2 *x,
                                       const SolverState *st, int mode, int lstatic,
                                       const double2 *src, float2 *xs_out) {
  WF_TRY(ready(P.pt32.ck));
  ++P.nlaunch;
  const int tile = anal_tile(4, P.npairs, P.lmax);
  k_pair_anal<float><<<P.lmax + 1, anal_threads(4, P.lmax), anal_smem(4, P.npairs, P.lmax, tile),
                     P.stream>>>(
      P.pt32, P.npairs, P.lmax, P.cl_d, P.omega, G, x, P.partials, src, xs_out, P.cl32, nullptr,
      nullptr, nullptr, nullptr, nullptr, st, mode, lstatic, tile);
  WF_CUDA(cudaGetLastError());
  return WF_OK;
}

template <int NP>
static void synth_dd(const Plan &P, const float4 *x, float4 *F, const SolverState *st,
                     int lstatic) {
  const SynthGrid g(8, P.npairs, P.ptdd.keq, P.lmax, PSYN_THREADS, NP, synth_forms<dd>(NP), false,
                    false);
  typedef Cx<dd>::type C;
  k_pair_synth<dd, NP><<<dim3(g.ctas, P.lmax + 1), PSYN_THREADS, g.smem, P.stream>>>(
      P.ptdd, P.npairs, P.lmax, reinterpret_cast<const C *>(x), reinterpret_cast<C *>(F), st,
      lstatic, g.nlow, g.eq_ofs);
}

wf_status launch_legendre_synth_dd(const Plan &P, const float4 *xs, float4 *F,
                                   const SolverState *st, int lstatic) {
  WF_TRY(ready(P.ptdd.ck));
  ++P.nlaunch;
  if (P.npairs >= 1024)
    synth_dd<2>(P, xs, F, st, lstatic);
  else
    synth_dd<1>(P, xs, F, st, lstatic);
  WF_CUDA(cudaGetLastError());
  return WF_OK;
}

wf_status launch_legendre_anal_dd(const Plan &P, const float4 *G, double2 *x,
                                  const SolverState *st, int mode, int lstatic,
                                  const double2 *src) {
  WF_TRY(ready(P.ptdd.ck));
  ++P.nlaunch;
  typedef Cx<dd>::type C;
  const int tile = anal_tile(8, P.npairs, P.lmax);
  const size_t smem = anal_smem(8, P.npairs, P.lmax, tile);
  k_pair_anal<dd><<<P.lmax + 1, anal_threads(8, P.lmax, smem), smem, P.stream>>>(
      P.ptdd, P.npairs, P.lmax, P.cl_d, P.omega, reinterpret_cast<const C *>(G), x, P.partials,
      src, nullptr, nullptr, P.pt64.se, P.pt64.sn, P.pt64.so, P.pt64.ge, P.pt64.go, st, mode,
      lstatic, tile);
  WF_CUDA(cudaGetLastError());
  return WF_OK;
}

// FP64 coefficients in the synthesis' FP32
__global__ void k_to_f32(const double2 *__restrict__ x, long n, float2 *__restrict__ xs) {
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long)gridDim.x * blockDim.x)
    xs[i] = make_float2((float)x[i].x, (float)x[i].y);
}

wf_status launch_to_f32(const Plan &P, const double2 *x, float2 *xs) {
  ++P.nlaunch;
  const unsigned grid = (unsigned)std::min((P.nalm + 255) / 256, 8L * P.num_sms);
  k_to_f32<<<grid, 256, 0, P.stream>>>(x, P.nalm, xs);
  WF_CUDA(cudaGetLastError());
  return WF_OK;
}

// FP64 coefficients in double-float, the dd synthesis' input
__global__ void k_alm_to_dd(const double2 *__restrict__ x, long n, float4 *__restrict__ xs) {
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long)gridDim.x * blockDim.x) {
    const dd re = dd_of(x[i].x), im = dd_of(x[i].y);
    xs[i] = make_float4(re.hi, re.lo, im.hi, im.lo);
  }
}

wf_status launch_alm_to_dd(const Plan &P, const double2 *x, float4 *xs) {
  ++P.nlaunch;
  const unsigned grid = (unsigned)std::min((P.nalm + 255) / 256, 8L * P.num_sms);
  k_alm_to_dd<<<grid, 256, 0, P.stream>>>(x, P.nalm, xs);
  WF_CUDA(cudaGetLastError());
  return WF_OK;
}

wf_status init_pair_attributes() {
  const int big = PAIR_SMEM;
  WF_CUDA(cudaFuncSetAttribute(k_pair_synth<double, 1>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, big));
  WF_CUDA(cudaFuncSetAttribute(k_pair_synth<double, 2>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, big));
  WF_CUDA(cudaFuncSetAttribute(k_pair_synth<double, 4>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, big));
  WF_CUDA(cudaFuncSetAttribute(k_pair_synth<float, 1>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, big));
  WF_CUDA(cudaFuncSetAttribute(k_pair_synth<float, 2>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, big));
  WF_CUDA(cudaFuncSetAttribute(k_pair_synth<float, 4>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, big));
  WF_CUDA(cudaFuncSetAttribute(k_pair_synth<dd, 1>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, big));
  WF_CUDA(cudaFuncSetAttribute(k_pair_synth<dd, 2>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, big));
  WF_CUDA(cudaFuncSetAttribute(k_pair_anal<dd>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               big));
  WF_CUDA(cudaFuncSetAttribute(k_pair_anal<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               big));
  WF_CUDA(cudaFuncSetAttribute(k_pair_anal<double>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               big));
  return WF_OK;
}

// ------------------------------------------------------------- tables
// s of every (m, pair): a walk from lam_mm (mantissa, exponent) in scaled FP64
// until |Q_j| reaches 2^-100, then plainly to the last j, leaving the seeds, the state
// before each block and, in FP32, the blocks where the seeds enter.
__global__ void k_pair_walk(int npairs, int lmax, const PairTab<double> t_,
                            const PairTab<float> u, const double *__restrict__ mant,
                            const int *__restrict__ expo) {
  const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long)npairs * (lmax + 1)) return;
  const int m = (int)(t / npairs), k = (int)(t % npairs);
  const int J = (lmax - m) / 2 + 1, stride = t_.cstride;
  const long q0 = pair_base(lmax, m), cb = block_base(lmax, m), mk = (long)m * t_.stride + k;
  const int form = t_.form(k);
  const double2 *rec = t_.rec[form] + q0;
  const double w = t_.w[form * t_.stride + k];
  double v = mant[t] * sqrt(2.0 * m + 3.0), vp = 0.0;  // Q_0 = lam_mm / eps_{m+1}
  int e = expo[t], j = 0;                              // value v 2^e
  if (k >= t_.keq) {  // the grouped tables' start; nothing else reads them
    v = ldexp(v, e);
    t_.seed[mk] = make_double2(v, J > 1 ? fma(rec[1].x, w, rec[1].y) * v : 0.0);
    return;
  }
  // the state before the block of j: rec[0] = (0, 0), so (0, s_0) yields s_0 at j = 0
  double b1 = 0.0, b2 = v;
  int be = e;
  bool found = false;
  for (;;) {
    const double a = fabs(v * t_.so[q0 + j]);
    if (e == 0 ? a >= 0x1p-100 : (e == -200 && a >= 0x1p+100)) {
      found = true;
      break;
    }
    if (j == J - 1) break;
    ++j;
    if ((j & 15) == 0) {
      b1 = v;
      b2 = vp;
      be = e;
    }
    const double2 r = rec[j];
    const double vn = fma(fma(r.x, w, r.y), v, vp);
    vp = v;
    v = vn;
    if (e < 0 && fabs(v) > 0x1p+200) {
      v *= 0x1p-200;
      vp *= 0x1p-200;
      e += 200;
    }
  }
  if (!found) return;  // the tables are zero, js and jin beyond every block
  const int js = j, bj = j >> 4;
  t_.js[mk] = js;
  for (int b = bj; b < (J + 15) / 16; ++b)
    if (k / 32 * 32 < t_.gfirst[cb + b]) atomicMin(t_.gfirst + cb + b, k / 32 * 32);
  double s1 = ldexp(v, e), s2 = ldexp(vp, e), nx = 0.0;
  if (j + 1 < J) {
    const double2 r = rec[j + 1];
    nx = fma(fma(r.x, w, r.y), s1, s2);
  }
  t_.seed[mk] = make_double2(s1, nx);
  u.seed[mk] = make_float2((float)s1, (float)nx);
  const double2 st = make_double2(ldexp(b1, be), ldexp(b2, be));
  if (t_.ck) t_.ck[(cb + bj) * stride + k] = st;
  if (!t_.ck && !u.ck) return;
  const bool fits = fmax(fabs(st.x), fabs(st.y)) >= 0x1p-120;
  if (fits && u.ck) u.ck[(cb + bj) * stride + k] = make_float2((float)st.x, (float)st.y);
  const double seed0 = s1;
  for (;;) {
    if ((j & 15) == 15 || j + 1 == J) {
      if (!fits && (j >> 4) == bj && u.ck) {
        u.ck[(cb + bj) * stride + k] = make_float2((float)seed0, (float)nx);
        u.jin[mk] = js;
      }
      if (j + 1 < J) {
        const long at = (cb + (j >> 4) + 1) * stride + k;
        if (t_.ck) t_.ck[at] = make_double2(s1, s2);
        if (u.ck) u.ck[at] = make_float2((float)s1, (float)s2);
      }
    }
    if (++j >= J) break;
    const double2 r = rec[j];
    const double s = fma(fma(r.x, w, r.y), s1, s2);
    s2 = s1;
    s1 = s;
  }
}

// The equatorial pairs' checkpoints: the one-step recurrence from lam_mm, (even, odd)
// before each block.
__global__ void k_eq_walk(int npairs, int lmax, const PairTab<double> t_, const PairTab<float> u,
                          const double *__restrict__ mant, const int *__restrict__ expo) {
  const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const int n = npairs - t_.keq;
  if (t >= (long)n * (lmax + 1)) return;
  const int m = (int)(t / n), k = t_.keq + (int)(t % n);
  const int J = (lmax - m) / 2 + 1;
  const double2 *rec = t_.rec_e + pair_base(lmax, m);
  const double z = t_.z[k];
  const long i = (long)m * npairs + k;
  long at = block_base(lmax, m) * t_.estride + k - t_.keq / 64 * 64;
  double even = ldexp(mant[i], expo[i]), odd = 0.0;  // rec[0].x = 0 leaves lam_mm
  for (int j = 0; j < J; ++j) {
    if ((j & 15) == 0) {
      if (t_.ck_e) t_.ck_e[at] = make_double2(even, odd);
      if (u.ck_e) u.ck_e[at] = make_float2((float)even, (float)odd);
      at += t_.estride;
    }
    const double2 r = rec[j];
    even = fma(r.x * z, odd, even);
    odd = fma(r.y * z, even, odd);
  }
}

// double-double on the device, for the coefficient tables only: their errors
// would add up along j
struct d2 {
  double h, l;
};
__device__ __forceinline__ d2 d2_norm(double s, double e) {
  const double h = __dadd_rn(s, e);
  return {h, __dsub_rn(e, __dsub_rn(h, s))};
}
__device__ __forceinline__ d2 d2_mul(d2 a, d2 b) {
  const double p = __dmul_rn(a.h, b.h);
  return d2_norm(p, fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h));
}
__device__ __forceinline__ d2 d2_div(d2 a, d2 b) {
  const double q = a.h / b.h;
  const d2 p = d2_mul({q, 0.0}, b);
  return d2_norm(q, ((a.h - p.h) - p.l + a.l) / b.h);
}
__device__ __forceinline__ d2 d2_sqrt(d2 a) {
  const double r = sqrt(a.h);
  const double p = __dmul_rn(r, r);
  return d2_norm(r, ((a.h - p) - fma(r, r, -p) + a.l) / (2.0 * r));
}
__device__ __forceinline__ d2 d2_add(d2 a, d2 b) {  // |a| >= |b|
  const double s = __dadd_rn(a.h, b.h);
  return d2_norm(s, (b.h - (s - a.h)) + (a.l + b.l));
}
__device__ __forceinline__ d2 d2_sum(d2 a, d2 b) {  // any order
  return fabs(a.h) >= fabs(b.h) ? d2_add(a, b) : d2_add(b, a);
}
// eps_l^2 = (l - m) (l + m) / ((2 l - 1) (2 l + 1)); the integers are exact
__device__ __forceinline__ d2 eps2(double l, int m) {
  return d2_div({(l - m) * (l + m), 0.0}, {(2.0 * l - 1.0) * (2.0 * l + 1.0), 0.0});
}

// Pair basis: with up_j = eps_{l+1} eps_{l+2} (l = m + 2j + 1),
// h_{j+1} = h_{j-1} up_{j-1} / up_j and A = h_j / (h_{j+1} up_j).  One-step
// recurrence (equator): lam = g u, g_l = g_{l-2} eps_{l-1} / eps_l,
// u_l = c_l z u_{l-1} - u_{l-2}, c_l = g_{l-1} / (g_l eps_l), sign-folded
// likewise (signs (-1)^floor((l - m) / 2)).
// One CTA per m: h and g are products over j, so the threads take runs of an even number
// of j, multiply up their factors, and start from the product of the runs before theirs.
// One thread per m took 0.47 ms at Nside 32 and 1.3 ms at Nside 90, most of what a plan
// took more than before the parity-pair basis.
constexpr int COEF_THREADS = 64;
__global__ void __launch_bounds__(COEF_THREADS) k_pair_coefs(int lmax, PairTab<double> t) {
  __shared__ d2 prod[4][COEF_THREADS];
  const int m = blockIdx.x, tid = threadIdx.x;
  const long q0 = pair_base(lmax, m);
  const int J = (lmax - m) / 2 + 1, run = 2 * ((J + 2 * COEF_THREADS - 1) / (2 * COEF_THREADS));
  const int j0 = tid * run, j1 = min(J, j0 + run);
  const d2 one = {1.0, 0.0};
  // eps of l = m + 2 j0 and eps^2, eps of the next l
  const d2 rm0 = j0 > 0 ? d2_sqrt(eps2(m + 2.0 * j0, m)) : one;
  const d2 e_l0 = eps2(m + 2.0 * j0 + 1.0, m), r_l0 = d2_sqrt(e_l0);
  {
    // of the run: h at even j, h at odd j, g at even and at odd l - m
    d2 f[4] = {one, one, one, one};
    d2 rm = rm0, r_l = r_l0, up0 = d2_mul(rm0, r_l0);
    for (int j = j0; j < j1; ++j) {
      const double l = m + 2.0 * j + 1.0;
      const d2 r1 = d2_sqrt(eps2(l + 1.0, m)), r2 = d2_sqrt(eps2(l + 2.0, m));
      const d2 up = d2_mul(r1, r2);
      if (j > 0) {
        f[1 - (j & 1)] = d2_mul(f[1 - (j & 1)], d2_div(up0, up));
        f[3] = d2_mul(f[3], d2_div(rm, r_l));
      }
      f[2] = d2_mul(f[2], d2_div(r_l, r1));
      up0 = up;
      rm = r1;
      r_l = r2;
    }
    for (int c = 0; c < 4; ++c) prod[c][tid] = f[c];
  }
  __syncthreads();
  for (int o = 1; o < COEF_THREADS; o <<= 1) {
    d2 f[4];
    for (int c = 0; c < 4; ++c)
      f[c] = tid >= o ? d2_mul(prod[c][tid - o], prod[c][tid]) : prod[c][tid];
    __syncthreads();
    for (int c = 0; c < 4; ++c) prod[c][tid] = f[c];
    __syncthreads();
  }
  if (j0 >= J) return;
  d2 h1 = one, h0 = one, g1 = one, g0 = one;  // h_j, h_{j-1}, g_{2j}, g_{2j-1}
  if (tid > 0) {
    h1 = prod[0][tid - 1];
    h0 = prod[1][tid - 1];
    g1 = prod[2][tid - 1];
    g0 = prod[3][tid - 1];
  }
  d2 e_l = e_l0, r_l = r_l0, rm = rm0;
  d2 up0 = d2_mul(rm0, r_l0);  // up_{j-1}
  for (int j = j0; j < j1; ++j) {
    const double l = m + 2.0 * j + 1.0;
    const double fold = ((j >> 1) & 1) ? -1.0 : 1.0;
    const d2 e1 = eps2(l + 1.0, m), e2 = eps2(l + 2.0, m);
    const d2 r1 = d2_sqrt(e1), r2 = d2_sqrt(e2);
    t.se[q0 + j] = fold * d2_mul(h1, r_l).h;
    t.sn[q0 + j] = fold * d2_mul(h1, r1).h;
    t.so[q0 + j] = fold * h1.h;
    const d2 up = d2_mul(r1, r2);
    const d2 hn = j == 0 ? one : d2_div(d2_mul(h0, up0), up);
    if (j == 0) t.rec[0][q0] = t.rec[1][q0] = t.rec[2][q0] = make_double2(0.0, 0.0);
    if (j + 1 < J) {
      const double sg = (j & 1) ? -1.0 : 1.0;
      const d2 A = d2_div(h1, d2_mul(hn, up));
      const d2 e = e_l.h > e1.h ? d2_add(e_l, e1) : d2_add(e1, e_l);
      const d2 me = {-e.h, -e.l};
      t.rec[0][q0 + j + 1] = make_double2(sg * A.h, sg * d2_mul(A, d2_add(one, me)).h);
      t.rec[1][q0 + j + 1] =
          make_double2(sg * A.h, sg * d2_mul(A, d2_sum({0.5, 0.0}, me)).h);
      t.rec[2][q0 + j + 1] = make_double2(sg * A.h, sg * d2_mul(A, me).h);
    }
    // one-step: l - m = 2 j (g1, c0 from the last j) and 2 j + 1
    const double f2 = (j & 1) ? -1.0 : 1.0;
    const d2 go = j == 0 ? one : d2_div(d2_mul(g0, rm), r_l);  // g_{2j+1}
    t.ge[q0 + j] = f2 * g1.h;
    t.go[q0 + j] = f2 * go.h;
    t.rec_e[q0 + j].y = d2_div(g1, d2_mul(go, r_l)).h;
    if (j == 0) t.rec_e[q0].x = 0.0;
    const d2 ge = d2_div(d2_mul(g1, r_l), r1);                 // g_{2j+2}
    if (j + 1 < J) t.rec_e[q0 + j + 1].x = -d2_div(go, d2_mul(ge, r1)).h;
    g0 = go;
    g1 = ge;
    rm = r1;
    h0 = h1;
    h1 = hn;
    up0 = up;
    e_l = e2;
    r_l = r2;
  }
}

static wf_status build_pair_tables32(Plan &P, long nq);
static wf_status build_pair_tables_dd(Plan &P, long nq);

// The first of the pairs that take the one-step recurrence: those with |z| < 1/6 (above,
// the two recurrences' errors are within a factor of two, and the parity-pair basis is
// the better one from |z| ~ 1/2 on), as far as lam_mm, where it starts, stays above 2^-90
// for every m.  From a multiple of 64 or 32 on where lam_mm allows it and |z| stays below
// 4/9: the kernels take 32 or 64 pairs at a time, and a part of them costs as much as all.
static int equatorial_pair(const Plan &P) {
  auto starts = [&P](int k) { return P.lmax * log2(P.pairs_h[k].sth) > -90.0; };
  int k = P.npairs;
  while (k > 0 && P.pairs_h[k - 1].z < 1.0 / 6.0 && starts(k - 1)) --k;
  for (int step = P.npairs < 512 ? 32 : 64; step >= 32; step /= 2) {
    const int whole = k / step * step;
    if (3 * whole >= 2 * P.npairs && starts(whole)) return whole;
  }
  return k;
}

// The tables and the checkpoints.  mant, expo: lam_mm of every (m, pair).
wf_status build_pair_tables(Plan &P, const double *mant, const int *expo) {
  const int lmax = P.lmax;
  const long nq = pair_base(lmax, lmax) + 1;
  const long nb = block_base(lmax, lmax) + 1;
  const int stride = (P.npairs + 63) / 64 * 64;  // rows padded to whole steps
  std::vector<double> w(3 * (size_t)stride, 0.0), z(stride, 0.0);
  std::vector<float> zl(stride, 0.f);
  // the forms' limits z^2 = 3/4 and 1/4, in whole warps of pairs
  int kform[2] = {0, 0};
  for (int k = 0; k < P.npairs; ++k) {
    z[k] = P.pairs_h[k].z;
    zl[k] = (float)(z[k] - (double)(float)z[k]);
    for (int f = 0; f < 2; ++f)
      if (z[k] * z[k] > (f ? 0.25 : 0.75)) kform[f] = k + 1;
    w[k] = -(1.0 - z[k]) * (1.0 + z[k]);
    w[stride + k] = fma(z[k], z[k], -0.5);
    w[2L * stride + k] = z[k] * z[k];
  }
  auto up = [](auto **dst, const auto &v) {
    WF_CUDA(cudaMalloc(dst, sizeof(v[0]) * v.size()));
    WF_CUDA(cudaMemcpy(*dst, v.data(), sizeof(v[0]) * v.size(), cudaMemcpyHostToDevice));
    return WF_OK;
  };
  const int keq = equatorial_pair(P);
  PairTab<double> &t = P.pt64;
  for (int f = 0; f < 2; ++f) t.kform[f] = (kform[f] + 16) / 32 * 32;
  t.keq = keq;
  t.cstride = (keq + 63) / 64 * 64;
  t.estride = stride - keq / 64 * 64;
  t.stride = stride;
  WF_TRY(up(&t.w, w));
  WF_TRY(up(&t.z, z));
  WF_TRY(up(&P.pt32.zl, zl));
  WF_TRY(uploads_done());
  for (double2 **a : {&t.rec[0], &t.rec[1], &t.rec[2], &t.rec_e})
    WF_CUDA(cudaMalloc(a, sizeof(double2) * nq));
  for (double **a : {&t.se, &t.sn, &t.so, &t.ge, &t.go})
    WF_CUDA(cudaMalloc(a, sizeof(double) * nq));
  k_pair_coefs<<<lmax + 1, COEF_THREADS, 0, P.stream>>>(lmax, t);
  WF_CUDA(cudaGetLastError());
  WF_TRY(build_pair_tables32(P, nq));
  PairTab<float> &u = P.pt32;
  // no seed: js and jin beyond every block; no checkpoint: zero (also the rows'
  // padding)
  const size_t mk = (size_t)stride * (lmax + 1), ck = (size_t)nb * std::max(t.cstride, 1),
               ce = (size_t)nb * t.estride;
  WF_CUDA(cudaMalloc(&t.js, sizeof(int) * mk));
  WF_CUDA(cudaMalloc(&u.jin, sizeof(int) * mk));
  WF_CUDA(cudaMalloc(&t.seed, sizeof(double2) * mk));
  WF_CUDA(cudaMalloc(&u.seed, sizeof(float2) * mk));
  // the checkpoints are most of a plan (Nside 1024: 3.3 of 5.1 GB, growing as Nside^3):
  // only for the transforms whose ring FFTs can run
  auto checkpoints = [&](auto **a, auto **b) {
    WF_CUDA(cudaMalloc(a, sizeof(**a) * ck));
    WF_CUDA(cudaMalloc(b, sizeof(**b) * ce));
    WF_CUDA(cudaMemsetAsync(*a, 0, sizeof(**a) * ck, P.stream));
    WF_CUDA(cudaMemsetAsync(*b, 0, sizeof(**b) * ce, P.stream));
    return WF_OK;
  };
  if (ring_fits(P, sizeof(double2))) WF_TRY(checkpoints(&t.ck, &t.ck_e));
  if (ring_fits(P, sizeof(float2))) WF_TRY(checkpoints(&u.ck, &u.ck_e));
  WF_CUDA(cudaMalloc(&t.gfirst, sizeof(int) * nb));
  WF_CUDA(cudaMemsetAsync(t.js, 0x3f, sizeof(int) * mk, P.stream));
  WF_CUDA(cudaMemsetAsync(u.jin, 0x3f, sizeof(int) * mk, P.stream));
  WF_CUDA(cudaMemsetAsync(t.gfirst, 0x7f, sizeof(int) * nb, P.stream));  // none
  u.js = t.js;
  u.gfirst = t.gfirst;
  const long n = (long)P.npairs * (lmax + 1);
  k_pair_walk<<<(unsigned)((n + 127) / 128), 128, 0, P.stream>>>(P.npairs, lmax, t, u, mant,
                                                                 expo);
  WF_CUDA(cudaGetLastError());
  if (keq < P.npairs && (t.ck_e || u.ck_e)) {
    const long ne = (long)(P.npairs - keq) * (lmax + 1);
    k_eq_walk<<<(unsigned)((ne + 127) / 128), 128, 0, P.stream>>>(P.npairs, lmax, t, u, mant, expo);
    WF_CUDA(cudaGetLastError());
  }
  return build_pair_tables_dd(P, nq);
}

// FP32 copies of the FP64 tables
__global__ void k_pair_round(const double *__restrict__ in, long n, float *__restrict__ out) {
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long)gridDim.x * blockDim.x)
    out[i] = (float)in[i];
}

static wf_status build_pair_tables32(Plan &P, long nq) {
  const PairTab<double> &t = P.pt64;
  PairTab<float> &u = P.pt32;
  auto round = [&P](auto **dst, const void *src, long n) {
    WF_CUDA(cudaMalloc(dst, sizeof(float) * n));
    const unsigned grid = (unsigned)std::min((n + 255) / 256, 4096L);
    k_pair_round<<<grid, 256, 0, P.stream>>>(static_cast<const double *>(src), n,
                                             reinterpret_cast<float *>(*dst));
    WF_CUDA(cudaGetLastError());
    return WF_OK;
  };
  for (int f = 0; f < 3; ++f) WF_TRY(round(&u.rec[f], t.rec[f], 2 * nq));
  WF_TRY(round(&u.se, t.se, nq));
  WF_TRY(round(&u.sn, t.sn, nq));
  WF_TRY(round(&u.so, t.so, nq));
  WF_TRY(round(&u.w, t.w, 3L * t.stride));
  WF_TRY(round(&u.z, t.z, t.stride));
  WF_TRY(round(&u.rec_e, t.rec_e, 2 * nq));
  WF_TRY(round(&u.ge, t.ge, nq));
  WF_TRY(round(&u.go, t.go, nq));
  u.stride = t.stride;
  for (int f = 0; f < 2; ++f) u.kform[f] = t.kform[f];
  u.keq = t.keq;
  u.cstride = t.cstride;
  u.estride = t.estride;
  return WF_OK;
}

// the FP64 tables as double-float pairs; js, the seeds and the checkpoints are shared
__global__ void k_pair_split(const double *__restrict__ in, long n, dd *__restrict__ out) {
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long)gridDim.x * blockDim.x)
    out[i] = dd_of(in[i]);
}

static wf_status build_pair_tables_dd(Plan &P, long nq) {
  const PairTab<double> &t = P.pt64;
  PairTab<dd> &u = P.ptdd;
  auto split = [&P](auto **dst, const void *src, long n) {
    WF_CUDA(cudaMalloc(dst, sizeof(dd) * n));
    const unsigned grid = (unsigned)std::min((n + 255) / 256, 4096L);
    k_pair_split<<<grid, 256, 0, P.stream>>>(static_cast<const double *>(src), n,
                                             reinterpret_cast<dd *>(*dst));
    WF_CUDA(cudaGetLastError());
    return WF_OK;
  };
  for (int f = 0; f < 3; ++f) WF_TRY(split(&u.rec[f], t.rec[f], 2 * nq));
  WF_TRY(split(&u.rec_e, t.rec_e, 2 * nq));
  WF_TRY(split(&u.se, t.se, nq));
  WF_TRY(split(&u.sn, t.sn, nq));
  WF_TRY(split(&u.so, t.so, nq));
  WF_TRY(split(&u.ge, t.ge, nq));
  WF_TRY(split(&u.go, t.go, nq));
  WF_TRY(split(&u.w, t.w, 3L * t.stride));
  WF_TRY(split(&u.z, t.z, t.stride));
  u.stride = t.stride;
  u.js = t.js;
  u.seed = t.seed;
  u.ck = t.ck;
  u.ck_e = t.ck_e;
  u.gfirst = t.gfirst;
  u.keq = t.keq;
  u.cstride = t.cstride;
  u.estride = t.estride;
  for (int f = 0; f < 2; ++f) u.kform[f] = t.kform[f];
  return WF_OK;
}

void free_pair_tables(Plan &P) {
  PairTab<dd> &d = P.ptdd;
  void *g[] = {d.rec[0], d.rec[1], d.rec[2], d.rec_e, d.se, d.sn, d.so, d.ge, d.go, d.w, d.z};
  for (void *p : g)
    if (p) cudaFree(p);
  PairTab<float> &u = P.pt32;
  void *f[] = {u.rec[0], u.rec[1], u.rec[2], u.se, u.sn, u.so, u.w, u.z, u.ck, u.jin, u.seed,
               u.rec_e, u.ge, u.go, u.zl, u.ck_e};
  for (void *p : f)
    if (p) cudaFree(p);
  PairTab<double> &t = P.pt64;
  void *b[] = {t.rec[0], t.rec[1], t.rec[2], t.rec_e, t.se, t.sn, t.so, t.ge, t.go, t.w, t.z,
               t.js, t.seed, t.ck, t.ck_e, t.gfirst};
  for (void *p : b)
    if (p) cudaFree(p);
}

}  // namespace wf
