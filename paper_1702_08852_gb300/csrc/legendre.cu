// legendre.cu -- the double-float Legendre transforms of the mixed solver's anchor
// steps, between ring Fourier coefficients F_r[m] and harmonic coefficients a_lm
// (legpair.cu holds the FP64 and FP32 ones).
//
// Synthesis (the Y step of the paper's Algorithm 2 moved to the sphere):
//   F_r[m] = sum_{l >= m} lam_lm(z_r) a_lm,
// computed for the north and south ring of a pair at once from the parity
// lam_lm(-z) = (-1)^(l+m) lam_lm(z); analysis a_lm = Omega sum_r lam_lm(z_r) G_r[m].
// Both run the rescaled recurrence u_l = c_l z u_{l-1} - u_{l-2} (lam = g u, tables
// from plan.cu) from FP64 seeds at the first l where |lam| >= 2^-100.
#include <limits.h>

#include <algorithm>
#include <atomic>

#include "wf_internal.cuh"

namespace wf {

__device__ __forceinline__ long lm_index(int lmax, int l, int m) {
  return (long)m * (2 * lmax + 1 - m) / 2 + l;
}

__device__ __forceinline__ int warp_min(int v) {
  for (int o = 16; o > 0; o >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ int warp_max(int v) {
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

constexpr int SYN_THREADS = 128;
constexpr int ANA_THREADS = 128;
constexpr int ANA_WARPS = ANA_THREADS / 32;
constexpr int ANA_Q_CTAS_PER_SM = 8;  // upper bound; the occupancy decides

// Epilogue of one coefficient (l, m), index i: a = Omega g_l (sr, si) (the
// ring sums in u-units), then in ANA_FILTER mode the source term of an
// anchored stage, the filter f_l = Sbar / (Sbar + xi Omega) and the Cauchy
// partial sums (weight wm = 1 for m = 0, 2 else); writes x and xs_out.
__device__ __forceinline__ void anal_finish(long i, int l, double sr, double si,
                                            double wm, int mode,
                                            const double *__restrict__ rg,
                                            const double *__restrict__ cl, double omega,
                                            double xi, double mu,
                                            const double2 *__restrict__ src,
                                            const double2 *__restrict__ xa,
                                            double2 *__restrict__ x,
                                            double &num, double &den, double &dx) {
  const double s = omega * rg[i];
  double ar = s * sr, ai = s * si;
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

// coefficients of this m above the band (l > L) are zero
__device__ __forceinline__ void anal_zero_above(int m, int L, int lmax, long base,
                                                double wm, int mode,
                                                double2 *__restrict__ x,
                                                double &num) {
  const int lz = max(m, L + 1);
  for (int l = lz + (int)threadIdx.x; l <= lmax; l += ANA_THREADS) {
    const long i = base + (l - m);
    if (mode == ANA_FILTER) {
      const double2 old = x[i];
      num += wm * (old.x * old.x + old.y * old.y);
    }
    x[i] = make_double2(0.0, 0.0);
  }
}

// block sums of the Cauchy partials -> partials[2m], partials[2m + 1] and
// (anchored stages) partials[2 (lmax + 1) + m] (fixed order: lanes by
// xor-butterfly, then warps in index order)
__device__ __forceinline__ void anal_partials(double num, double den, double dx, int m,
                                              int lmax, double *__restrict__ partials) {
  __shared__ double wsum[3][ANA_WARPS];
  for (int o = 16; o > 0; o >>= 1) {
    num += __shfl_xor_sync(0xffffffffu, num, o);
    den += __shfl_xor_sync(0xffffffffu, den, o);
    dx += __shfl_xor_sync(0xffffffffu, dx, o);
  }
  const int warp = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    wsum[0][warp] = num;
    wsum[1][warp] = den;
    wsum[2][warp] = dx;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0, c = 0.0;
    for (int w = 0; w < ANA_WARPS; ++w) {
      a += wsum[0][w];
      b += wsum[1][w];
      c += wsum[2][w];
    }
    partials[2 * m] = a;
    partials[2 * m + 1] = b;
    partials[2 * (lmax + 1) + m] = c;
  }
}

// Sum the tiles of every (l, m) of one m in tile order and finish as the
// per-m kernel does.  Block 0 resets the queue counter for the next launch
// (the analysis kernel has finished: same stream).
__global__ void __launch_bounds__(ANA_THREADS)
    k_anal_combine(int lmax, long nalm, int ntiles, const double *__restrict__ scratch,
                   const int *__restrict__ lstart, int *__restrict__ counter,
                   const double *__restrict__ rg, const double *__restrict__ cl,
                   double omega, double2 *__restrict__ x, double *__restrict__ partials,
                   const double2 *__restrict__ src,
                   const SolverState *__restrict__ st, int mode, int lstatic) {
  const int m = blockIdx.x;
  int L = lstatic;
  double xi = 0.0, mu = 0.0;
  const double2 *xa = nullptr;  // anchored stage: the anchor iterate x_a
  if (st) {
    if (st->done) return;
    L = st->lcur;
    xi = st->xi;
    mu = filter_mu(*st, st->mu);  // the signal step's truncation
    xa = st->xa;
  }
  if (m == 0 && threadIdx.x == 0) *counter = 0;
  const long base = lm_index(lmax, m, m);
  const double wm = (m == 0) ? 1.0 : 2.0;
  double num = 0.0, den = 0.0, dx = 0.0;
  if (m <= L) {
    for (int j = threadIdx.x; j <= L - m; j += ANA_THREADS) {
      const int l = m + j;
      double sr = 0.0, si = 0.0;
      for (int t = 0; t < ntiles; ++t) {
        if (l < __ldg(lstart + (long)m * ntiles + t)) continue;
        const double *p = scratch + 2 * ((long)t * nalm + base + j);
        sr += p[0];
        si += p[1];
      }
      anal_finish(base + j, l, sr, si, wm, mode, rg, cl, omega, xi, mu, src, xa, x,
                     num, den, dx);
    }
  }
  anal_zero_above(m, L, lmax, base, wm, mode, x, num);
  if (mode == ANA_FILTER) anal_partials(num, den, dx, m, lmax, partials);
}

// ------------------------------------------- double-float (df64) kernels
// The anchors of the mixed solver need the FP64 iteration map to ~1e-10, not
// to FP64's last bit, and this part's FP64 pipe is ~1/64 of its FP32 pipe.
// These kernels carry every value as an unevaluated sum hi + lo of two
// floats (~48-bit significand: products by FMA two-product, sums by
// two-sum, Dekker/Knuth), so the same transforms run on the FP32 pipe.
// Inputs and outputs are FP64 (double2), the recurrence is the FP64 one
// (u-convention, table rc), the analysis writes per-tile FP64 partial sums
// that k_anal_combine<double> adds in tile order.  Every operation is an
// explicit _rn intrinsic or fmaf, so nothing is contracted or reassociated.
struct dd {
  float hi, lo;
};
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
__device__ __forceinline__ dd dd_add(dd a, dd b) {
  const float s = __fadd_rn(a.hi, b.hi);
  const float bb = __fsub_rn(s, a.hi);
  const float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(b.hi, bb));
  return dd_quick(s, __fadd_rn(e, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ dd dd_sub(dd a, dd b) { return dd_add(a, {-b.hi, -b.lo}); }
__device__ __forceinline__ dd dd_mul(dd a, dd b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, e));
  return dd_quick(p, e);
}
// acc += u x with acc kept unnormalised (hi carries the running sum, lo the
// accumulated rounding errors); read it with dd_val
__device__ __forceinline__ void dd_acc(dd &acc, dd u, dd x) {
  const float p = __fmul_rn(u.hi, x.hi);
  float e = fmaf(u.hi, x.hi, -p);
  e = fmaf(u.hi, x.lo, fmaf(u.lo, x.hi, e));
  const float s = __fadd_rn(acc.hi, p);
  const float bb = __fsub_rn(s, acc.hi);
  const float err = __fadd_rn(__fsub_rn(acc.hi, __fsub_rn(s, bb)), __fsub_rn(p, bb));
  acc.hi = s;
  acc.lo = __fadd_rn(acc.lo, __fadd_rn(err, e));
}
// u_l = c_l z u_{l-1} - u_{l-2}: t = c u_{l-1} in double-float, then the
// product t z (two-product, unnormalised) and the difference with u_{l-2}
// (two-sum) with one final normalisation
__device__ __forceinline__ dd dd_rec(dd c, dd z, dd u1, dd u2) {
  const dd t = dd_mul(c, u1);
  const float p = __fmul_rn(t.hi, z.hi);
  float e = fmaf(t.hi, z.hi, -p);
  e = fmaf(t.hi, z.lo, fmaf(t.lo, z.hi, e));
  const float s = __fsub_rn(p, u2.hi);
  const float bb = __fsub_rn(s, p);
  const float err = __fadd_rn(__fsub_rn(p, __fsub_rn(s, bb)), __fsub_rn(-u2.hi, bb));
  return dd_quick(s, __fadd_rn(__fsub_rn(e, u2.lo), err));
}

constexpr int DD_NP_SYN = 2, DD_NP_ANA = 4;

// (kh + kl) + (rh + rl) for unnormalised double-float sums: a two-sum of
// the hi parts whose rounding error joins the lo parts
__device__ __forceinline__ void dd_add_unnorm(float &kh, float &kl, float rh, float rl) {
  const float t = __fadd_rn(kh, rh);
  const float bb = __fsub_rn(t, kh);
  const float e = __fadd_rn(__fsub_rn(kh, __fsub_rn(t, bb)), __fsub_rn(rh, bb));
  kh = t;
  kl = __fadd_rn(__fadd_rn(kl, rl), e);
}

// Cross-lane sum of NV double-float values per lane (vh + vl): the
// transpose-reduce of transpose_reduce<T, NV> in double-float; lane i holds
// the total of value index i / (32 / NV).  FP32 pipe only: this part's FP64
// pipe runs at ~1/64 of the FP32 rate.
template <int NV>
__device__ __forceinline__ dd transpose_reduce_dd(float (&vh)[NV], float (&vl)[NV], int lane) {
  constexpr int R = 32 / NV;
#pragma unroll
  for (int s = 16; s >= R; s >>= 1) {
    const int h = s / R;
    const bool upper = (lane & s) != 0;
#pragma unroll
    for (int j = 0; j < h; ++j) {
      const float sh = upper ? vh[j] : vh[j + h];
      const float sl = upper ? vl[j] : vl[j + h];
      float kh = upper ? vh[j + h] : vh[j];
      float kl = upper ? vl[j + h] : vl[j];
      dd_add_unnorm(kh, kl, __shfl_xor_sync(0xffffffffu, sh, s),
                    __shfl_xor_sync(0xffffffffu, sl, s));
      vh[j] = kh;
      vl[j] = kl;
    }
  }
#pragma unroll
  for (int s = R / 2; s >= 1; s >>= 1)
    dd_add_unnorm(vh[0], vl[0], __shfl_xor_sync(0xffffffffu, vh[0], s),
                  __shfl_xor_sync(0xffffffffu, vl[0], s));
  return {vh[0], vl[0]};
}

// l values per chunk of the double-float analysis: its chunk body (LC l x
// DD_NP_ANA ring pairs of double-float arithmetic, fully unrolled) must fit
// the instruction cache (16 l: ~3500 instructions, stalled on instruction
// fetch)
constexpr int DD_LC_ANA = 8;


// synthesis: as k_legendre_synth (one CTA row per m, one thread per
// DD_NP_SYN ring pairs), E/O parity sums in df64
__global__ void __launch_bounds__(SYN_THREADS)
    k_legendre_synth_dd(const RingPair *__restrict__ pairs, int npairs, int lmax,
                        const float2 *__restrict__ rcdd, const int *__restrict__ seed_l,
                        const double2 *__restrict__ seed_u, const float4 *__restrict__ xs,
                        float4 *__restrict__ F, const SolverState *__restrict__ st,
                        int lstatic) {
  constexpr int NP = DD_NP_SYN;
  const int m = blockIdx.y;
  int L = lstatic;
  if (st) {
    if (st->done) return;
    L = st->lcur;
  }
  if (m > L) return;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int nl = L - m + 1;
  dd *sxr = reinterpret_cast<dd *>(smraw);
  dd *sxi = sxr + nl;
  dd *sc = sxi + nl;
  const long base = lm_index(lmax, m, m);
  for (int j = threadIdx.x; j < nl; j += blockDim.x) {
    const float4 xv = xs[base + j];
    const float2 cv = rcdd[base + j];
    sxr[j] = {xv.x, xv.y};
    sxi[j] = {xv.z, xv.w};
    sc[j] = {cv.x, cv.y};
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int pair0 = (blockIdx.x * (SYN_THREADS / 32) + warp) * 32 * NP;
  if (pair0 >= npairs) return;
  const dd zero = {0.f, 0.f};
  dd z[NP], u1[NP], u2[NP], s0[NP], s1[NP], er[NP], ei[NP], orr[NP], oi[NP];
  int ls[NP];
  int lmin = INT_MAX, linj = -1;
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    const int k = pair0 + lane + 32 * j;
    u1[j] = u2[j] = er[j] = ei[j] = orr[j] = oi[j] = zero;
    z[j] = s0[j] = s1[j] = zero;
    ls[j] = INT_MAX - 2;
    if (k < npairs) {
      z[j] = dd_of(pairs[k].z);
      ls[j] = seed_l[(long)m * npairs + k];
      const double2 su = seed_u[(long)m * npairs + k];
      s0[j] = dd_of(su.x);
      s1[j] = dd_of(su.y);
    }
    if (ls[j] <= L) {
      lmin = min(lmin, ls[j]);
      linj = max(linj, ls[j] + 1);
    }
  }
  lmin = warp_min(lmin);
  linj = warp_max(linj);
  // one l at a time: seeds may enter (inj), parity of l - m picks the sums
  auto step = [&](int l, bool inj) {
    const dd c = sc[l - m], xr = sxr[l - m], xi = sxi[l - m];
    const bool even = ((l - m) & 1) == 0;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      dd u = dd_rec(c, z[j], u1[j], u2[j]);
      if (inj) {
        u = (l == ls[j]) ? s0[j] : u;
        u = (l == ls[j] + 1) ? s1[j] : u;
      }
      u2[j] = u1[j];
      u1[j] = u;
      if (even) {
        dd_acc(er[j], u, xr);
        dd_acc(ei[j], u, xi);
      } else {
        dd_acc(orr[j], u, xr);
        dd_acc(oi[j], u, xi);
      }
    }
  };
  int l = lmin;
  for (; l <= L && l <= linj; ++l) step(l, true);
  if (l <= L && ((l - m) & 1)) step(l++, false);
  // plain recurrence two l at a time (l - m even, then odd): the same
  // operations in the same order, without the parity branch and with the
  // u_{l-1}, u_{l-2} rotation left to register renaming
  for (; l + 1 <= L; l += 2) {
    const dd c0 = sc[l - m], xr0 = sxr[l - m], xi0 = sxi[l - m];
    const dd c1 = sc[l + 1 - m], xr1 = sxr[l + 1 - m], xi1 = sxi[l + 1 - m];
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      const dd w = dd_rec(c0, z[j], u1[j], u2[j]);
      dd_acc(er[j], w, xr0);
      dd_acc(ei[j], w, xi0);
      const dd v = dd_rec(c1, z[j], w, u1[j]);
      dd_acc(orr[j], v, xr1);
      dd_acc(oi[j], v, xi1);
      u2[j] = w;
      u1[j] = v;
    }
  }
  if (l <= L) step(l, false);
  const long stride = lmax + 1;
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    const int k = pair0 + lane + 32 * j;
    if (k >= npairs) continue;
    const RingPair &rp = pairs[k];
    // north = E + O, south = E - O, as double-float pairs (re hi, re lo,
    // im hi, im lo): the double-float ring transform reads them unconverted
    const dd nr = dd_add(er[j], orr[j]), ni = dd_add(ei[j], oi[j]);
    F[2 * ((long)m * npairs + k)] = make_float4(nr.hi, nr.lo, ni.hi, ni.lo);
    if (rp.ringS >= 0) {
      const dd sr = dd_sub(er[j], orr[j]), si = dd_sub(ei[j], oi[j]);
      F[2 * ((long)m * npairs + k) + 1] = make_float4(sr.hi, sr.lo, si.hi, si.lo);
    }
  }
}

// analysis: queue-scheduled like k_legendre_anal_q; per (m, tile of 32
// DD_NP_ANA ring pairs) item, per chunk of DD_LC_ANA l the lane's df64 sums
// are reduced across the warp in double-float (transpose_reduce_dd) and
// rounded to FP64 once per output
__global__ void __launch_bounds__(ANA_THREADS)
    k_legendre_anal_dd(const RingPair *__restrict__ pairs, int npairs, int lmax, long nalm,
                       const float2 *__restrict__ rcdd, const int *__restrict__ seed_l,
                       const double2 *__restrict__ seed_u, const float4 *__restrict__ G,
                       double *__restrict__ scratch, int *__restrict__ lstart,
                       int *__restrict__ counter, const SolverState *__restrict__ st,
                       int lstatic) {
  constexpr int NP = DD_NP_ANA;
  int L = lstatic;
  if (st) {
    if (st->done) return;
    L = st->lcur;
  }
  if (L < 0) return;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  extern __shared__ __align__(16) unsigned char smraw[];
  dd *sc = reinterpret_cast<dd *>(smraw) + (long)warp * (lmax + 1);
  constexpr int TP = 32 * NP;
  const int ntiles = (npairs + TP - 1) / TP;
  const int nitems = (L + 1) * ntiles;
  const long stride = lmax + 1;
  const dd zero = {0.f, 0.f};
  for (;;) {
    int item = 0;
    if (lane == 0) item = atomicAdd(counter, 1);
    item = __shfl_sync(0xffffffffu, item, 0);
    if (item >= nitems) break;
    const int m = item / ntiles, tile = item - m * ntiles;
    const long base = lm_index(lmax, m, m);
    const int pair0 = tile * TP;
    dd z[NP], u1[NP], u2[NP], s0[NP], s1[NP], pr[NP], pim[NP], qr[NP], qim[NP];
    int ls[NP];
    int lmin = INT_MAX, linj = -1;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      const int k = pair0 + lane + 32 * j;
      u1[j] = u2[j] = z[j] = s0[j] = s1[j] = pr[j] = pim[j] = qr[j] = qim[j] = zero;
      ls[j] = INT_MAX - 2;
      if (k < npairs) {
        const RingPair &rp = pairs[k];
        z[j] = dd_of(rp.z);
        ls[j] = seed_l[(long)m * npairs + k];
        const double2 su = seed_u[(long)m * npairs + k];
        s0[j] = dd_of(su.x);
        s1[j] = dd_of(su.y);
        // ring coefficients as double-float pairs (re hi, re lo, im hi, im lo)
        const float4 gn = G[2 * ((long)m * npairs + k)];
        float4 gs = make_float4(0.f, 0.f, 0.f, 0.f);
        if (rp.ringS >= 0) gs = G[2 * ((long)m * npairs + k) + 1];
        const dd nre = {gn.x, gn.y}, nim = {gn.z, gn.w};
        const dd sre = {gs.x, gs.y}, sim = {gs.z, gs.w};
        pr[j] = dd_add(nre, sre);
        pim[j] = dd_add(nim, sim);
        qr[j] = dd_sub(nre, sre);
        qim[j] = dd_sub(nim, sim);
      }
      if (ls[j] <= L) {
        lmin = min(lmin, ls[j]);
        linj = max(linj, ls[j] + 1);
      }
    }
    lmin = warp_min(lmin);
    linj = warp_max(linj);
    constexpr int LC = DD_LC_ANA;
    const int lc0 = lmin <= L ? m + ((lmin - m) / LC) * LC : L + 1;
    if (lane == 0) lstart[(long)m * ntiles + tile] = lc0;
    if (lmin > L) continue;
    __syncwarp();
    for (int j = lane; j <= L - m; j += 32) {
      const float2 cv = rcdd[base + j];
      sc[j] = {cv.x, cv.y};
    }
    __syncwarp();
    double *out = scratch + 2 * ((long)tile * nalm + base - m);  // out[2 l + re/im]
    for (int lc = lc0; lc <= L; lc += LC) {
      float vh[2 * LC], vl[2 * LC];
      const bool inj = lc <= linj;
#pragma unroll
      for (int jj = 0; jj < LC; ++jj) {
        const int l = lc + jj;
        dd ar = zero, ai = zero;
        if (l <= L) {
          const dd c = sc[l - m];
          const bool even = (jj & 1) == 0;  // lc - m is a multiple of LC (even)
#pragma unroll
          for (int j = 0; j < NP; ++j) {
            dd u = dd_rec(c, z[j], u1[j], u2[j]);
            if (inj) {
              u = (l == ls[j]) ? s0[j] : u;
              u = (l == ls[j] + 1) ? s1[j] : u;
            }
            u2[j] = u1[j];
            u1[j] = u;
            dd_acc(ar, u, even ? pr[j] : qr[j]);
            dd_acc(ai, u, even ? pim[j] : qim[j]);
          }
        }
        vh[2 * jj] = ar.hi;
        vl[2 * jj] = ar.lo;
        vh[2 * jj + 1] = ai.hi;
        vl[2 * jj + 1] = ai.lo;
      }
      const dd tot = transpose_reduce_dd<2 * LC>(vh, vl, lane);
      constexpr int R = 16 / LC;  // lanes holding each total
      const int idx = lane / R;
      const int l = lc + (idx >> 1);
      if (lane % R == 0 && l <= L) out[2 * l + (idx & 1)] = dd_val(tot);
    }
  }
}

// double-float transforms for the anchors of the mixed solver (FP64 in and
// out; see the kernels above)
wf_status launch_legendre_synth_dd(const Plan &P, const float4 *xs, float4 *F,
                                   const SolverState *st, int lstatic) {
  const size_t smem = 3 * sizeof(dd) * (P.lmax + 1);
  const int pairs_per_cta = SYN_THREADS * DD_NP_SYN;
  dim3 grid((P.npairs + pairs_per_cta - 1) / pairs_per_cta, P.lmax + 1);
  ++P.nlaunch;
  k_legendre_synth_dd<<<grid, SYN_THREADS, smem, P.stream>>>(
      P.pairs, P.npairs, P.lmax, P.rcdd, P.seed_l, P.seed_u, xs, F, st, lstatic);
  WF_CUDA(cudaGetLastError());
  return WF_OK;
}

wf_status launch_legendre_anal_dd(const Plan &P, const float4 *G, double2 *x,
                                  const SolverState *st, int mode, int lstatic,
                                  const double2 *src) {
  const size_t smem = sizeof(dd) * (P.lmax + 1) * ANA_WARPS;
  const int ntiles = (P.npairs + 32 * DD_NP_ANA - 1) / (32 * DD_NP_ANA);
  // one resident wave (occupancy queried once; the anchor steps that call
  // this are plain launches, never captured)
  static std::atomic<int> per_sm_cache{0};
  int per_sm = per_sm_cache.load();
  if (per_sm == 0) {
    int n = 0;
    WF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_legendre_anal_dd,
                                                          ANA_THREADS, smem));
    per_sm = std::max(1, std::min(n, ANA_Q_CTAS_PER_SM));
    per_sm_cache.store(per_sm);
  }
  double *scratch = reinterpret_cast<double *>(P.ana_scratch);
  ++P.nlaunch;
  k_legendre_anal_dd<<<P.num_sms * per_sm, ANA_THREADS, smem, P.stream>>>(
      P.pairs, P.npairs, P.lmax, P.nalm, P.rcdd, P.seed_l, P.seed_u, G, scratch,
      P.ana_lstart, P.ana_counter, st, lstatic);
  WF_CUDA(cudaGetLastError());
  ++P.nlaunch;
  k_anal_combine<<<P.lmax + 1, ANA_THREADS, 0, P.stream>>>(
      P.lmax, P.nalm, ntiles, scratch, P.ana_lstart, P.ana_counter, P.rg, P.cl_d, P.omega,
      x, P.partials, src, st, mode, lstatic);
  WF_CUDA(cudaGetLastError());
  return WF_OK;
}

// Dynamic shared memory limit of a kernel: `big`, less what its own static
// shared memory (the FP32 analysis kernels' reduction buffer) takes of the
// per-block limit.
template <typename K>
static cudaError_t set_dyn_smem(K kern, int big) {
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, kern);
  if (e != cudaSuccess) return e;
  int dev = 0, optin = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) !=
      cudaSuccess)
    return e;
  const int room = optin - (int)fa.sharedSizeBytes;
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              big < room ? big : room);
}

wf_status init_legendre_attributes() {
  const int big = 220 * 1024;
  WF_CUDA(set_dyn_smem(k_legendre_synth_dd, big));
  WF_CUDA(set_dyn_smem(k_legendre_anal_dd, big));
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

// the synthesis input of the double-float transforms: g_lm x_lm (FP64
// product) as double-float pairs (re hi, re lo, im hi, im lo)
__global__ void k_prescale_dd(const double2 *__restrict__ x, const double *__restrict__ rg,
                              int lmax, float4 *__restrict__ xs) {
  const int m = blockIdx.x;
  const long base = lm_index(lmax, m, m) - m;
  for (int l = m + threadIdx.x; l <= lmax; l += blockDim.x) {
    const long i = base + l;
    const dd re = dd_of(rg[i] * x[i].x), im = dd_of(rg[i] * x[i].y);
    xs[i] = make_float4(re.hi, re.lo, im.hi, im.lo);
  }
}

wf_status launch_prescale_dd(const Plan &P, const double2 *x, float4 *xs) {
  ++P.nlaunch;
  k_prescale_dd<<<P.lmax + 1, 128, 0, P.stream>>>(x, P.rg, P.lmax, xs);
  WF_CUDA(cudaGetLastError());
  return WF_OK;
}

}  // namespace wf
