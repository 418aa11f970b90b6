// fft.cuh -- power-of-two FFTs of one sequence in shared memory by a whole CTA, in
// FP64, FP32 and double-float, for the ring transforms (ringfft.cu) and the flat sky
// (flatsky.cu): decimation in frequency (natural -> bit-reversed order) and in time
// (bit-reversed -> natural), so that no permutation pass is needed.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <vector>

namespace wf {

template <typename T2> struct CT;
template <> struct CT<double2> {
  typedef double T;
  typedef double2 G;  // element type of the global data arrays (F, G)
  typedef double2 W;  // element type of the tables (twiddles, chirps)
  static __device__ __forceinline__ double2 ld(const G *p) { return *p; }
  static __device__ __forceinline__ double2 ldw(const W *p) { return *p; }
  static __device__ __forceinline__ void st(G *p, double2 v) { *p = v; }
  static __device__ __forceinline__ double2 mk(double a, double b) {
    return make_double2(a, b);
  }
  // sin, cos of pi r / den
  static __device__ __forceinline__ void sincospi_(int r, int den, double *s,
                                                   double *c) {
    sincospi((double)r / (double)den, s, c);
  }
};
template <> struct CT<float2> {
  typedef float T;
  typedef float2 G;
  typedef float2 W;
  static __device__ __forceinline__ float2 ld(const G *p) { return *p; }
  static __device__ __forceinline__ float2 ldw(const W *p) { return *p; }
  static __device__ __forceinline__ void st(G *p, float2 v) { *p = v; }
  static __device__ __forceinline__ float2 mk(float a, float b) {
    return make_float2(a, b);
  }
  static __device__ __forceinline__ void sincospi_(int r, int den, float *s,
                                                   float *c) {
    sincospif((float)r / (float)den, s, c);
  }
};

// one entry of the twiddle table (TwPass)
template <typename T2> struct alignas(16) TwPair { typename CT<T2>::W a, b; };

template <typename T2>
__device__ __forceinline__ T2 cmul(T2 a, T2 b) {
  return CT<T2>::mk(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename T2>
__device__ __forceinline__ T2 cmulc(T2 a, T2 b) {  // a * conj(b)
  return CT<T2>::mk(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
template <typename T2>
__device__ __forceinline__ T2 cadd(T2 a, T2 b) {
  return CT<T2>::mk(a.x + b.x, a.y + b.y);
}
template <typename T2>
__device__ __forceinline__ T2 csub(T2 a, T2 b) {
  return CT<T2>::mk(a.x - b.x, a.y - b.y);
}
template <typename T2>
__device__ __forceinline__ T2 cconj(T2 a) {
  return CT<T2>::mk(a.x, -a.y);
}

// multiply by -i (forward) or +i (inverse)
template <typename T2, bool INV>
__device__ __forceinline__ T2 rot_q(T2 a) {
  return INV ? CT<T2>::mk(-a.y, a.x) : CT<T2>::mk(a.y, -a.x);
}

// Shared-memory layout of the FFT buffer: element i is stored at
// sw(i) = i ^ (h(i >> 4) & 15), h(b) = b ^ (b << 2) -- an XOR inside each
// aligned block of 16 complex values.  Unit-stride sweeps stay conflict-free,
// and the radix-2^2 passes of short span (whose four operands sit 1..8
// elements apart, 16 lanes in the same few banks) spread over all banks:
// with it every pass of every power-of-two length needs the minimum number
// of shared-memory wavefronts.
__device__ __forceinline__ int sw(int i) {
  const int b = i >> 4;
  return i ^ ((b ^ (b << 2)) & 15);
}

// Twiddles of one pass of span h: pair(j), j < h / 2, gives W_2h^j = e^{-i pi j / h}
// and W_h^j = (W_2h^j)^2, side by side in a table that holds every span's entries at
// h / 2 - 1 (twiddle_table: Mmax / 2 - 1 entries for lengths up to Mmax), one vector load
// per butterfly instead of two scattered ones or a complex square (FP32 transform pair at
// Nside 256: 156 -> 144 us with the chirp tables in shared memory, flat solve at n = 256
// 1.10 times as fast).  The table
// (16 KB in FP32 for 2048 points) stays in L1; computing the pair in FP32 by sincospi
// took 40 of a butterfly's ~100 instructions.
template <typename T2>
struct TwPass {
  const TwPair<T2> *t;
  __device__ __forceinline__ TwPass(int h, const TwPair<T2> *tw) : t(tw + (h / 2 - 1)) {}
  __device__ __forceinline__ void pair(int j, T2 &w2h, T2 &wh) const {
    const TwPair<T2> v = t[j];
    w2h = CT<T2>::ldw(&v.a);
    wh = CT<T2>::ldw(&v.b);
  }
};

// ---------------------------------------------------------- double-float
// ddr: an unevaluated sum hi + lo of two floats (~48-bit significand) with
// the operations the ring transforms use -- sums by two-sum, products by
// the FMA two-product, one normalisation each (Dekker, Knuth); explicit _rn
// intrinsics, so nothing is contracted or reassociated.  The mixed solver's
// anchor steps run their ring FFTs in it on the FP32 pipe: this part's FP64
// pipe runs at ~1/64 of the FP32 rate, and those FFTs were FP64-bound.
// The ring coefficients F, G (written and read by the double-float Legendre
// kernels), the twiddle, chirp, kernel-spectrum and phase tables and the
// pixel step's d and sigma^2 are kept as (hi, lo) float pairs, so no FP64
// arithmetic is left but the maps of the API's own FP64 input and output.
struct ddr {
  float hi, lo;
  __device__ __forceinline__ ddr() : hi(0.f), lo(0.f) {}
  __device__ __forceinline__ ddr(float h, float l) : hi(h), lo(l) {}
  __device__ __forceinline__ ddr(int v) : hi((float)v), lo(0.f) {}
  __device__ __forceinline__ ddr(double v) {
    hi = (float)v;
    lo = (float)(v - (double)hi);
  }
  __device__ __forceinline__ explicit operator double() const {
    return (double)hi + (double)lo;
  }
};
__device__ __forceinline__ ddr ddr_norm(float s, float e) {
  const float h = __fadd_rn(s, e);
  return ddr(h, __fsub_rn(e, __fsub_rn(h, s)));
}
__device__ __forceinline__ ddr operator+(ddr a, ddr b) {
  const float s = __fadd_rn(a.hi, b.hi);
  const float bb = __fsub_rn(s, a.hi);
  const float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(b.hi, bb));
  return ddr_norm(s, __fadd_rn(e, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ ddr operator-(ddr a) { return ddr(-a.hi, -a.lo); }
__device__ __forceinline__ ddr operator-(ddr a, ddr b) { return a + (-b); }
__device__ __forceinline__ ddr operator*(ddr a, ddr b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, e));
  return ddr_norm(p, e);
}
__device__ __forceinline__ ddr &operator*=(ddr &a, ddr b) {
  a = a * b;
  return a;
}
// a / b: the quotient of the hi parts, corrected by the remainder a - q b
// (finite b only)
__device__ __forceinline__ ddr operator/(ddr a, ddr b) {
  const float q1 = __fdiv_rn(a.hi, b.hi);
  const ddr r = a - ddr(q1, 0.f) * b;
  return ddr_norm(q1, __fdiv_rn(r.hi, b.hi));
}
__device__ __forceinline__ bool operator<(ddr a, ddr b) {
  return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo);
}

struct ddc {
  ddr x, y;
};
template <> struct CT<ddc> {
  typedef ddr T;
  typedef float4 G;  // F, G as double-float pairs (re hi, re lo, im hi, im lo)
  typedef float4 W;  // tables in the same form
  static __device__ __forceinline__ ddc ld(const G *p) {
    const float4 v = *p;
    return {ddr(v.x, v.y), ddr(v.z, v.w)};
  }
  static __device__ __forceinline__ ddc ldw(const W *p) {
    const float4 v = *p;
    return {ddr(v.x, v.y), ddr(v.z, v.w)};
  }
  static __device__ __forceinline__ void st(G *p, ddc v) {
    *p = make_float4(v.x.hi, v.x.lo, v.y.hi, v.y.lo);
  }
  static __device__ __forceinline__ ddc mk(ddr a, ddr b) { return {a, b}; }
  // sin, cos of pi r / den, rounded from FP64
  static __device__ __forceinline__ void sincospi_(int r, int den, ddr *s, ddr *c) {
    double sd, cd;
    sincospi((double)r / (double)den, &sd, &cd);
    *s = ddr(sd);
    *c = ddr(cd);
  }
};
// natural -> bit-reversed; INV uses e^{+2 pi i jk/M}.  Two radix-2 stages
// (spans h and h/2) per pass over shared memory ("radix-2^2"): the output
// order stays bit-reversed, and the barriers and shared-memory round trips
// halve.  An odd number of stages ends with one radix-2 pass of span 1.
// Where the twiddle index j = b mod q is the same for all of a thread's
// butterflies (q <= blockDim), the twiddles are loaded once per pass.
template <typename T2, bool INV>
__device__ void fft_dif(T2 *buf, int M, const TwPair<T2> *__restrict__ tw) {
  int h = M >> 1;
  for (; h >= 2; h >>= 2) {
    const int q = h >> 1;
    const TwPass<T2> tp(h, tw);
    const bool fixed = q <= (int)blockDim.x;
    T2 w1f, w2f;
    if (fixed) tp.pair((int)threadIdx.x & (q - 1), w1f, w2f);
    #pragma unroll 4
    for (int b = threadIdx.x; b < (M >> 2); b += blockDim.x) {
      const int j = b & (q - 1);
      const int i0 = ((b - j) << 2) + j, i1 = i0 + q, i2 = i0 + h, i3 = i2 + q;
      T2 w1 = w1f, w2 = w2f;  // W_2h^j, W_h^j
      if (!fixed) tp.pair(j, w1, w2);
      const T2 x0 = buf[sw(i0)], x1 = buf[sw(i1)], x2 = buf[sw(i2)], x3 = buf[sw(i3)];
      const T2 a0 = cadd(x0, x2), a1 = cadd(x1, x3);
      const T2 a2 = INV ? cmulc(csub(x0, x2), w1) : cmul(csub(x0, x2), w1);
      const T2 a3 = rot_q<T2, INV>(INV ? cmulc(csub(x1, x3), w1) : cmul(csub(x1, x3), w1));
      buf[sw(i0)] = cadd(a0, a1);
      buf[sw(i1)] = INV ? cmulc(csub(a0, a1), w2) : cmul(csub(a0, a1), w2);
      buf[sw(i2)] = cadd(a2, a3);
      buf[sw(i3)] = INV ? cmulc(csub(a2, a3), w2) : cmul(csub(a2, a3), w2);
    }
    __syncthreads();
  }
  if (h == 1) {
    for (int b = threadIdx.x; b < (M >> 1); b += blockDim.x) {
      const T2 a = buf[sw(2 * b)], c = buf[sw(2 * b + 1)];
      buf[sw(2 * b)] = cadd(a, c);
      buf[sw(2 * b + 1)] = csub(a, c);
    }
    __syncthreads();
  }
}

// bit-reversed -> natural; an odd number of stages starts with one radix-2
// pass of span 1, then pairs of stages (spans h and 2h) per pass
template <typename T2, bool INV>
__device__ void fft_dit(T2 *buf, int M, const TwPair<T2> *__restrict__ tw) {
  int h = 1;
  int bits = 0;
  while ((1 << bits) < M) ++bits;
  if (bits & 1) {
    for (int b = threadIdx.x; b < (M >> 1); b += blockDim.x) {
      const T2 a = buf[sw(2 * b)], c = buf[sw(2 * b + 1)];
      buf[sw(2 * b)] = cadd(a, c);
      buf[sw(2 * b + 1)] = csub(a, c);
    }
    __syncthreads();
    h = 2;
  }
  for (; h < M; h <<= 2) {
    const TwPass<T2> tp(2 * h, tw);  // pair(j) = (W_4h^j, W_2h^j)
    const bool fixed = h <= (int)blockDim.x;
    T2 waf, wbf;
    if (fixed) tp.pair((int)threadIdx.x & (h - 1), wbf, waf);
    #pragma unroll 4
    for (int b = threadIdx.x; b < (M >> 2); b += blockDim.x) {
      const int j = b & (h - 1);
      const int i0 = ((b - j) << 2) + j, i1 = i0 + h, i2 = i0 + 2 * h, i3 = i2 + h;
      T2 wa = waf, wb = wbf;  // W_2h^j, W_4h^j
      if (!fixed) tp.pair(j, wb, wa);
      const T2 x0 = buf[sw(i0)], x1 = buf[sw(i1)], x2 = buf[sw(i2)], x3 = buf[sw(i3)];
      const T2 c1 = INV ? cmulc(x1, wa) : cmul(x1, wa);
      const T2 c3 = INV ? cmulc(x3, wa) : cmul(x3, wa);
      const T2 a0 = cadd(x0, c1), a1 = csub(x0, c1);
      const T2 a2 = cadd(x2, c3), a3 = csub(x2, c3);
      const T2 d2 = INV ? cmulc(a2, wb) : cmul(a2, wb);
      const T2 d3 = rot_q<T2, INV>(INV ? cmulc(a3, wb) : cmul(a3, wb));
      buf[sw(i0)] = cadd(a0, d2);
      buf[sw(i2)] = csub(a0, d2);
      buf[sw(i1)] = cadd(a1, d3);
      buf[sw(i3)] = csub(a1, d3);
    }
    __syncthreads();
  }
}

__device__ __forceinline__ int bitrev_n(int x, int bits) {
  return (int)(__brev((unsigned)x) >> (32 - bits));
}

// the host table of TwPass in FP64: a = e^{-i pi j / h}, b = e^{-2 i pi j / h}
inline std::vector<TwPair<double2>> twiddle_table(int Mmax) {
  std::vector<TwPair<double2>> t(std::max(1, Mmax / 2 - 1));
  for (int h = 2; h <= Mmax / 2; h <<= 1)
    for (int j = 0; j < h / 2; ++j) {
      const double x = M_PI * (double)j / (double)h;
      t[h / 2 - 1 + j] = {make_double2(cos(x), -sin(x)), make_double2(cos(2.0 * x), -sin(2.0 * x))};
    }
  return t;
}

}  // namespace wf
