// nn.cu -- the learned warm start: a small network that maps (d, log sigma^2,
// mask) to an initial messenger field t0 and initial signal coefficients a0,
// with its forward pass, backward pass and Adam update as CUDA kernels.
//
// Network (weights kept in FP32, used rounded to BF16 when bf16 = 1; all
// accumulation in FP32):
//   input channels per pixel (observed: 1 - m, masked: m = 1):
//     c0 = (1-m) d / sigma_d, c1 = (1-m) (log sigma^2 - mu) / s, c2 = m
//   per-ring circular 1-D convolutions (kernel K, zero-based taps centred):
//     h1 = relu(W1 * c + b1)   (3 -> H channels)
//     h2 = relu(W2 * h1 + b2)  (H -> H)
//     r  = W3 * h2 + b3        (H -> 1)
//   t0 = (1-m) d + sigma_d r                       (messenger warm start)
//   a  = Omega Y^T t0                              (FP32 transform)
//   per-l MLP on features f_l = (l/lmax, log C_l, log P_d(l)/C_l,
//   log alpha Omega / C_l): q_l = sigmoid(V3 relu(V2 relu(V1 f_l + c1) + c2) + c3)
//   a0_lm = q_l a_lm                               (signal warm start)
// Loss: L = sum w |a0 - a*|^2 / sum w |a*|^2 against the solver's solution a*
// (real-basis weights w = 1 for m = 0, 2 for m > 0).
#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>
#include <vector>

#include "wf_internal.cuh"

struct wf_net_s;

namespace wf {

struct Net {
  Plan *P = nullptr;
  int H = 16, K = 9, Hm = 32, bf16 = 1;
  long npar = 0, nconv = 0, nmlp = 0;
  long oW1, ob1, oW2, ob2, oW3, ob3, oV1, oc1, oV2, oc2, oV3, oc3;
  float *par = nullptr, *grad = nullptr, *am = nullptr, *av = nullptr;
  long step = 0;
  int2 *quads = nullptr;    // [npix/4]: first quad and number of quads of its ring
  int4 *tiles = nullptr;    // weight-gradient tiles: ring's first quad, quads, first quad
  int ntiles = 0;
  float *in = nullptr, *h1 = nullptr, *h2 = nullptr, *r = nullptr;   // activations
  float *g1 = nullptr, *g2 = nullptr, *g3 = nullptr;                 // their gradients
  double *t0 = nullptr, *dmask = nullptr, *gmap = nullptr;
  double2 *a = nullptr, *ad = nullptr, *a0 = nullptr, *b = nullptr;
  float *feat = nullptr, *m1 = nullptr, *m2 = nullptr, *q = nullptr, *dq = nullptr;
  float *mpart = nullptr;   // [lmax+1][nmlp] per-l gradient contributions
  float *wpart = nullptr;   // conv weight-gradient partials
  double *red = nullptr;
  double sig_d = 1.0, mu_log = 0.0, sd_log = 1.0;
  int have_grad = 0;
};

constexpr int NN_THREADS = 256;
constexpr int NN_PARTS = 304;   // CTAs (partial sums) of a weight gradient
constexpr int NN_TQ = 64;       // quads of pixels per weight-gradient tile
constexpr int NN_MAXC = 32;     // max channels
constexpr int NN_MAXK = 15;     // max kernel width
constexpr int NN_MAXHM = 64;    // max MLP width
constexpr int NN_FEAT = 4;

__device__ __forceinline__ float wround(float w, int bf16) {
  return bf16 ? __bfloat162float(__float2bfloat16_rn(w)) : w;
}

// ---------------------------------------------------------------- inputs
// also leaves log sigma^2 in lgout (an FP64 logarithm is most of this kernel's time)
__global__ void k_nn_stats(const double *d, const double *nvar, long npix, double *out,
                           double *lgout) {
  __shared__ double s[4][NN_THREADS];
  double a = 0, b = 0, c = 0, n = 0;
  for (long p = (long)blockIdx.x * blockDim.x + threadIdx.x; p < npix;
       p += (long)gridDim.x * blockDim.x) {
    const double v = nvar[p];
    if (isinf(v)) continue;
    const double lg = log(v);
    lgout[p] = lg;
    a += d[p] * d[p];
    b += lg;
    c += lg * lg;
    n += 1.0;
  }
  s[0][threadIdx.x] = a;
  s[1][threadIdx.x] = b;
  s[2][threadIdx.x] = c;
  s[3][threadIdx.x] = n;
  __syncthreads();
  for (int k = blockDim.x / 2; k > 0; k >>= 1) {
    if (threadIdx.x < k)
      for (int j = 0; j < 4; ++j) s[j][threadIdx.x] += s[j][threadIdx.x + k];
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int j = 0; j < 4; ++j) out[4 * blockIdx.x + j] = s[j][0];
}

__global__ void k_nn_inputs(const double *d, const double *nvar, const double *lg, long npix,
                            double inv_sig, double mu, double inv_sd, float *in,
                            double *dmask) {
  for (long p = (long)blockIdx.x * blockDim.x + threadIdx.x; p < npix;
       p += (long)gridDim.x * blockDim.x) {
    const double v = nvar[p];
    const bool m = isinf(v);
    in[p] = m ? 0.f : (float)(d[p] * inv_sig);
    in[npix + p] = m ? 0.f : (float)((lg[p] - mu) * inv_sd);
    in[2 * npix + p] = m ? 1.f : 0.f;
    dmask[p] = m ? 0.0 : d[p];
  }
}

// ---------------------------------------------------------------- convolution
// HEALPix rings have 4 i pixels and start at a multiple of 4, so pixels go in quads
// (one float4) that never straddle a ring, and a convolution's neighbours are quads of
// the same ring, wrapped by quads.
//
// Forward:   out[co][p] = b[co] + sum_{ci,k} W[co][ci][k] in[ci][ring(p, j + k - K/2)],
//            optionally ReLU.
// Backward (BWD; cin, cout are those of this product: the layer's outputs and inputs):
//            gin[ci][p] = mask(p) sum_{co,k} W[co][ci][k] gout[co][ring(p, j - (k - K/2))],
//            mask = (act[ci][p] > 0) where act is given (ReLU of the layer below).
// One thread per quad and CO output channels (4 CO accumulators): per input channel the
// quad's window comes in 2 ceil((K/2)/4) + 1 16-byte loads and serves 4 CO K
// multiply-adds on weights broadcast from shared memory, so the FP32 pipe bounds the
// 16 -> 16 layer (1.8 G multiply-adds at Nside 256, K = 9: 46 us of it) and the
// activations' traffic the others.  Measured there: 82 us forward, 90 us backward
// (1064 and 1083 us with one pixel per thread, wrapped by a modulo per tap).
template <int K, int CO, bool BWD>
__global__ void __launch_bounds__(NN_THREADS)
    k_nn_conv(const int2 *__restrict__ quads, long nquad, const float *__restrict__ in, int cin,
              const float *__restrict__ W, const float *__restrict__ bias, int cout, int relu,
              int bf16, const float *__restrict__ act, float *__restrict__ out) {
  constexpr int h = K / 2, D = (h + 3) / 4;
  extern __shared__ __align__(16) float sw[];  // [cin][K][CO]
  const int c0 = blockIdx.y * CO;
  for (int i = threadIdx.x; i < cin * K * CO; i += blockDim.x) {
    const int co = c0 + i % CO, k = (i / CO) % K, ci = i / (CO * K);
    float w = 0.f;
    if (co < cout) w = wround(BWD ? W[((long)ci * cout + co) * K + k] : W[((long)co * cin + ci) * K + k], bf16);
    sw[i] = w;
  }
  __syncthreads();
  const long q = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nquad) return;
  const int2 r = quads[q];
  const int jq = (int)(q - r.x);
  long at[2 * D + 1];
#pragma unroll
  for (int d = -D; d <= D; ++d) {
    int j = jq + d;
    while (j < 0) j += r.y;
    while (j >= r.y) j -= r.y;
    at[d + D] = r.x + j;
  }
  float acc[CO][4];
#pragma unroll
  for (int c = 0; c < CO; ++c) {
    const float b = (bias && c0 + c < cout) ? wround(bias[c0 + c], bf16) : 0.f;
#pragma unroll
    for (int x = 0; x < 4; ++x) acc[c][x] = b;
  }
  for (int ci = 0; ci < cin; ++ci) {
    const float4 *src = reinterpret_cast<const float4 *>(in) + ci * nquad;
    float x[4 * (2 * D + 1)];
#pragma unroll
    for (int d = 0; d <= 2 * D; ++d) {
      const float4 v = src[at[d]];
      x[4 * d] = v.x;
      x[4 * d + 1] = v.y;
      x[4 * d + 2] = v.z;
      x[4 * d + 3] = v.w;
    }
    const float *wk = sw + ci * K * CO;
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
      for (int c = 0; c < CO; ++c) {
        const float w = wk[k * CO + c];
#pragma unroll
        for (int px = 0; px < 4; ++px)
          acc[c][px] = fmaf(w, x[4 * D + px + (BWD ? h - k : k - h)], acc[c][px]);
      }
  }
#pragma unroll
  for (int c = 0; c < CO; ++c) {
    if (c0 + c >= cout) break;
    float4 o = make_float4(acc[c][0], acc[c][1], acc[c][2], acc[c][3]);
    const long i = (long)(c0 + c) * nquad + q;
    if (relu) o = make_float4(fmaxf(o.x, 0.f), fmaxf(o.y, 0.f), fmaxf(o.z, 0.f), fmaxf(o.w, 0.f));
    if (act) {
      const float4 a = reinterpret_cast<const float4 *>(act)[i];
      o = make_float4(a.x > 0.f ? o.x : 0.f, a.y > 0.f ? o.y : 0.f, a.z > 0.f ? o.z : 0.f,
                      a.w > 0.f ? o.w : 0.f);
    }
    reinterpret_cast<float4 *>(out)[i] = o;
  }
}

// Partial sums of dW[co][ci][k] = sum_p gout[co][p] in[ci][ring(p, j + k - K/2)] and
// db[co] = sum_p gout[co][p] over tiles of NN_TQ quads (one ring each), part[CTA][(co
// (cin + 1) + ci) K + k] with ci = cin the bias.  The tile's channels are staged in
// shared memory once; one thread owns a (co, ci) pair (all K taps), and with fewer than
// 256 pairs S threads share one, each with every S-th quad.  Sums run per tile, then
// over the tiles, then over the S threads, in a fixed order.  16 x 16 channels, Nside
// 256, K = 9: 138 us (1897 us with a CTA per pair that read both maps again); the
// shared-memory loads, 2 ceil((K/2)/4) + 2 per 4 K multiply-adds, are its bound.
template <int K>
__global__ void __launch_bounds__(NN_THREADS)
    k_nn_conv_wgrad(const int4 *__restrict__ tiles, int ntiles, long nquad,
                    const float *__restrict__ gout, int cout, const float *__restrict__ in,
                    int cin, int lcin, int pairs2, float *__restrict__ part) {
  constexpr int h = K / 2, D = (h + 3) / 4, SG = NN_TQ + 1, SI = NN_TQ + 2 * D + 1;
  extern __shared__ __align__(16) float sw[];
  float4 *sg = reinterpret_cast<float4 *>(sw);  // [cout][SG]
  float4 *si = sg + cout * SG;                  // [cin][SI]
  const int P = min(pairs2, NN_THREADS), S = NN_THREADS / P;
  const int slice = threadIdx.x / P, pair = blockIdx.y * NN_THREADS + threadIdx.x % P;
  const int co = pair >> lcin, ci = pair & ((1 << lcin) - 1);
  const bool on = co < cout && ci < cin;
  float tot[K] = {}, totb = 0.f;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int4 tl = tiles[t];  // ring's first quad, its quads, the tile's first quad
    const int nq = min(NN_TQ, tl.y - tl.z);
    __syncthreads();
    for (int i = threadIdx.x; i < cout * NN_TQ; i += NN_THREADS) {
      const int c = i / NN_TQ, j = i % NN_TQ;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (j < nq) v = reinterpret_cast<const float4 *>(gout)[c * nquad + tl.x + tl.z + j];
      sg[c * SG + j] = v;
    }
    for (int i = threadIdx.x; i < cin * (SI - 1); i += NN_THREADS) {
      const int c = i / (SI - 1), j = i % (SI - 1);
      int jq = tl.z + j - D;
      while (jq < 0) jq += tl.y;
      while (jq >= tl.y) jq -= tl.y;
      si[c * SI + j] = reinterpret_cast<const float4 *>(in)[c * nquad + tl.x + jq];
    }
    __syncthreads();
    if (!on) continue;
    float acc[K] = {}, accb = 0.f;
    for (int j = slice; j < nq; j += S) {
      const float4 gv = sg[co * SG + j];
      const float g[4] = {gv.x, gv.y, gv.z, gv.w};
      float x[4 * (2 * D + 1)];
#pragma unroll
      for (int d = 0; d <= 2 * D; ++d) {
        const float4 v = si[ci * SI + j + d];
        x[4 * d] = v.x;
        x[4 * d + 1] = v.y;
        x[4 * d + 2] = v.z;
        x[4 * d + 3] = v.w;
      }
#pragma unroll
      for (int px = 0; px < 4; ++px) {
        accb += g[px];
#pragma unroll
        for (int k = 0; k < K; ++k) acc[k] = fmaf(g[px], x[4 * D + px + k - h], acc[k]);
      }
    }
#pragma unroll
    for (int k = 0; k < K; ++k) tot[k] += acc[k];
    totb += accb;
  }
  // the S threads of a pair, in order
  __syncthreads();
  float *red = sw;  // [K + 1][NN_THREADS]
#pragma unroll
  for (int k = 0; k < K; ++k) red[k * NN_THREADS + threadIdx.x] = tot[k];
  red[K * NN_THREADS + threadIdx.x] = totb;
  __syncthreads();
  if (slice != 0 || !on) return;
  float *o = part + (long)blockIdx.x * cout * (cin + 1) * K;
  for (int k = 0; k <= K; ++k) {
    float v = 0.f;
    for (int i = 0; i < S; ++i) v += red[k * NN_THREADS + i * P + threadIdx.x];
    if (k < K)
      o[(co * (cin + 1) + ci) * K + k] = v;
    else if (ci == 0)
      o[(co * (cin + 1) + cin) * K] = v;
  }
}

// fixed-order sum of the parts into the gradient vector: 32 outputs x 8 threads, each
// with every 8th part
__global__ void __launch_bounds__(NN_THREADS)
    k_nn_wgrad_reduce(const float *__restrict__ part, int nparts, int cout, int cin, int K,
                      float *__restrict__ gW, float *__restrict__ gb) {
  __shared__ float red[8][32];
  const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5;
  const int t = blockIdx.x * 32 + lane;
  const int nW = cout * cin * K;
  const long row = (long)cout * (cin + 1) * K;
  long at = -1;
  if (t < nW) {
    const int co = t / (cin * K), ci = (t / K) % cin, k = t % K;
    at = (long)(co * (cin + 1) + ci) * K + k;
  } else if (t < nW + cout) {
    at = (long)((t - nW) * (cin + 1) + cin) * K;
  }
  float v = 0.f;
  if (at >= 0)
    for (int c = sl; c < nparts; c += 8) v += part[c * row + at];
  red[sl][lane] = v;
  __syncthreads();
  if (sl != 0 || at < 0) return;
  for (int i = 1; i < 8; ++i) v += red[i][lane];
  if (t < nW)
    gW[t] = v;
  else
    gb[t - nW] = v;
}

__global__ void k_nn_make_t0(const double *dmask, const float *r, double sig_d, long npix,
                             double *t0) {
  for (long p = (long)blockIdx.x * blockDim.x + threadIdx.x; p < npix;
       p += (long)gridDim.x * blockDim.x)
    t0[p] = dmask[p] + sig_d * (double)r[p];
}

// ---------------------------------------------------------------- harmonic MLP
__device__ __forceinline__ long nn_idx(int lmax, int l, int m) {
  return (long)m * (2 * lmax + 1 - m) / 2 + l;
}

// sum over y of v (blockDim (32, Y)), fixed order; the result in threadIdx.y = 0
__device__ __forceinline__ double sum_y(double v, double (*sh)[33]) {
  sh[threadIdx.y][threadIdx.x] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.y == 0)
    for (int y = 0; y < (int)blockDim.y; ++y) s += sh[y][threadIdx.x];
  return s;
}

// 32 l per CTA (x: consecutive l, coalesced in the m-major layout), the m split over y
__global__ void k_nn_features(const double2 *ad, const double *cl, int lmax, double aom,
                              float *feat) {
  __shared__ double sh[32][33];
  const int l = blockIdx.x * 32 + threadIdx.x;
  double part = 0.0;
  if (l <= lmax)
    for (int m = threadIdx.y; m <= l; m += blockDim.y) {
      const double2 v = ad[nn_idx(lmax, l, m)];
      part += (m == 0 ? 1.0 : 2.0) * (v.x * v.x + v.y * v.y);
    }
  double pd = sum_y(part, sh);
  if (l > lmax || threadIdx.y != 0) return;
  pd /= (2.0 * l + 1.0);
  const double c = cl[l] + 1e-30;
  feat[NN_FEAT * l + 0] = (float)((double)l / lmax);
  feat[NN_FEAT * l + 1] = (float)fmin(fmax(log10(c) / 10.0, -4.0), 4.0);
  feat[NN_FEAT * l + 2] = (float)fmin(fmax(log10((pd + 1e-30) / c) / 5.0, -4.0), 4.0);
  feat[NN_FEAT * l + 3] = (float)fmin(fmax(log10(aom / c) / 5.0, -4.0), 4.0);
}

// one CTA per l, thread o = unit o: q_l = sigmoid(V3 relu(V2 relu(V1 f + c1) + c2) + c3)
__global__ void __launch_bounds__(NN_MAXHM)
    k_nn_mlp_fwd(const float *feat, const float *par, long oV1, long oc1, long oV2, long oc2,
                 long oV3, long oc3, int Hm, int lmax, int bf16, float *m1, float *m2,
                 float *q) {
  __shared__ float a1[NN_MAXHM], a2[NN_MAXHM];
  const int l = blockIdx.x, o = threadIdx.x;
  if (o < Hm) {
    float s = wround(par[oc1 + o], bf16);
    for (int i = 0; i < NN_FEAT; ++i)
      s = fmaf(wround(par[oV1 + o * NN_FEAT + i], bf16), feat[NN_FEAT * l + i], s);
    a1[o] = fmaxf(s, 0.f);
    m1[(long)l * Hm + o] = a1[o];
  }
  __syncthreads();
  if (o < Hm) {
    float s = wround(par[oc2 + o], bf16);
    for (int i = 0; i < Hm; ++i) s = fmaf(wround(par[oV2 + o * Hm + i], bf16), a1[i], s);
    a2[o] = fmaxf(s, 0.f);
    m2[(long)l * Hm + o] = a2[o];
  }
  __syncthreads();
  if (o == 0) {
    float s = wround(par[oc3], bf16);
    for (int i = 0; i < Hm; ++i) s = fmaf(wround(par[oV3 + i], bf16), a2[i], s);
    q[l] = 1.f / (1.f + expf(-s));
  }
}

// a0 = q_l a
__global__ void k_nn_gain(const double2 *a, const float *q, int lmax, double2 *a0) {
  const int m = blockIdx.x;
  for (int l = m + threadIdx.x; l <= lmax; l += blockDim.x) {
    const long i = nn_idx(lmax, l, m);
    a0[i] = make_double2(q[l] * a[i].x, q[l] * a[i].y);
  }
}

// per-m partial sums of sum w |a0 - a*|^2 and sum w |a*|^2
__global__ void k_nn_loss(const double2 *a0, const double2 *at, int lmax, double *part) {
  __shared__ double s0[128], s1[128];
  const int m = blockIdx.x;
  const double w = m == 0 ? 1.0 : 2.0;
  double e = 0.0, n = 0.0;
  for (int l = m + threadIdx.x; l <= lmax; l += blockDim.x) {
    const long i = nn_idx(lmax, l, m);
    const double dx = a0[i].x - at[i].x, dy = a0[i].y - at[i].y;
    e += w * (dx * dx + dy * dy);
    n += w * (at[i].x * at[i].x + at[i].y * at[i].y);
  }
  s0[threadIdx.x] = e;
  s1[threadIdx.x] = n;
  __syncthreads();
  for (int k = blockDim.x / 2; k > 0; k >>= 1) {
    if (threadIdx.x < k) {
      s0[threadIdx.x] += s0[threadIdx.x + k];
      s1[threadIdx.x] += s1[threadIdx.x + k];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    part[2 * m] = s0[0];
    part[2 * m + 1] = s1[0];
  }
}

// dL/dq_l = sum_m w 2 Re(conj(a0 - a*) a) / norm;  b = 2 q (a0 - a*) / norm
__global__ void k_nn_dq(const double2 *a0, const double2 *at, const double2 *a,
                        const float *q, int lmax, double inv_norm, float *dq, double2 *b) {
  __shared__ double sh[32][33];
  const int l = blockIdx.x * 32 + threadIdx.x;
  double part = 0.0;
  if (l <= lmax)
    for (int m = threadIdx.y; m <= l; m += blockDim.y) {
      const long i = nn_idx(lmax, l, m);
      const double w = m == 0 ? 1.0 : 2.0;
      const double dx = a0[i].x - at[i].x, dy = a0[i].y - at[i].y;
      part += w * 2.0 * (dx * a[i].x + dy * a[i].y);
      b[i] = make_double2(2.0 * q[l] * dx * inv_norm, 2.0 * q[l] * dy * inv_norm);
    }
  const double s = sum_y(part, sh);
  if (l <= lmax && threadIdx.y == 0) dq[l] = (float)(s * inv_norm);
}

// per-l contributions to the MLP gradient, row l of mpart; one CTA per l, thread i =
// unit i (rows of V2's gradient written by consecutive threads)
__global__ void __launch_bounds__(NN_MAXHM)
    k_nn_mlp_bwd(const float *feat, const float *par, long oV1, long oV2, long oV3, int Hm,
                 int lmax, int bf16, const float *m1, const float *m2, const float *q,
                 const float *dq, long nmlp, float *mpart) {
  __shared__ float d2[NN_MAXHM];
  const int l = blockIdx.x, i = threadIdx.x;
  float *g = mpart + (long)l * nmlp;
  // local offsets inside the MLP block: V1, c1, V2, c2, V3, c3
  const long lV1 = 0, lc1 = lV1 + (long)Hm * NN_FEAT, lV2 = lc1 + Hm,
             lc2 = lV2 + (long)Hm * Hm, lV3 = lc2 + Hm, lc3 = lV3 + Hm;
  const float qq = q[l];
  const float dz = dq[l] * qq * (1.f - qq);  // through the sigmoid
  if (i < Hm) {
    const float a2 = m2[(long)l * Hm + i];
    if (i == 0) g[lc3] = dz;
    g[lV3 + i] = dz * a2;
    d2[i] = a2 > 0.f ? dz * wround(par[oV3 + i], bf16) : 0.f;
    g[lc2 + i] = d2[i];
  }
  __syncthreads();
  if (i >= Hm) return;
  const float a1 = m1[(long)l * Hm + i];
  float d1 = 0.f;
  for (int o = 0; o < Hm; ++o) {
    g[lV2 + (long)o * Hm + i] = d2[o] * a1;
    d1 = fmaf(wround(par[oV2 + (long)o * Hm + i], bf16), d2[o], d1);
  }
  const float dd = a1 > 0.f ? d1 : 0.f;
  g[lc1 + i] = dd;
  for (int f = 0; f < NN_FEAT; ++f) g[lV1 + (long)i * NN_FEAT + f] = dd * feat[NN_FEAT * l + f];
}

// column sums: 32 columns x 32 threads, each with every 32nd row, then in order
__global__ void __launch_bounds__(1024)
    k_nn_rows_sum(const float *__restrict__ mpart, int rows, long ncol, float *__restrict__ out) {
  __shared__ float sh[32][33];
  const long c = blockIdx.x * 32L + threadIdx.x;
  float s = 0.f;
  if (c < ncol)
    for (int r = threadIdx.y; r < rows; r += 32) s += mpart[(long)r * ncol + c];
  sh[threadIdx.y][threadIdx.x] = s;
  __syncthreads();
  if (threadIdx.y != 0 || c >= ncol) return;
  for (int y = 1; y < 32; ++y) s += sh[y][threadIdx.x];
  out[c] = s;
}

// gradient of L w.r.t. the last conv output r: sig_d * Omega * (Y b)
__global__ void k_nn_gmap(const double *gmap, double scale, long npix, float *g3) {
  for (long p = (long)blockIdx.x * blockDim.x + threadIdx.x; p < npix;
       p += (long)gridDim.x * blockDim.x)
    g3[p] = (float)(scale * gmap[p]);
}

__global__ void k_nn_adam(float *par, const float *grad, float *m, float *v, long n,
                          float lr, float b1, float b2, float eps, float c1, float c2) {
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long)gridDim.x * blockDim.x) {
    const float g = grad[i];
    const float mi = b1 * m[i] + (1.f - b1) * g;
    const float vi = b2 * v[i] + (1.f - b2) * g * g;
    m[i] = mi;
    v[i] = vi;
    par[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// ---------------------------------------------------------------- host
static void free_net_buffers(Net *N) {
  if (!N) return;
  void *bufs[] = {N->par, N->grad, N->am, N->av, N->quads, N->tiles, N->in, N->h1, N->h2, N->r,
                  N->g1, N->g2, N->g3, N->t0, N->dmask, N->gmap, N->a, N->ad, N->a0,
                  N->b, N->feat, N->m1, N->m2, N->q, N->dq, N->mpart, N->wpart, N->red};
  for (void *b : bufs)
    if (b) cudaFree(b);
}

static wf_status net_alloc(Net &N) {
  Plan &P = *N.P;
  const long np = P.npix;
  std::vector<int2> quads(np / 4);
  std::vector<int4> tiles;
  auto ring = [&](long start, int n) {
    for (int j = 0; j < n / 4; ++j) quads[start / 4 + j] = make_int2((int)(start / 4), n / 4);
    for (int j = 0; j < n / 4; j += NN_TQ) tiles.push_back(make_int4((int)(start / 4), n / 4, j, 0));
  };
  for (const RingPair &p : P.pairs_h) {
    ring(p.ofsN, p.nphi);
    if (p.ringS >= 0) ring(p.ofsS, p.nphi);
  }
  N.ntiles = (int)tiles.size();
  WF_CUDA(cudaMalloc(&N.quads, sizeof(int2) * quads.size()));
  WF_CUDA(cudaMemcpy(N.quads, quads.data(), sizeof(int2) * quads.size(), cudaMemcpyHostToDevice));
  WF_CUDA(cudaMalloc(&N.tiles, sizeof(int4) * tiles.size()));
  WF_CUDA(cudaMemcpy(N.tiles, tiles.data(), sizeof(int4) * tiles.size(), cudaMemcpyHostToDevice));
  const int H = N.H, K = N.K, Hm = N.Hm;
  long o = 0;
  N.oW1 = o; o += (long)H * 3 * K; N.ob1 = o; o += H;
  N.oW2 = o; o += (long)H * H * K; N.ob2 = o; o += H;
  N.oW3 = o; o += (long)H * K;     N.ob3 = o; o += 1;
  N.nconv = o;
  N.oV1 = o; o += (long)Hm * NN_FEAT; N.oc1 = o; o += Hm;
  N.oV2 = o; o += (long)Hm * Hm;      N.oc2 = o; o += Hm;
  N.oV3 = o; o += Hm;                 N.oc3 = o; o += 1;
  N.npar = o;
  N.nmlp = N.npar - N.nconv;
  WF_CUDA(cudaMalloc(&N.par, sizeof(float) * N.npar));
  WF_CUDA(cudaMalloc(&N.grad, sizeof(float) * N.npar));
  WF_CUDA(cudaMalloc(&N.am, sizeof(float) * N.npar));
  WF_CUDA(cudaMalloc(&N.av, sizeof(float) * N.npar));
  WF_CUDA(cudaMemset(N.par, 0, sizeof(float) * N.npar));
  WF_CUDA(cudaMemset(N.am, 0, sizeof(float) * N.npar));
  WF_CUDA(cudaMemset(N.av, 0, sizeof(float) * N.npar));
  WF_CUDA(cudaMalloc(&N.in, sizeof(float) * 3 * np));
  WF_CUDA(cudaMalloc(&N.h1, sizeof(float) * H * np));
  WF_CUDA(cudaMalloc(&N.h2, sizeof(float) * H * np));
  WF_CUDA(cudaMalloc(&N.r, sizeof(float) * np));
  WF_CUDA(cudaMalloc(&N.g1, sizeof(float) * H * np));
  WF_CUDA(cudaMalloc(&N.g2, sizeof(float) * H * np));
  WF_CUDA(cudaMalloc(&N.g3, sizeof(float) * np));
  WF_CUDA(cudaMalloc(&N.t0, sizeof(double) * np));
  WF_CUDA(cudaMalloc(&N.dmask, sizeof(double) * np));
  WF_CUDA(cudaMalloc(&N.gmap, sizeof(double) * np));
  WF_CUDA(cudaMalloc(&N.a, sizeof(double2) * P.nalm));
  WF_CUDA(cudaMalloc(&N.ad, sizeof(double2) * P.nalm));
  WF_CUDA(cudaMalloc(&N.a0, sizeof(double2) * P.nalm));
  WF_CUDA(cudaMalloc(&N.b, sizeof(double2) * P.nalm));
  WF_CUDA(cudaMalloc(&N.feat, sizeof(float) * NN_FEAT * (P.lmax + 1)));
  WF_CUDA(cudaMalloc(&N.m1, sizeof(float) * Hm * (P.lmax + 1)));
  WF_CUDA(cudaMalloc(&N.m2, sizeof(float) * Hm * (P.lmax + 1)));
  WF_CUDA(cudaMalloc(&N.q, sizeof(float) * (P.lmax + 1)));
  WF_CUDA(cudaMalloc(&N.dq, sizeof(float) * (P.lmax + 1)));
  WF_CUDA(cudaMalloc(&N.mpart, sizeof(float) * N.nmlp * (P.lmax + 1)));
  const long wout = std::max((long)H * (H + 1), (long)H * 4) * K;
  WF_CUDA(cudaMalloc(&N.wpart, sizeof(float) * wout * NN_PARTS));
  WF_CUDA(cudaMalloc(&N.red, sizeof(double) * 4 * 304 + sizeof(double) * 2 * (P.lmax + 1)));
  return uploads_done();
}

// the kernels' width is a template parameter: f.template operator()<K>()
template <typename Fn>
static void with_width(int K, Fn &&f) {
  switch (K) {
    case 1: f.template operator()<1>(); break;
    case 3: f.template operator()<3>(); break;
    case 5: f.template operator()<5>(); break;
    case 7: f.template operator()<7>(); break;
    case 9: f.template operator()<9>(); break;
    case 11: f.template operator()<11>(); break;
    case 13: f.template operator()<13>(); break;
    default: f.template operator()<15>(); break;
  }
}

// 8 output channels per thread; a single one where the layer has only one
struct ConvLaunch {
  const Net &N;
  const float *in;
  int cin;
  const float *W, *bias;
  int cout, relu;
  const float *act;
  float *out;
  bool bwd;
  template <int K>
  void operator()() {
    const long nq = N.P->npix / 4;
    const unsigned gx = (unsigned)((nq + NN_THREADS - 1) / NN_THREADS);
    const int co = cout == 1 ? 1 : 8;
    const dim3 grid(gx, (cout + co - 1) / co);
    const size_t sm = sizeof(float) * cin * K * co;
    cudaStream_t s = N.P->stream;
    if (bwd && co == 8)
      k_nn_conv<K, 8, true><<<grid, NN_THREADS, sm, s>>>(N.quads, nq, in, cin, W, bias, cout, relu, N.bf16, act, out);
    else if (bwd)
      k_nn_conv<K, 1, true><<<grid, NN_THREADS, sm, s>>>(N.quads, nq, in, cin, W, bias, cout, relu, N.bf16, act, out);
    else if (co == 8)
      k_nn_conv<K, 8, false><<<grid, NN_THREADS, sm, s>>>(N.quads, nq, in, cin, W, bias, cout, relu, N.bf16, act, out);
    else
      k_nn_conv<K, 1, false><<<grid, NN_THREADS, sm, s>>>(N.quads, nq, in, cin, W, bias, cout, relu, N.bf16, act, out);
  }
};

static size_t wgrad_smem(int cout, int cin, int K) {
  const int D = (K / 2 + 3) / 4;
  return std::max(sizeof(float4) * (cout * (NN_TQ + 1) + (size_t)cin * (NN_TQ + 2 * D + 1)),
                  sizeof(float) * (K + 1) * NN_THREADS);
}

struct WgradLaunch {
  const Net &N;
  const float *gout;
  int cout;
  const float *in;
  int cin;
  float *gW, *gb;
  cudaError_t err = cudaSuccess;
  template <int K>
  void operator()() {
    int lcin = 0, lcout = 0;
    while ((1 << lcin) < cin) ++lcin;
    while ((1 << lcout) < cout) ++lcout;
    const int pairs2 = 1 << (lcin + lcout);
    const int parts = std::min(N.ntiles, NN_PARTS);
    const size_t sm = wgrad_smem(cout, cin, K);
    err = cudaFuncSetAttribute(k_nn_conv_wgrad<K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               100 * 1024);
    if (err != cudaSuccess) return;
    const dim3 grid(parts, (pairs2 + NN_THREADS - 1) / NN_THREADS);
    cudaStream_t s = N.P->stream;
    k_nn_conv_wgrad<K><<<grid, NN_THREADS, sm, s>>>(N.tiles, N.ntiles, N.P->npix / 4, gout, cout,
                                                    in, cin, lcin, pairs2, N.wpart);
    k_nn_wgrad_reduce<<<(cout * cin * K + cout + 31) / 32, NN_THREADS, 0, s>>>(
        N.wpart, parts, cout, cin, K, gW, gb);
  }
};

// forward pass for data d: t0, a, q, a0 in the net's buffers
static wf_status net_forward(Net &N, const double *d) {
  Plan &P = *N.P;
  const long np = P.npix;
  cudaStream_t s = P.stream;
  k_nn_stats<<<304, NN_THREADS, 0, s>>>(d, P.nvar, np, N.red, N.gmap);
  WF_CUDA(cudaGetLastError());
  std::vector<double> h(4 * 304);
  WF_CUDA(cudaMemcpyAsync(h.data(), N.red, sizeof(double) * h.size(), cudaMemcpyDeviceToHost, s));
  WF_CUDA(cudaStreamSynchronize(s));
  double a = 0, b = 0, c = 0, n = 0;
  for (int i = 0; i < 304; ++i) {
    a += h[4 * i];
    b += h[4 * i + 1];
    c += h[4 * i + 2];
    n += h[4 * i + 3];
  }
  N.sig_d = n > 0 && a > 0 ? sqrt(a / n) : 1.0;
  N.mu_log = n > 0 ? b / n : 0.0;
  const double var = n > 0 ? c / n - N.mu_log * N.mu_log : 1.0;
  N.sd_log = var > 1e-24 ? sqrt(var) : 1.0;
  k_nn_inputs<<<304, NN_THREADS, 0, s>>>(d, P.nvar, N.gmap, np, 1.0 / N.sig_d, N.mu_log,
                                         1.0 / N.sd_log, N.in, N.dmask);
  const int H = N.H, K = N.K;
  auto conv = [&](const float *in, int cin, long oW, long ob, int cout, int relu, float *out) {
    with_width(K, ConvLaunch{N, in, cin, N.par + oW, N.par + ob, cout, relu, nullptr, out, false});
  };
  conv(N.in, 3, N.oW1, N.ob1, H, 1, N.h1);
  conv(N.h1, H, N.oW2, N.ob2, H, 1, N.h2);
  conv(N.h2, H, N.oW3, N.ob3, 1, 0, N.r);
  k_nn_make_t0<<<304, NN_THREADS, 0, s>>>(N.dmask, N.r, N.sig_d, np, N.t0);
  WF_CUDA(cudaGetLastError());
  WF_TRY(map2alm_f32(P, N.t0, reinterpret_cast<double *>(N.a)));
  WF_TRY(map2alm_f32(P, N.dmask, reinterpret_cast<double *>(N.ad)));
  const int lb = (P.lmax + 32) / 32;
  k_nn_features<<<lb, dim3(32, 32), 0, s>>>(N.ad, P.cl_d, P.lmax, P.alpha * P.omega, N.feat);
  k_nn_mlp_fwd<<<P.lmax + 1, NN_MAXHM, 0, s>>>(N.feat, N.par, N.oV1, N.oc1, N.oV2, N.oc2, N.oV3, N.oc3,
                                  N.Hm, P.lmax, N.bf16, N.m1, N.m2, N.q);
  k_nn_gain<<<P.lmax + 1, 128, 0, s>>>(N.a, N.q, P.lmax, N.a0);
  WF_CUDA(cudaGetLastError());
  P.nlaunch += 11;
  return WF_OK;
}

static wf_status net_loss_grad(Net &N, const double *d, const double2 *at, double *loss) {
  Plan &P = *N.P;
  const long np = P.npix;
  cudaStream_t s = P.stream;
  WF_TRY(net_forward(N, d));
  double *part = N.red + 4 * 304;
  k_nn_loss<<<P.lmax + 1, 128, 0, s>>>(N.a0, at, P.lmax, part);
  WF_CUDA(cudaGetLastError());
  std::vector<double> h(2 * (P.lmax + 1));
  WF_CUDA(cudaMemcpyAsync(h.data(), part, sizeof(double) * h.size(), cudaMemcpyDeviceToHost, s));
  WF_CUDA(cudaStreamSynchronize(s));
  double e = 0, nn = 0;
  for (int m = 0; m <= P.lmax; ++m) {
    e += h[2 * m];
    nn += h[2 * m + 1];
  }
  const double inv = nn > 0 ? 1.0 / nn : 0.0;
  if (loss) *loss = e * inv;
  // harmonic MLP
  k_nn_dq<<<(P.lmax + 32) / 32, dim3(32, 32), 0, s>>>(N.a0, at, N.a, N.q, P.lmax, inv, N.dq, N.b);
  k_nn_mlp_bwd<<<P.lmax + 1, NN_MAXHM, 0, s>>>(N.feat, N.par, N.oV1, N.oV2, N.oV3, N.Hm, P.lmax, N.bf16,
                                  N.m1, N.m2, N.q, N.dq, N.nmlp, N.mpart);
  k_nn_rows_sum<<<(unsigned)((N.nmlp + 31) / 32), dim3(32, 32), 0, s>>>(N.mpart, P.lmax + 1, N.nmlp,
                                                                 N.grad + N.nconv);
  WF_CUDA(cudaGetLastError());
  // back through a = Omega Y^T t0: dL/dt0 = Omega Y b, dL/dr = sig_d dL/dt0
  WF_TRY(alm2map_f32(P, reinterpret_cast<const double *>(N.b), N.gmap));
  k_nn_gmap<<<304, NN_THREADS, 0, s>>>(N.gmap, N.sig_d * P.omega, np, N.g3);
  const int H = N.H, K = N.K;
  auto wgrad = [&](const float *gout, int cout, const float *in, int cin, long oW, long ob) {
    WgradLaunch w{N, gout, cout, in, cin, N.grad + oW, N.grad + ob};
    with_width(K, w);
    return w.err;
  };
  auto back = [&](const float *gout, int cout, long oW, int cin, const float *act, float *gin) {
    with_width(K, ConvLaunch{N, gout, cout, N.par + oW, nullptr, cin, 0, act, gin, true});
  };
  // layer 3 (H -> 1, no ReLU)
  WF_CUDA(wgrad(N.g3, 1, N.h2, H, N.oW3, N.ob3));
  back(N.g3, 1, N.oW3, H, N.h2, N.g2);
  // layer 2 (H -> H, ReLU)
  WF_CUDA(wgrad(N.g2, H, N.h1, H, N.oW2, N.ob2));
  back(N.g2, H, N.oW2, H, N.h1, N.g1);
  // layer 1 (3 -> H, ReLU; no gradient into the inputs)
  WF_CUDA(wgrad(N.g1, H, N.in, 3, N.oW1, N.ob1));
  WF_CUDA(cudaGetLastError());
  P.nlaunch += 14;
  N.have_grad = 1;
  return WF_OK;
}

}  // namespace wf

struct wf_net_s : public wf::Net {};

using namespace wf;

extern "C" {

wf_status wf_net_create(wf_net_t *out, wf_plan_t plan, int channels, int kernel, int hidden,
                        int bf16) {
  if (!out || !plan) {
    set_error("wf_net_create: NULL argument");
    return WF_ERR_ARG;
  }
  *out = nullptr;
  if (channels < 1 || channels > NN_MAXC || kernel < 1 || kernel > NN_MAXK ||
      (kernel & 1) == 0 || hidden < 1 || hidden > NN_MAXHM) {
    set_error("wf_net_create: channels in [1, 32], odd kernel in [1, 15], hidden in [1, 64]");
    return WF_ERR_ARG;
  }
  if (!plan->has_noise) {
    set_error("wf_net_create: the plan needs noise and mask");
    return WF_ERR_STATE;
  }
  wf_net_s *N = new wf_net_s();
  N->P = plan;
  N->H = channels;
  N->K = kernel;
  N->Hm = hidden;
  N->bf16 = bf16 ? 1 : 0;
  wf_status s = net_alloc(*N);
  if (s != WF_OK) {
    free_net_buffers(N);
    delete N;
    return s;
  }
  *out = N;
  return WF_OK;
}

long wf_net_num_params(wf_net_t net) { return net ? net->npar : 0; }

wf_status wf_net_set_params(wf_net_t net, const float *host, long n) {
  if (!net || !host || n != net->npar) {
    set_error("wf_net_set_params: wrong size or NULL");
    return WF_ERR_ARG;
  }
  WF_CUDA(cudaMemcpy(net->par, host, sizeof(float) * n, cudaMemcpyHostToDevice));
  WF_CUDA(cudaMemset(net->am, 0, sizeof(float) * n));
  WF_CUDA(cudaMemset(net->av, 0, sizeof(float) * n));
  net->step = 0;
  return uploads_done();
}

wf_status wf_net_get_params(wf_net_t net, float *host, long n) {
  if (!net || !host || n != net->npar) {
    set_error("wf_net_get_params: wrong size or NULL");
    return WF_ERR_ARG;
  }
  WF_CUDA(cudaMemcpy(host, net->par, sizeof(float) * n, cudaMemcpyDeviceToHost));
  return WF_OK;
}

wf_status wf_net_forward(wf_net_t net, const double *d_dev, double *t0_dev,
                         double *alm0_dev) {
  if (!net || !d_dev) {
    set_error("wf_net_forward: NULL argument");
    return WF_ERR_ARG;
  }
  Plan &P = *net->P;
  WF_TRY(net_forward(*net, d_dev));
  if (t0_dev)
    WF_CUDA(cudaMemcpyAsync(t0_dev, net->t0, sizeof(double) * P.npix,
                            cudaMemcpyDeviceToDevice, P.stream));
  if (alm0_dev)
    WF_CUDA(cudaMemcpyAsync(alm0_dev, net->a0, sizeof(double2) * P.nalm,
                            cudaMemcpyDeviceToDevice, P.stream));
  WF_CUDA(cudaStreamSynchronize(P.stream));
  return WF_OK;
}

wf_status wf_net_loss_grad(wf_net_t net, const double *d_dev, const double *alm_target_dev,
                           double *loss, float *grad_host) {
  if (!net || !d_dev || !alm_target_dev) {
    set_error("wf_net_loss_grad: NULL argument");
    return WF_ERR_ARG;
  }
  WF_TRY(net_loss_grad(*net, d_dev, reinterpret_cast<const double2 *>(alm_target_dev), loss));
  if (grad_host)
    WF_CUDA(cudaMemcpyAsync(grad_host, net->grad, sizeof(float) * net->npar,
                            cudaMemcpyDeviceToHost, net->P->stream));
  WF_CUDA(cudaStreamSynchronize(net->P->stream));
  return WF_OK;
}

wf_status wf_net_adam_step(wf_net_t net, float lr, float beta1, float beta2, float eps) {
  if (!net || !net->have_grad) {
    set_error("wf_net_adam_step: no gradient (call wf_net_loss_grad first)");
    return WF_ERR_STATE;
  }
  net->step += 1;
  const float c1 = 1.f - powf(beta1, (float)net->step);
  const float c2 = 1.f - powf(beta2, (float)net->step);
  k_nn_adam<<<64, 256, 0, net->P->stream>>>(net->par, net->grad, net->am, net->av, net->npar,
                                            lr, beta1, beta2, eps, c1, c2);
  WF_CUDA(cudaGetLastError());
  net->P->nlaunch += 1;
  WF_CUDA(cudaStreamSynchronize(net->P->stream));
  return WF_OK;
}

void wf_net_destroy(wf_net_t net) {
  if (!net) return;
  free_net_buffers(net);
  delete net;
}

}  // extern "C"
