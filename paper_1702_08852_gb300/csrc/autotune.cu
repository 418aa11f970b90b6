// autotune.cu -- pick the launch variant (ring pairs per thread) of each
// Legendre kernel for a geometry by timing them once at full band.
//
// The synthesis' best number of ring pairs per thread depends on the number of
// pairs and the band limit: more give more independent recurrences and share the
// loads of the coefficients, fewer fill the chip on small maps.  The analysis has
// one kernel; its time is reported in every slot that its earlier variants had.
// Results are cached per (nside, lmax) for the process.
#include <string.h>

#include <map>
#include <mutex>
#include <utility>

#include "wf_internal.cuh"

namespace wf {

namespace {
struct Choice {
  int syn[2];
  float syn_ms[2][6], ana_ms[2][15];  // the timings the choice was made from
};
std::mutex g_tune_mu;
std::map<std::pair<int, int>, Choice> g_tune_cache;
}  // namespace

template <typename T2>
static wf_status time_synth(Plan &P, T2 *xs, T2 *F, cudaEvent_t e0, cudaEvent_t e1,
                            float *ms) {
  WF_TRY(launch_legendre_synth<T2>(P, xs, F, nullptr, P.lmax));  // warm
  WF_CUDA(cudaEventRecord(e0, P.stream));
  for (int r = 0; r < 2; ++r) WF_TRY(launch_legendre_synth<T2>(P, xs, F, nullptr, P.lmax));
  WF_CUDA(cudaEventRecord(e1, P.stream));
  WF_CUDA(cudaEventSynchronize(e1));
  WF_CUDA(cudaEventElapsedTime(ms, e0, e1));
  return WF_OK;
}

template <typename T2>
static wf_status time_anal(Plan &P, T2 *G, cudaEvent_t e0, cudaEvent_t e1, float *ms) {
  WF_TRY(launch_legendre_anal<T2>(P, G, P.xtmp, nullptr, ANA_PLAIN, P.lmax));
  WF_CUDA(cudaEventRecord(e0, P.stream));
  for (int r = 0; r < 2; ++r)
    WF_TRY(launch_legendre_anal<T2>(P, G, P.xtmp, nullptr, ANA_PLAIN, P.lmax));
  WF_CUDA(cudaEventRecord(e1, P.stream));
  WF_CUDA(cudaEventSynchronize(e1));
  WF_CUDA(cudaEventElapsedTime(ms, e0, e1));
  return WF_OK;
}

wf_status autotune(Plan &P) {
  const std::pair<int, int> key(P.nside, P.lmax);
  {
    std::lock_guard<std::mutex> lock(g_tune_mu);
    auto it = g_tune_cache.find(key);
    if (it != g_tune_cache.end()) {
      for (int k = 0; k < 2; ++k) P.syn_np[k] = it->second.syn[k];
      memcpy(P.tune_syn_ms, it->second.syn_ms, sizeof(P.tune_syn_ms));
      memcpy(P.tune_ana_ms, it->second.ana_ms, sizeof(P.tune_ana_ms));
      return WF_OK;
    }
  }
  // inputs are zeros: the kernels' work does not depend on the values
  WF_CUDA(cudaMemsetAsync(P.xs32, 0, sizeof(float2) * P.nalm, P.stream));
  WF_CUDA(cudaMemsetAsync(P.xtmp, 0, sizeof(double2) * P.nalm, P.stream));
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  WF_CUDA(cudaEventCreate(&e0));
  WF_CUDA(cudaEventCreate(&e1));
  static const int syn_cand[6] = {1, 2, 4, 2, 4, 2};  // slots 3 .. 5 (FP32): packed
  wf_status st = WF_OK;
  for (int k = 0; k < 2 && st == WF_OK; ++k) {  // 0 = FP64, 1 = FP32
    if (k ? !P.pt32.ck : !P.pt64.ck) continue;  // no transform of this type can run
    float best = 1e30f;
    int pick = P.syn_np[k];
    for (int ci = 0; ci < 3 && st == WF_OK; ++ci) {
      P.syn_np[k] = syn_cand[ci];
      float ms = 0.f;
      st = k ? time_synth<float2>(P, P.xs32, P.F32, e0, e1, &ms)
             : time_synth<double2>(P, P.xtmp, P.F64, e0, e1, &ms);
      if (st != WF_OK) break;
      for (int c = ci; c < (k ? 6 : 3); ++c)
        if (syn_cand[c] == syn_cand[ci]) P.tune_syn_ms[k][c] = ms;
      if (ms < best) {
        best = ms;
        pick = syn_cand[ci];
      }
    }
    P.syn_np[k] = pick;
    if (st != WF_OK) break;
    float ms = 0.f;
    st = k ? time_anal<float2>(P, P.G32, e0, e1, &ms)
           : time_anal<double2>(P, P.G64, e0, e1, &ms);
    for (int c = 0; st == WF_OK && c < (k ? 15 : 3); ++c) P.tune_ana_ms[k][c] = ms;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (st != WF_OK) return st;
  std::lock_guard<std::mutex> lock(g_tune_mu);
  Choice c;
  for (int k = 0; k < 2; ++k) c.syn[k] = P.syn_np[k];
  memcpy(c.syn_ms, P.tune_syn_ms, sizeof(c.syn_ms));
  memcpy(c.ana_ms, P.tune_ana_ms, sizeof(c.ana_ms));
  g_tune_cache[key] = c;
  return WF_OK;
}

}  // namespace wf
