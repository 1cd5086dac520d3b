// sdv_sampler.cuh - the sampler's model and round state, shared by its translation units.
#pragma once

#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "sdv_device.cuh"
#include "sdv_host.h"

namespace sdv {

struct Sched {
  int K;
  float churn, beta_min, beta_max, t_floor, delta;
  __device__ __forceinline__ float tfwd(int k) const {
    return fmaxf((float)(K - k) / (float)K, t_floor);  // 1 - t_k, t_k = k / K
  }
  __device__ __forceinline__ float beta(float tf) const { return beta_min + (beta_max - beta_min) * tf; }
  __device__ __forceinline__ float abar(float tf) const {
    return expf(-(beta_min * tf + 0.5f * (beta_max - beta_min) * tf * tf));
  }
  __device__ __forceinline__ float sigma(int k) const {
    return sqrtf(delta) * churn * sqrtf(beta(tfwd(k)));
  }
};

struct Gmm {
  const float* means;  // [C, d]
  const float* log_w;  // [C]
  int C;
  float comp_var;
};

__host__ __device__ __forceinline__ uint64_t splitmix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Seed of round r: the (r+1)-th SplitMix64 output of a stream started at `seed`.
__host__ __device__ __forceinline__ uint64_t round_seed(uint64_t seed, int r) {
  return splitmix64(seed + (uint64_t)(r + 1) * 0x9E3779B97F4A7C15ull);
}

// Device-resident state of the round loop: the seed of the current round, the rounds
// run, and the chains k_round_update found still active in the current round.
struct SamplerCtl {
  uint64_t seed_r;
  int32_t r;
  uint32_t active;
  uint32_t done;  // k_round_update CTAs that finished this round
};

constexpr int kRoundThreads = 256;
constexpr int64_t kRoundMaxD = 4 * 4 * kRoundThreads;   // NG <= 4
// How k_rounds takes a row: a chain's threads, groups of four per thread, and the CTAs of an SM
// by threads and registers (long windows of short rows can ask for more shared memory than
// leaves place for as many).
struct RoundShape {
  int threads, groups, per_sm;
};
inline RoundShape round_shape(int64_t d, bool vec) {
  if (d > 1024) return {kRoundThreads, vec && d <= 2048 ? 2 : 4, 1};
  const int t = vec ? (d <= 128 ? 32 : (d <= 256 ? 64 : (d <= 512 ? 128 : kRoundThreads))) : (d <= 256 ? 64 : kRoundThreads);
  return {t, 1, (vec ? 768 : 1024) / t};
}

struct RoundsArgs {
  float* y;       // [B, d] states
  float* sc;      // [B, d] cached scores
  float* rows;    // [B, L, dp] drafted states, dp = d rounded up to whole groups
  int32_t *kk, *gam, *rounds, *tsum;
  // nullable: y, kk, rounds and tsum once more (sdv_sampler_run's outputs)
  float* y_out;
  int32_t *k_out, *rounds_out, *tsum_out;
  SamplerCtl* ctl;
  int B, L;
  int64_t d;
  Sched S;
  Gmm G;
  uint64_t seed;
  int mode, max_rounds, frozen;
  int one_round;  // host-driven: one round, and the round counter advances in any case
  int fresh;      // a whole run: the chains start here, at step 0 from Y_0
  int pre;        // draft rows whose noise is drawn ahead into shared memory
};

// Runs RoundsArgs' rounds (sdv_rounds.cuh), for mixtures of up to MAXC components; vec: rows
// of whole groups of four, 16-byte aligned.
template <int MAXC>
int launch_rounds_c(const RoundsArgs& A, bool vec, cudaStream_t s);

inline int launch_check() {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_last_cuda_error((int)e);
    return SDV_ECUDA;
  }
  return SDV_OK;
}

}  // namespace sdv
