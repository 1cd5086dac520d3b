// sdv_sampler.cu - end-to-end speculative diffusion sampler on an analytic Gaussian-
// mixture target (sm_103a): the target-mean kernel, the Free / Frozen drafter, the
// round update, the plain Euler-Maruyama chain, and the native round loop.
//
// Model (Eq. forward-process / backward-process / target-distribution):
//   VP schedule beta(t) = beta_min + (beta_max - beta_min) t, f = -beta/2, g = sqrt(beta),
//   abar_t = exp(-int_0^t beta); q_t = sum_c w_c N(sqrt(abar) mu_c, v I), v = abar s^2 + 1 - abar;
//   score s_t(x) = sum_c r_c (sqrt(abar) mu_c - x) / v, r = softmax(log w_c - |x - sqrt(abar) mu_c|^2/(2v));
//   m^q_k(y) = y + delta [beta/2 y + (1 + eps^2)/2 beta s(y)] at forward time 1 - t_k (floored),
//   sigma_k = sqrt(delta) eps sqrt(beta).
// Drafter (Eq. frozen-draft-drift and the Free drafter of Sec. "Self-Speculative Drafter"):
//   m^p = yhat + delta [beta/2 yhat + (1 + eps^2)/2 beta s_cache], yhat' = m^p + sigma G.
// Round (Alg. full-block-verification): draft gamma_k = min(L, K - k) steps, target means
// at yhat_k .. yhat_{k+gamma_k}, sdv_verify_ex, then advance k by tau (no bonus step when
// the window reaches K), keep the score at the next round's start state.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "sdv_device.cuh"
#include "sdv_host.h"
#include "sdv_sampler.cuh"

namespace sdv {

constexpr int kGmmThreads = 256;              // 8 warps, one state row per warp at a time
constexpr int kGmmWarps = kGmmThreads / 32;
constexpr size_t kGmmSmemCap = 96 * 1024;     // stage the means in shared memory up to this size

// One state row of a target call: state z at generative step k; outputs mq / score
// (either may be null; z may alias mq: each lane reads a group of four elements
// before it writes it, and no other lane touches that group).  add_sigma != 0 adds
// sigma * G to mq (Philox stream noise_stream of chain `chain`, sub-counter k; one
// Philox block per group of four).
struct GmmRow {
  const float* z;
  float* mq;
  float* score;
  int k;
  uint32_t chain;
  float add_sigma;
};

// m^q and the score for nr <= RB rows by one warp: every mean group read from `mu`
// (shared or global memory) serves all nr rows.  nr is warp-uniform.
// VEC: d % 4 == 0 and 16-byte aligned rows (float4 accesses); MAXC >= C components.
template <int MAXC, bool VEC, int RB>
__device__ __forceinline__ void gmm_rows_warp(const GmmRow (&R)[RB], int nr, int64_t d, const Sched& S,
                                              const Gmm& G, const float* mu, uint64_t noise_seed,
                                              uint32_t noise_stream) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int C = G.C;
  float sab[RB], v[RB], inv_v[RB], be[RB];
#pragma unroll
  for (int q = 0; q < RB; ++q) {
    const float tf = S.tfwd(R[q].k);
    const float ab = S.abar(tf);
    sab[q] = sqrtf(ab);
    v[q] = ab * G.comp_var + 1.0f - ab;
    inv_v[q] = 1.0f / v[q];
    be[q] = S.beta(tf);
  }
  const float cst = 0.5f * (1.0f + S.churn * S.churn);
  const int64_t ng = (d + 3) / 4;
  // groups in flight per lane: RB rows, times the unrolled sweeps
  constexpr int kU = RB >= 3 ? 1 : (RB == 2 ? 2 : 4);
  auto load_group = [&](const float* p, int64_t gi, float (&f)[4]) {
    if (VEC) {
      const float4 t = *reinterpret_cast<const float4*>(p + 4 * gi);
      f[0] = t.x; f[1] = t.y; f[2] = t.z; f[3] = t.w;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) f[e] = (4 * gi + e < d) ? p[4 * gi + e] : 0.f;
    }
  };
  // pass 1: squared distances to the scaled centres sqrt(abar) mu_c
  float acc[RB][MAXC];
#pragma unroll
  for (int q = 0; q < RB; ++q)
#pragma unroll
    for (int c = 0; c < MAXC; ++c) acc[q][c] = 0.f;
#pragma unroll kU
  for (int64_t gi = lane; gi < ng; gi += 32) {
    float zf[RB][4];
#pragma unroll
    for (int q = 0; q < RB; ++q) {
      if (q < nr) load_group(R[q].z, gi, zf[q]);
    }
#pragma unroll
    for (int c = 0; c < MAXC; ++c) {
      if (c < C) {
        float mf[4];
        load_group(mu + (int64_t)c * d, gi, mf);
#pragma unroll
        for (int q = 0; q < RB; ++q) {
          if (q < nr) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              // the tail check is only needed without VEC (d % 4 == 0 otherwise)
              const float df = (VEC || 4 * gi + e < d) ? zf[q][e] - sab[q] * mf[e] : 0.f;
              acc[q][c] = fmaf(df, df, acc[q][c]);
            }
          }
        }
      }
    }
  }
  // responsibilities r_c = softmax(log w_c - d2_c / (2 v)), identical in every lane;
  // acc becomes r, w_sc folds the softmax normaliser and sqrt(abar)
  float w_sc[RB];
#pragma unroll
  for (int q = 0; q < RB; ++q) {
    float mx = -INFINITY;
#pragma unroll
    for (int c = 0; c < MAXC; ++c) {
      float a = acc[q][c];
      if (c < C) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(FULL, a, o);
      }
      acc[q][c] = (c < C) ? __ldg(G.log_w + c) - 0.5f * a * inv_v[q] : -INFINITY;
      mx = fmaxf(mx, acc[q][c]);
    }
    float den = 0.f;
#pragma unroll
    for (int c = 0; c < MAXC; ++c) {
      acc[q][c] = (c < C) ? expf(acc[q][c] - mx) : 0.f;
      den += acc[q][c];
    }
    w_sc[q] = sab[q] / den;
  }
  // pass 2: score and target mean
#pragma unroll kU
  for (int64_t gi = lane; gi < ng; gi += 32) {
    float zf[RB][4], wsum[RB][4];
#pragma unroll
    for (int q = 0; q < RB; ++q) {
      if (q < nr) load_group(R[q].z, gi, zf[q]);
#pragma unroll
      for (int e = 0; e < 4; ++e) wsum[q][e] = 0.f;
    }
#pragma unroll
    for (int c = 0; c < MAXC; ++c) {
      if (c < C) {
        float mf[4];
        load_group(mu + (int64_t)c * d, gi, mf);
#pragma unroll
        for (int q = 0; q < RB; ++q)
#pragma unroll
          for (int e = 0; e < 4; ++e) wsum[q][e] = fmaf(acc[q][c], mf[e], wsum[q][e]);
      }
    }
#pragma unroll
    for (int q = 0; q < RB; ++q) {
      if (q < nr) {
        float G4[4] = {0.f, 0.f, 0.f, 0.f};
        if (R[q].add_sigma != 0.f) {
          const float4 n4 = normals4(noise_seed, R[q].chain, (uint32_t)gi, noise_stream, (uint32_t)R[q].k);
          G4[0] = n4.x; G4[1] = n4.y; G4[2] = n4.z; G4[3] = n4.w;
        }
        float sc[4], m[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          sc[e] = (w_sc[q] * wsum[q][e] - zf[q][e]) * inv_v[q];
          m[e] = zf[q][e] + S.delta * (0.5f * be[q] * zf[q][e] + cst * be[q] * sc[e]) + R[q].add_sigma * G4[e];
        }
        float* score = R[q].score;
        float* mq = R[q].mq;
        if (VEC) {
          if (score) *reinterpret_cast<float4*>(score + 4 * gi) = make_float4(sc[0], sc[1], sc[2], sc[3]);
          if (mq) *reinterpret_cast<float4*>(mq + 4 * gi) = make_float4(m[0], m[1], m[2], m[3]);
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            if (4 * gi + e < d) {
              if (score) score[4 * gi + e] = sc[e];
              if (mq) mq[4 * gi + e] = m[e];
            }
          }
        }
      }
    }
  }
}

// Stage the means in dynamic shared memory (when the launch gave it room); returns the
// pointer the warps read from.
__device__ __forceinline__ const float* stage_means(const Gmm& G, int64_t d, bool use_smem) {
  extern __shared__ float mu_s[];
  if (!use_smem) return G.means;
  const int64_t n = (int64_t)G.C * d;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) mu_s[i] = __ldg(G.means + i);
  __syncthreads();
  return mu_s;
}

// Target means and scores for rows of a [n, d] array at steps k[row]; one warp per row;
// rows whose window mask (if given) is 0 are skipped.
template <int MAXC, bool VEC>
__global__ void __launch_bounds__(kGmmThreads)
k_gmm_rows(const float* __restrict__ states, const int32_t* __restrict__ k, const int32_t* __restrict__ mask,
           int n, int64_t d, Sched S, Gmm G, bool use_smem, float* mq, float* score) {
  const float* mu = stage_means(G, d, use_smem);
  const int warp = threadIdx.x >> 5;
  for (int row = blockIdx.x * kGmmWarps + warp; row < n; row += gridDim.x * kGmmWarps) {
    if (mask && mask[row] == 0) continue;
    const int64_t o = (int64_t)row * d;
    const GmmRow R[1] = {{states + o, mq ? mq + o : nullptr, score ? score + o : nullptr, k[row], 0u, 0.f}};
    gmm_rows_warp<MAXC, VEC, 1>(R, 1, d, S, G, mu, 0, 0);
  }
}

// Rows of a round's parallel target call per warp.
template <int MAXC> struct RoundRows { static constexpr int value = MAXC <= 8 ? 3 : 1; };

// Parallel target call of a round.  Row (b, j), j = 0 .. gamma_b, is state y[b]
// (j = 0) or x_draft[b, j-1] at step k[b] + j; its mean goes to mu_target[b, j]
// (j < gamma_b) or mu_bonus[b] (j = gamma_b, with sigma_bonus[b] = sigma_{k+gamma}),
// its score to sc_all[b, j].  The B (L+1) row slots are dealt to warps RB at a time
// (slots past gamma_b are skipped), grid-stride over persistent CTAs.
template <int MAXC, bool VEC>
__global__ void __launch_bounds__(kGmmThreads, 2)
k_round_target(const float* __restrict__ y, const float* __restrict__ x_draft,
               const int32_t* __restrict__ kk, const int32_t* __restrict__ gam, int B, int L, int64_t d,
               Sched S, Gmm G, bool use_smem, float* mu_target, float* mu_bonus, float* sigma_bonus,
               float* sc_all) {
  constexpr int RB = RoundRows<MAXC>::value;
  const float* mu = stage_means(G, d, use_smem);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t slots = (int64_t)B * (L + 1);
  for (int64_t r0 = ((int64_t)blockIdx.x * kGmmWarps + warp) * RB; r0 < slots;
       r0 += (int64_t)gridDim.x * kGmmWarps * RB) {
    GmmRow R[RB];
    int nr = 0;
#pragma unroll
    for (int q = 0; q < RB; ++q) {
      R[q] = GmmRow{nullptr, nullptr, nullptr, 0, 0u, 0.f};
      const int64_t slot = r0 + q;
      if (slot >= slots) continue;
      const int b = (int)(slot / (L + 1));
      const int j = (int)(slot - (int64_t)b * (L + 1));
      const int g = gam[b];
      if (j > g || g == 0) continue;
      const int kb = kk[b];
      GmmRow row;
      row.z = (j == 0) ? y + (int64_t)b * d : x_draft + ((int64_t)b * L + j - 1) * d;
      row.mq = (j < g) ? mu_target + ((int64_t)b * L + j) * d : mu_bonus + (int64_t)b * d;
      row.score = sc_all + ((int64_t)b * (L + 1) + j) * d;
      row.k = kb + j;
      row.chain = 0u;
      row.add_sigma = 0.f;
      if (j == g && lane == 0) sigma_bonus[b] = S.sigma(kb + g);
      // compact the live rows to the front (q is a compile-time index after unrolling)
#pragma unroll
      for (int t = 0; t < RB; ++t)
        if (t == nr) R[t] = row;
      ++nr;
    }
    if (nr > 0) gmm_rows_warp<MAXC, VEC, RB>(R, nr, d, S, G, mu, 0, 0);
  }
}

// Row slots of a round's target call, shared by the target-call kernels: slot
// (b, j), j = 0 .. L, is live when j <= gamma_b (and gamma_b > 0).
struct RoundRow {
  const float* z;
  float* mq;
  float* score;
  int k;
  bool live;
};

__device__ __forceinline__ RoundRow round_row(int64_t slot, int64_t slots, const float* y, const float* x_draft,
                                              const int32_t* kk, const int32_t* gam, int L, int64_t d,
                                              const Sched& S, float* mu_target, float* mu_bonus,
                                              float* sigma_bonus, float* sc_all, bool write_sigma) {
  RoundRow R{nullptr, nullptr, nullptr, 0, false};
  if (slot >= slots) return R;
  const int b = (int)(slot / (L + 1));
  const int j = (int)(slot - (int64_t)b * (L + 1));
  const int g = gam[b];
  if (j > g || g == 0) return R;
  const int kb = kk[b];
  R.z = (j == 0) ? y + (int64_t)b * d : x_draft + ((int64_t)b * L + j - 1) * d;
  R.mq = (j < g) ? mu_target + ((int64_t)b * L + j) * d : mu_bonus + (int64_t)b * d;
  R.score = sc_all + ((int64_t)b * (L + 1) + j) * d;
  R.k = kb + j;
  R.live = true;
  if (j == g && write_sigma) sigma_bonus[b] = S.sigma(kb + g);
  return R;
}

// Resident CTAs per SM k_round_target_reg is built for (its register budget).
constexpr int round_reg_blocks(int maxc) { return maxc <= 8 ? 3 : 2; }

// Parallel target call of a round for rows of up to 4 kGmmThreads elements
// (d % 4 == 0, 16-byte aligned rows): each thread owns one group of four elements
// and holds that group of every mean in registers for the whole kernel; a CTA takes
// RB = 32 / MAXC row slots at a time (grid-stride), keeps each row's group in
// registers across both passes, and reduces the RB x MAXC squared distances with one
// warp reduce-scatter (value v ends in lane v) and one pass over the warps.  Warp 0
// resolves the next batch's rows and their schedule constants into shared memory
// (three buffers: the batch being written, the one being finished and the next),
// and every thread loads the next batch's states while this batch finishes.
template <int MAXC>
__global__ void __launch_bounds__(kGmmThreads, round_reg_blocks(MAXC))
k_round_target_reg(const float* __restrict__ y, const float* __restrict__ x_draft,
                   const int32_t* __restrict__ kk, const int32_t* __restrict__ gam, int B, int L, int64_t d,
                   Sched S, Gmm G, float* mu_target, float* mu_bonus, float* sigma_bonus, float* sc_all) {
  constexpr int RB = 32 / MAXC;
  constexpr int NV = RB * MAXC;  // 32
  struct RowC {
    const float* z;
    float* mq;
    float* score;
    float sab, inv_v, be;
    int live;
  };
  __shared__ float red[kGmmWarps][NV];
  __shared__ float resp[RB][MAXC];
  __shared__ float wsc[RB];
  __shared__ RowC rows_s[3][RB];
  const unsigned FULL = 0xffffffffu;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int C = G.C;
  const int64_t ng = d / 4;
  const bool own = tid < ng;  // this thread's group exists
  const int64_t slots = (int64_t)B * (L + 1);
  const int64_t stride = (int64_t)gridDim.x * RB;
  // warp 0, lane r < RB: row slot s + r -> rows_s[buf][r]
  auto resolve = [&](int64_t s, int buf) {
    if (warp == 0 && lane < RB) {
      const RoundRow R = round_row(s + lane, slots, y, x_draft, kk, gam, L, d, S, mu_target, mu_bonus,
                                   sigma_bonus, sc_all, true);
      RowC rc;
      rc.z = R.z; rc.mq = R.mq; rc.score = R.score; rc.live = R.live ? 1 : 0;
      const float tf = S.tfwd(R.k);
      const float ab = S.abar(tf);
      rc.sab = sqrtf(ab);
      rc.inv_v = 1.0f / (ab * G.comp_var + 1.0f - ab);
      rc.be = S.beta(tf);
      rows_s[buf][lane] = rc;
    }
  };
  float4 m4[MAXC];
#pragma unroll
  for (int c = 0; c < MAXC; ++c)
    m4[c] = (own && c < C) ? __ldg(reinterpret_cast<const float4*>(G.means + (int64_t)c * d) + tid)
                           : make_float4(0.f, 0.f, 0.f, 0.f);
  const float cst = 0.5f * (1.0f + S.churn * S.churn);
  int64_t s0 = (int64_t)blockIdx.x * RB;
  int cur = 0;
  resolve(s0, cur);
  __syncthreads();
  float4 z[RB];
#pragma unroll
  for (int r = 0; r < RB; ++r)
    z[r] = (rows_s[cur][r].live && own) ? *(reinterpret_cast<const float4*>(rows_s[cur][r].z) + tid)
                                        : make_float4(0.f, 0.f, 0.f, 0.f);
  for (; s0 < slots; s0 += stride) {
    const int nxt = cur == 2 ? 0 : cur + 1;
    const RowC* R = rows_s[cur];
    // pass 1: this thread's share of |z_r - sqrt(abar_r) mu_c|^2
    float v[NV];
#pragma unroll
    for (int r = 0; r < RB; ++r) {
      const float zf[4] = {z[r].x, z[r].y, z[r].z, z[r].w};
#pragma unroll
      for (int c = 0; c < MAXC; ++c) {
        const float mf[4] = {m4[c].x, m4[c].y, m4[c].z, m4[c].w};
        float a = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float df = zf[e] - R[r].sab * mf[e];
          a = fmaf(df, df, a);
        }
        v[r * MAXC + c] = a;
      }
    }
    // warp reduce-scatter: after the halving steps lane l holds the warp sum of value l
#pragma unroll
    for (int h = NV / 2; h >= 1; h >>= 1) {
      const bool up = (lane & h) != 0;
#pragma unroll
      for (int k = 0; k < h; ++k) {
        const float send = up ? v[k] : v[k + h];
        const float keep = up ? v[k + h] : v[k];
        v[k] = keep + __shfl_xor_sync(FULL, send, h);
      }
    }
    red[warp][lane] = v[0];
    resolve(s0 + stride, nxt);  // last read two batches ago, before this batch's first barrier
    __syncthreads();
    // the next batch's states, in flight while this batch finishes
    float4 zn[RB];
#pragma unroll
    for (int r = 0; r < RB; ++r)
      zn[r] = (rows_s[nxt][r].live && own) ? *(reinterpret_cast<const float4*>(rows_s[nxt][r].z) + tid)
                                           : make_float4(0.f, 0.f, 0.f, 0.f);
    if (warp == 0) {
      // responsibilities r_c = softmax(log w_c - d2_c / (2 v)) over each row's MAXC lanes
      float t = 0.f;
#pragma unroll
      for (int w = 0; w < kGmmWarps; ++w) t += red[w][lane];
      const int r = lane / MAXC, c = lane - r * MAXC;
      float ivr = R[0].inv_v, sabr = R[0].sab;
#pragma unroll
      for (int q = 1; q < RB; ++q) {
        ivr = (r == q) ? R[q].inv_v : ivr;
        sabr = (r == q) ? R[q].sab : sabr;
      }
      const float a = (c < C) ? __ldg(G.log_w + c) - 0.5f * t * ivr : -INFINITY;
      float mx = a;
#pragma unroll
      for (int o = MAXC / 2; o >= 1; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(FULL, mx, o));
      const float ex = (c < C) ? expf(a - mx) : 0.f;
      float den = ex;
#pragma unroll
      for (int o = MAXC / 2; o >= 1; o >>= 1) den += __shfl_xor_sync(FULL, den, o);
      resp[r][c] = ex;
      if (c == 0) wsc[r] = sabr / den;  // folds the softmax normaliser and sqrt(abar)
    }
    __syncthreads();
    // pass 2: score and target mean of this thread's group
#pragma unroll
    for (int r = 0; r < RB; ++r) {
      if (R[r].live && own) {
        float ws[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int c = 0; c < MAXC; ++c) {
          const float rc = resp[r][c];
          ws[0] = fmaf(rc, m4[c].x, ws[0]);
          ws[1] = fmaf(rc, m4[c].y, ws[1]);
          ws[2] = fmaf(rc, m4[c].z, ws[2]);
          ws[3] = fmaf(rc, m4[c].w, ws[3]);
        }
        const float w = wsc[r];
        const float zf[4] = {z[r].x, z[r].y, z[r].z, z[r].w};
        float sc[4], m[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          sc[e] = (w * ws[e] - zf[e]) * R[r].inv_v;
          m[e] = zf[e] + S.delta * (0.5f * R[r].be * zf[e] + cst * R[r].be * sc[e]);
        }
        reinterpret_cast<float4*>(R[r].score)[tid] = make_float4(sc[0], sc[1], sc[2], sc[3]);
        reinterpret_cast<float4*>(R[r].mq)[tid] = make_float4(m[0], m[1], m[2], m[3]);
      }
    }
#pragma unroll
    for (int r = 0; r < RB; ++r) z[r] = zn[r];
    cur = nxt;
  }
}

// Free / Frozen drafter: gamma_b elementwise steps from y[b] with the cached score.
// One thread per group of four elements; VEC: d % 4 == 0 and 16-byte aligned rows
// (float4 loads and stores).  The Philox draws do not depend on the state, so the
// unrolled step loop overlaps the next step's draws with this step's stores.
template <bool VEC>
__global__ void __launch_bounds__(256)
k_draft(const float* __restrict__ y, const float* __restrict__ s_cache, const int32_t* __restrict__ kk,
        const int32_t* __restrict__ gam, int B, int L, int64_t d, Sched S, uint64_t seed_v,
        const uint64_t* __restrict__ seed_dev, float* __restrict__ x_draft, float* __restrict__ mu_draft,
        float* __restrict__ sigma) {
  const int64_t ng = (d + 3) / 4;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)B * ng) return;
  const int b = (int)(t / ng);
  const int64_t gi = t - (int64_t)b * ng;
  const int g = gam[b];
  if (g == 0) return;
  const uint64_t seed = seed_dev ? *seed_dev : seed_v;
  const int k = kk[b];
  const float cst = 0.5f * (1.0f + S.churn * S.churn);
  const int64_t i0 = 4 * gi;
  float cur[4], sc[4];
  if (VEC) {
    const float4 a = *reinterpret_cast<const float4*>(y + (int64_t)b * d + i0);
    const float4 c = *reinterpret_cast<const float4*>(s_cache + (int64_t)b * d + i0);
    cur[0] = a.x; cur[1] = a.y; cur[2] = a.z; cur[3] = a.w;
    sc[0] = c.x; sc[1] = c.y; sc[2] = c.z; sc[3] = c.w;
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      cur[q] = (i0 + q < d) ? y[(int64_t)b * d + i0 + q] : 0.f;
      sc[q] = (i0 + q < d) ? s_cache[(int64_t)b * d + i0 + q] : 0.f;
    }
  }
#pragma unroll 4
  for (int step = 1; step <= g; ++step) {
    const int kc = k + step - 1;
    const float be = S.beta(S.tfwd(kc));
    const float sg = S.sigma(kc);
    const float4 n4 = normals4(seed, (uint32_t)b, (uint32_t)gi, kStreamDraft, (uint32_t)(step - 1));
    const float nz[4] = {n4.x, n4.y, n4.z, n4.w};
    const int64_t row = ((int64_t)b * L + step - 1) * d;
    float m[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      m[q] = cur[q] + S.delta * (0.5f * be * cur[q] + cst * be * sc[q]);
      cur[q] = m[q] + sg * nz[q];
    }
    if (VEC) {
      *reinterpret_cast<float4*>(mu_draft + row + i0) = make_float4(m[0], m[1], m[2], m[3]);
      *reinterpret_cast<float4*>(x_draft + row + i0) = make_float4(cur[0], cur[1], cur[2], cur[3]);
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (i0 + q < d) {
          mu_draft[row + i0 + q] = m[q];
          x_draft[row + i0 + q] = cur[q];
        }
      }
    }
    if (gi == 0) sigma[(int64_t)b * L + step - 1] = sg;
  }
}

// End of a round (the k_round_update CTA holding the round's last ticket): advance the
// round counter and seed, reset the round's counters, and (inside the round graph)
// keep the loop going while a chain is active and fewer than max_rounds rounds ran.
__device__ __forceinline__ void close_round(SamplerCtl* ctl, uint64_t seed, int max_rounds, int in_loop,
                                            cudaGraphConditionalHandle h) {
  const int r = ctl->r + 1;
  ctl->r = r;
  ctl->seed_r = round_seed(seed, r);
  const bool more = ctl->active != 0u && r < max_rounds;
  ctl->active = 0u;
  ctl->done = 0u;
  if (in_loop) cudaGraphSetConditional(h, more ? 1u : 0u);
}

// Round bookkeeping, one warp per chain and kUpdateChains chains per CTA: the emitted
// state, the score cache, k, the next window length and the statistics; each CTA adds
// its chains that remain active with one atomic, and the CTA holding the round's last
// ticket closes the round (close_round).  (One CTA per chain made 1024 same-address
// atomics per round, and that serialisation cost most of the kernel's time.)
// VEC: d % 4 == 0 (workspace rows are then 16-byte aligned).
constexpr int kUpdateChains = 8;

template <bool VEC>
__global__ void __launch_bounds__(32 * kUpdateChains)
k_round_update(const int32_t* __restrict__ acc, const float* __restrict__ y_out,
               const float* __restrict__ x_draft, const float* __restrict__ sc_all, int B, int L, int64_t d,
               int K, float* y, float* s_cache, int32_t* kk, int32_t* gam, int32_t* rounds,
               int32_t* tau_sum, SamplerCtl* ctl, uint64_t seed, int max_rounds, int in_loop,
               cudaGraphConditionalHandle h) {
  __shared__ unsigned int act_s[kUpdateChains];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b = blockIdx.x * kUpdateChains + w;
  unsigned int act = 0u;
  if (b < B) {
    const int g = gam[b];
    const int k = kk[b];
    __syncwarp();  // every lane has read k and gamma before lane 0 updates them
    const int tau = acc[b] + 1;
    if (g > 0) {
      const bool end = (tau == g + 1) && (k + g >= K);  // no bonus step past the end of sampling
      const float* ysrc = end ? x_draft + ((int64_t)b * L + g - 1) * d : y_out + (int64_t)b * d;
      const float* ssrc = sc_all + ((int64_t)b * (L + 1) + min(tau, g)) * d;
      if (VEC) {
        const float4* ys4 = reinterpret_cast<const float4*>(ysrc);
        const float4* ss4 = reinterpret_cast<const float4*>(ssrc);
        float4* yd4 = reinterpret_cast<float4*>(y + (int64_t)b * d);
        float4* sd4 = reinterpret_cast<float4*>(s_cache + (int64_t)b * d);
        for (int64_t i = lane; i < d / 4; i += 32) {
          yd4[i] = ys4[i];
          sd4[i] = ss4[i];
        }
      } else {
        for (int64_t i = lane; i < d; i += 32) {
          y[(int64_t)b * d + i] = ysrc[i];
          s_cache[(int64_t)b * d + i] = ssrc[i];
        }
      }
      if (lane == 0) {
        const int kn = min(k + tau, K);
        kk[b] = kn;
        const int gn = kn < K ? min(L, K - kn) : 0;
        gam[b] = gn;
        rounds[b] += 1;
        tau_sum[b] += tau;
        act = gn > 0 ? 1u : 0u;
      }
    }
  }
  if (lane == 0) act_s[w] = act;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned int n = 0u;
#pragma unroll
    for (int i = 0; i < kUpdateChains; ++i) n += act_s[i];
    if (n) atomicAdd(&ctl->active, n);
    if (ticket_acq_rel(&ctl->done) == gridDim.x - 1) close_round(ctl, seed, max_rounds, in_loop, h);
  }
}

__global__ void __launch_bounds__(256)
k_sampler_init(int B, int L, int64_t d, int K, uint64_t seed, float* y, int32_t* kk, int32_t* gam,
               int32_t* rounds, int32_t* tau_sum, SamplerCtl* ctl) {
  const int64_t ng = (d + 3) / 4;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)B * ng) return;
  const int b = (int)(t / ng);
  const int64_t gi = t - (int64_t)b * ng;
  const float4 n4 = normals4(seed, (uint32_t)b, (uint32_t)gi, kStreamInit, 0u);
  const float nz[4] = {n4.x, n4.y, n4.z, n4.w};
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (4 * gi + q < d) y[(int64_t)b * d + 4 * gi + q] = nz[q];
  if (t == 0 && ctl != nullptr) {
    ctl->seed_r = round_seed(seed, 0);
    ctl->r = 0;
    ctl->active = 0u;
    ctl->done = 0u;
  }
  if (gi == 0 && kk != nullptr) {
    kk[b] = 0;
    gam[b] = min(L, K);
    rounds[b] = 0;
    tau_sum[b] = 0;
  }
}

// The plain Euler-Maruyama chain for rows of up to 128 NG elements: a team of T warps runs
// a chain's K steps with the state in registers (every warp holds all of it, lane l the
// groups l, l + 32, ...) and the means in shared memory, one copy per CTA.  Per step the
// warps share out the components (squared distances, pass 1), then the groups (score,
// mean and noise, pass 2), and exchange the logits and the new state through shared
// memory.  The sums have the order of gmm_rows_warp, so that both give the same states.
// It is bound by instruction issue: 77 % of the issue slots, 567 instructions of a warp per 32
// groups of four and step, waiting warps mostly ready but not selected.  One launch per step
// with the state in HBM took 13.1 us a step at B = 1024, d = 1024, C = 8, this kernel 4.7 us
// with T = 4 (T = 2: 5.5, too few warps; 8: 5.4, seven eighths of the softmax repeated and two
// waves of CTAs).
constexpr int kEmMaxTeams = 7;   // chains per CTA: 152 SMs x 7 hold 1024 chains in one wave

template <int MAXC, int NG, int T>
__global__ void __launch_bounds__(32 * T * (T == 8 ? 1 : kEmMaxTeams))
k_em_chain(float* __restrict__ y, int B, int64_t d, Sched S, Gmm G, uint64_t seed) {
  extern __shared__ float4 em_s[];
  constexpr int GP = 32 * NG;            // groups of a padded row
  constexpr int CPW = MAXC / T;          // components per warp
  const unsigned FULL = 0xffffffffu;
  const int C = G.C;
  const int dn = (int)d;
  const int teams = blockDim.x / (32 * T);
  const int team = threadIdx.x / (32 * T), lane = threadIdx.x & 31;
  const int tw = (threadIdx.x >> 5) - team * T;
  float4* mu_s = em_s;                                           // [C][GP], zero past d
  float4* z_s = em_s + (size_t)C * GP + (size_t)team * GP;       // [teams][GP]
  float* lg_s = reinterpret_cast<float*>(em_s + (size_t)(C + teams) * GP) + team * MAXC;
  for (int i = threadIdx.x; i < C * GP * 4; i += blockDim.x) {
    const int c = i / (GP * 4), e = i - c * (GP * 4);
    reinterpret_cast<float*>(mu_s)[i] = e < dn ? __ldg(G.means + (int64_t)c * d + e) : 0.f;
  }
  __syncthreads();
  const int b = blockIdx.x * teams + team;
  if (b >= B) return;                    // the whole team
  auto team_sync = [&] { asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "n"(32 * T) : "memory"); };
  // elements past d hold 0 (they then add exactly nothing to the distances)
  auto masked = [&](float4 v, int gi) {
    const int e = dn - 4 * gi;
    if (e < 4) {
      if (e < 1) v.x = 0.f;
      if (e < 2) v.y = 0.f;
      if (e < 3) v.z = 0.f;
      v.w = 0.f;
    }
    return v;
  };
  float4 z[NG];
  for (int i = tw; i < NG; i += T) {
    const int gi = lane + 32 * i;
    z_s[gi] = masked(normals4(seed, (uint32_t)b, (uint32_t)gi, kStreamInit, 0u), gi);
  }
  team_sync();
#pragma unroll
  for (int i = 0; i < NG; ++i) z[i] = z_s[lane + 32 * i];
  const float cst = 0.5f * (1.0f + S.churn * S.churn);
  float sab_l = 0.f, iv_l = 0.f, be_l = 0.f, sg_l = 0.f;   // schedule of step (k & ~31) + lane
  for (int k = 0; k < S.K; ++k) {
    if ((k & 31) == 0) {
      const int kl = min(k + lane, S.K);
      const float tf = S.tfwd(kl);
      const float ab = S.abar(tf);
      sab_l = sqrtf(ab);
      const float v = ab * G.comp_var + 1.0f - ab;
      iv_l = 1.0f / v;
      be_l = S.beta(tf);
      sg_l = S.sigma(kl);
    }
    const float sab = __shfl_sync(FULL, sab_l, k & 31), inv_v = __shfl_sync(FULL, iv_l, k & 31);
    const float be = __shfl_sync(FULL, be_l, k & 31), sg = __shfl_sync(FULL, sg_l, k & 31);
    // pass 1: squared distances to this warp's scaled centres
    float acc[CPW];
#pragma unroll
    for (int m = 0; m < CPW; ++m) acc[m] = 0.f;
#pragma unroll
    for (int i = 0; i < NG; ++i) {
      const float zf[4] = {z[i].x, z[i].y, z[i].z, z[i].w};
#pragma unroll
      for (int m = 0; m < CPW; ++m) {
        const int c = tw * CPW + m;
        if (c < C) {
          const float4 t = mu_s[c * GP + lane + 32 * i];
          const float mf[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float df = zf[e] - sab * mf[e];
            acc[m] = fmaf(df, df, acc[m]);
          }
        }
      }
    }
#pragma unroll
    for (int m = 0; m < CPW; ++m) {
      const int c = tw * CPW + m;
      float a = acc[m];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(FULL, a, o);
      if (lane == 0) lg_s[c] = (c < C) ? __ldg(G.log_w + c) - 0.5f * a * inv_v : -INFINITY;
    }
    team_sync();
    float r[MAXC];
    float mx = -INFINITY;
#pragma unroll
    for (int c = 0; c < MAXC; ++c) {
      r[c] = lg_s[c];
      mx = fmaxf(mx, r[c]);
    }
    float den = 0.f;
#pragma unroll
    for (int c = 0; c < MAXC; ++c) {
      r[c] = (c < C) ? expf(r[c] - mx) : 0.f;
      den += r[c];
    }
    const float w_sc = sab / den;
    // pass 2: this warp's groups of the new state
#pragma unroll
    for (int ii = 0; ii < (NG + T - 1) / T; ++ii) {
      const int i = tw + ii * T;
      if (NG % T != 0 && i >= NG) break;   // warp-uniform
      const int gi = lane + 32 * i;
      const float4 n4 = normals4(seed, (uint32_t)b, (uint32_t)gi, kStreamEM, (uint32_t)k);
      const float G4[4] = {n4.x, n4.y, n4.z, n4.w};
      const float4 zo = z_s[gi];
      const float zf[4] = {zo.x, zo.y, zo.z, zo.w};
      float wsum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int c = 0; c < MAXC; ++c) {
        if (c < C) {
          const float4 t = mu_s[c * GP + gi];
          const float mf[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) wsum[e] = fmaf(r[c], mf[e], wsum[e]);
        }
      }
      float m[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float sc = (w_sc * wsum[e] - zf[e]) * inv_v;
        m[e] = zf[e] + S.delta * (0.5f * be * zf[e] + cst * be * sc) + sg * G4[e];
      }
      z_s[gi] = masked(make_float4(m[0], m[1], m[2], m[3]), gi);
    }
    team_sync();
#pragma unroll
    for (int i = 0; i < NG; ++i) z[i] = z_s[lane + 32 * i];
  }
  float* row = y + (int64_t)b * d;
  const float* zr = reinterpret_cast<const float*>(z_s);
  for (int e = tw * 32 + lane; e < dn; e += 32 * T) row[e] = zr[e];
}

// The plain Euler-Maruyama chain for longer rows: one warp runs a chain's K steps, the
// state in its row of y (each group read and written by one lane only).
template <int MAXC, bool VEC>
__global__ void __launch_bounds__(kGmmThreads)
k_em_rows(float* y, int B, int64_t d, Sched S, Gmm G, bool use_smem, uint64_t seed) {
  const float* mu = stage_means(G, d, use_smem);
  const int b = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (b >= B) return;
  float* row = y + (int64_t)b * d;
  for (int k = 0; k < S.K; ++k) {
    const GmmRow R[1] = {{row, row, nullptr, k, (uint32_t)b, S.sigma(k)}};
    gmm_rows_warp<MAXC, VEC, 1>(R, 1, d, S, G, mu, seed, kStreamEM);
  }
}

// Launch geometry of the one-warp-per-row kernels: dynamic shared memory for the means
// when they fit, the component bound, vector accesses, and the grid for n rows.
struct GmmLaunch {
  bool smem;
  size_t smem_bytes;
  bool vec;
  int maxc;
};

// The kernels' limit of dynamic shared memory, which all host threads share: its largest value.
template <int MAXC, bool VEC>
static void gmm_set_smem() {
  cudaFuncSetAttribute(k_gmm_rows<MAXC, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGmmSmemCap);
  cudaFuncSetAttribute(k_round_target<MAXC, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGmmSmemCap);
  cudaFuncSetAttribute(k_em_rows<MAXC, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGmmSmemCap);
}

// rows_aligned: every state / output row the kernel touches starts on a 16-byte boundary
static GmmLaunch gmm_launch(int C, int64_t d, const void* means, bool rows_aligned) {
  GmmLaunch g{};
  const size_t bytes = (size_t)C * (size_t)d * sizeof(float);
  g.smem = bytes <= kGmmSmemCap;
  g.smem_bytes = g.smem ? bytes : 0;
  g.vec = (d % 4 == 0) && (reinterpret_cast<uintptr_t>(means) % 16 == 0) && rows_aligned;
  g.maxc = C <= 8 ? 8 : 16;
  if (g.smem_bytes > 48 * 1024) {
    if (g.maxc == 8) { gmm_set_smem<8, true>(); gmm_set_smem<8, false>(); }
    else { gmm_set_smem<16, true>(); gmm_set_smem<16, false>(); }
  }
  return g;
}

static unsigned rows_grid(int n) { return (unsigned)std::max(1, (n + kGmmWarps - 1) / kGmmWarps); }

// Grid of k_round_target: one warp per RB row slots, at most four CTAs per SM (each
// CTA stages the means once and strides over its share of the slots).
static unsigned round_target_grid(const GmmLaunch& gl, int B, int L) {
  const int64_t rb = gl.maxc <= 8 ? RoundRows<8>::value : RoundRows<16>::value;
  const int64_t need = ((int64_t)B * (L + 1) + kGmmWarps * rb - 1) / (kGmmWarps * rb);
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>(need, 4 * (int64_t)sm_count()));
}

// Rows of up to 4 kGmmThreads elements with 16-byte aligned rows and means take the
// register-resident k_round_target_reg (grid-stride over its resident CTAs); others
// the shared-memory k_round_target.
static bool round_target_reg(const GmmLaunch& gl, int64_t d) { return gl.vec && d <= 4 * kGmmThreads; }

static unsigned round_target_reg_grid(const GmmLaunch& gl, int B, int L) {
  const int64_t rb = 32 / (gl.maxc <= 8 ? 8 : 16);
  const int64_t need = ((int64_t)B * (L + 1) + rb - 1) / rb;
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>(need, round_reg_blocks(gl.maxc) * (int64_t)sm_count()));
}

#define SDV_GMM_DISPATCH(GL, KERNEL, GRID, STREAM, ...)                                          \
  do {                                                                                          \
    if ((GL).maxc == 8) {                                                                       \
      if ((GL).vec) KERNEL<8, true><<<GRID, kGmmThreads, (GL).smem_bytes, STREAM>>>(__VA_ARGS__);  \
      else KERNEL<8, false><<<GRID, kGmmThreads, (GL).smem_bytes, STREAM>>>(__VA_ARGS__);          \
    } else {                                                                                    \
      if ((GL).vec) KERNEL<16, true><<<GRID, kGmmThreads, (GL).smem_bytes, STREAM>>>(__VA_ARGS__); \
      else KERNEL<16, false><<<GRID, kGmmThreads, (GL).smem_bytes, STREAM>>>(__VA_ARGS__);         \
    }                                                                                           \
  } while (0)

// The plain chain of rows of up to 1024 elements: teams of T warps, chains dealt evenly to
// the SMs, at most kEmMaxTeams to a CTA.
template <int MAXC, int NG, int T>
static int launch_em_t(int B, int64_t d, const Sched& S, const Gmm& G, uint64_t seed, float* y, cudaStream_t s) {
  const int sms = sm_count();
  const int teams = T == 8 ? 1 : std::min(kEmMaxTeams, std::max(1, (B + sms - 1) / sms));
  constexpr auto bytes = [](int c, int n) { return sizeof(float4) * (size_t)(c + n) * 32 * NG + sizeof(float) * (size_t)n * MAXC; };
  const size_t smem = bytes(G.C, teams);
  if (smem > 48 * 1024) {
    // the limit is shared by all host threads: its largest value
    constexpr int kMost = (int)bytes(MAXC, T == 8 ? 1 : kEmMaxTeams);
    const cudaError_t e = cudaFuncSetAttribute(k_em_chain<MAXC, NG, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost);
    if (e != cudaSuccess) {
      set_last_cuda_error((int)e);
      cudaGetLastError();
      return SDV_ECUDA;
    }
  }
  k_em_chain<MAXC, NG, T><<<(unsigned)((B + teams - 1) / teams), 32 * T * teams, smem, s>>>(y, B, d, S, G, seed);
  return launch_check();
}

template <int MAXC>
static int launch_em(int B, int64_t d, const Sched& S, const Gmm& G, uint64_t seed, float* y, cudaStream_t s) {
  // eight warps to a chain while every chain has an SM to itself, else four
  const bool wide = B <= sm_count();
#define SDV_EM(NG)                                                    \
  return wide ? launch_em_t<MAXC, NG, 8>(B, d, S, G, seed, y, s)       \
              : launch_em_t<MAXC, NG, 4>(B, d, S, G, seed, y, s)
  if (d <= 128) { SDV_EM(1); }
  if (d <= 256) { SDV_EM(2); }
  if (d <= 512) { SDV_EM(4); }
  SDV_EM(8);
#undef SDV_EM
}

static bool valid_sched(int K, float churn, float bmin, float bmax, float tfl) {
  return K >= 1 && std::isfinite(churn) && churn > 0.f && std::isfinite(bmin) && std::isfinite(bmax) &&
         bmin > 0.f && bmax >= bmin && tfl > 0.f && tfl <= 1.f;
}

static Sched make_sched(int K, float churn, float bmin, float bmax, float tfl) {
  Sched S;
  S.K = K; S.churn = churn; S.beta_min = bmin; S.beta_max = bmax; S.t_floor = tfl;
  S.delta = 1.0f / (float)K;
  return S;
}

struct SamplerLayout {
  size_t y, s, k, g, x, mp, mq, mqb, sg, sgb, sc, acc, yo, rounds, tausum, ctl, vws, total;
};

static SamplerLayout sampler_layout(int B, int L, int64_t d) {
  SamplerLayout w{};
  auto up = [](size_t v) { return (v + 255) & ~(size_t)255; };
  const size_t Bd = (size_t)B * d * sizeof(float);
  const size_t BLd = (size_t)B * L * d * sizeof(float);
  size_t o = 0;
  w.y = o; o = up(o + Bd);
  w.s = o; o = up(o + Bd);
  w.k = o; o = up(o + (size_t)B * 4);
  w.g = o; o = up(o + (size_t)B * 4);
  w.x = o; o = up(o + BLd);
  w.mp = o; o = up(o + BLd);
  w.mq = o; o = up(o + BLd);
  w.mqb = o; o = up(o + Bd);
  w.sg = o; o = up(o + (size_t)B * L * 4);
  w.sgb = o; o = up(o + (size_t)B * 4);
  w.sc = o; o = up(o + (size_t)B * (L + 1) * d * sizeof(float));
  w.acc = o; o = up(o + (size_t)B * 4);
  w.yo = o; o = up(o + Bd);
  w.rounds = o; o = up(o + (size_t)B * 4);
  w.tausum = o; o = up(o + (size_t)B * 4);
  w.ctl = o; o = up(o + sizeof(SamplerCtl));
  w.vws = o; o = up(o + sdv_workspace_bytes(B, L, d, SDV_F32));
  w.total = o;
  return w;
}

// A sampler problem and the views of its workspace.
struct SamplerRun {
  int B, L;
  int64_t d;
  int K, mode, drafter;
  uint64_t seed;
  Sched S;
  Gmm G;
  GmmLaunch gl;
  unsigned eg;
  float *y, *sc, *xd, *mpd, *mqd, *mqb, *sg, *sgb, *scall, *yo;
  int32_t *kk, *gam, *acc, *rounds, *tsum;
  SamplerCtl* ctl;
  void* vws;
  size_t vws_bytes;
};

static void sampler_views(const SamplerLayout& w, char* ws, SamplerRun* R) {
  R->y = (float*)(ws + w.y);
  R->sc = (float*)(ws + w.s);
  R->kk = (int32_t*)(ws + w.k);
  R->gam = (int32_t*)(ws + w.g);
  R->xd = (float*)(ws + w.x);
  R->mpd = (float*)(ws + w.mp);
  R->mqd = (float*)(ws + w.mq);
  R->mqb = (float*)(ws + w.mqb);
  R->sg = (float*)(ws + w.sg);
  R->sgb = (float*)(ws + w.sgb);
  R->scall = (float*)(ws + w.sc);
  R->acc = (int32_t*)(ws + w.acc);
  R->yo = (float*)(ws + w.yo);
  R->rounds = (int32_t*)(ws + w.rounds);
  R->tsum = (int32_t*)(ws + w.tausum);
  R->ctl = (SamplerCtl*)(ws + w.ctl);
  R->vws = ws + w.vws;
  R->vws_bytes = w.total - w.vws;
}

static int sampler_setup(int B, int L, int64_t d, const float* means, const float* log_weights, int C,
                         float comp_var, int K, float churn, float beta_min, float beta_max, float t_floor,
                         uint64_t seed, int mode, int drafter, void* workspace, size_t workspace_bytes,
                         SamplerRun* R) {
  if (!means || !log_weights) return SDV_EINVAL;
  if (B < 1 || L < 1 || L > SDV_MAX_L || d < 1 || C < 1 || C > kSdvMaxComponents) return SDV_EINVAL;
  if (!(comp_var > 0.f) || !valid_sched(K, churn, beta_min, beta_max, t_floor)) return SDV_EINVAL;
  if (mode != SDV_MODE_SAMPLE && mode != SDV_MODE_BLOCK) return SDV_EINVAL;
  if (drafter != SDV_DRAFTER_FREE && drafter != SDV_DRAFTER_FROZEN) return SDV_EINVAL;
  const SamplerLayout w = sampler_layout(B, L, d);
  if (!workspace || workspace_bytes < w.total) return SDV_ENOWORKSPACE;
  if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return SDV_EALIGN;
  R->B = B; R->L = L; R->d = d; R->K = K; R->mode = mode; R->drafter = drafter; R->seed = seed;
  R->S = make_sched(K, churn, beta_min, beta_max, t_floor);
  R->G = Gmm{means, log_weights, C, comp_var};
  // workspace arrays start on 256-byte boundaries
  R->gl = gmm_launch(C, d, means, reinterpret_cast<uintptr_t>(workspace) % 16 == 0);
  R->eg = (unsigned)(((int64_t)B * ((d + 3) / 4) + 255) / 256);
  sampler_views(w, (char*)workspace, R);
  return SDV_OK;
}

// Initial states, bookkeeping and round state, and the only explicit target call: the
// score at Y_0 (step 0).
static int enqueue_begin(const SamplerRun& R, cudaStream_t s) {
  k_sampler_init<<<R.eg, 256, 0, s>>>(R.B, R.L, R.d, R.K, R.seed, R.y, R.kk, R.gam, R.rounds, R.tsum, R.ctl);
  int rc = launch_check();
  if (rc != SDV_OK) return rc;
  SDV_GMM_DISPATCH(R.gl, k_gmm_rows, rows_grid(R.B), s, R.y, R.kk, nullptr, R.B, R.d, R.S, R.G, R.gl.smem,
                   nullptr, R.sc);
  return launch_check();
}

// Rounds that sdv_sampler_run enqueues directly at most.
constexpr int kDirectRounds = 32;

// One round on stream cs (captured into the round graph's loop body when `loop`,
// whose condition the round's last update CTA then sets; launched directly
// otherwise).
static int enqueue_round(const SamplerRun& R, cudaStream_t cs, int max_rounds, bool loop,
                         cudaGraphConditionalHandle handle) {
  const int B = R.B, L = R.L;
  const int64_t d = R.d;
  const GmmLaunch& gl = R.gl;
  int rc = SDV_OK;
  if (R.drafter == SDV_DRAFTER_FROZEN) {  // a fresh score at the round's start state
    SDV_GMM_DISPATCH(gl, k_gmm_rows, rows_grid(B), cs, R.y, R.kk, R.gam, B, d, R.S, R.G, gl.smem, nullptr, R.sc);
    if ((rc = launch_check()) != SDV_OK) return rc;
  }
  if (gl.vec)
    k_draft<true><<<R.eg, 256, 0, cs>>>(R.y, R.sc, R.kk, R.gam, B, L, d, R.S, 0, &R.ctl->seed_r, R.xd, R.mpd, R.sg);
  else
    k_draft<false><<<R.eg, 256, 0, cs>>>(R.y, R.sc, R.kk, R.gam, B, L, d, R.S, 0, &R.ctl->seed_r, R.xd, R.mpd, R.sg);
  if ((rc = launch_check()) != SDV_OK) return rc;
  if (round_target_reg(gl, d)) {
    const unsigned grid = round_target_reg_grid(gl, B, L);
    if (gl.maxc == 8)
      k_round_target_reg<8><<<grid, kGmmThreads, 0, cs>>>(R.y, R.xd, R.kk, R.gam, B, L, d, R.S, R.G, R.mqd, R.mqb,
                                                         R.sgb, R.scall);
    else
      k_round_target_reg<16><<<grid, kGmmThreads, 0, cs>>>(R.y, R.xd, R.kk, R.gam, B, L, d, R.S, R.G, R.mqd, R.mqb,
                                                          R.sgb, R.scall);
  } else {
    SDV_GMM_DISPATCH(gl, k_round_target, round_target_grid(gl, B, L), cs, R.y, R.xd, R.kk, R.gam, B, L, d, R.S,
                     R.G, gl.smem, R.mqd, R.mqb, R.sgb, R.scall);
  }
  if ((rc = launch_check()) != SDV_OK) return rc;
  rc = verify_ex_impl(R.xd, R.mqd, R.mpd, R.sg, L, B, L, d, SDV_F32, 0, &R.ctl->seed_r, R.mode, R.gam, R.mqb,
                      R.sgb, SDV_RESIDUAL_DECOMPOSITION, 1.0f, R.acc, R.yo, nullptr, nullptr, nullptr, nullptr,
                      R.vws, R.vws_bytes, false, cs);
  if (rc != SDV_OK) return rc;
  if (d % 4 == 0)
    k_round_update<true><<<(B + kUpdateChains - 1) / kUpdateChains, 32 * kUpdateChains, 0, cs>>>(
        R.acc, R.yo, R.xd, R.scall, B, L, d, R.K, R.y, R.sc, R.kk, R.gam, R.rounds, R.tsum, R.ctl, R.seed,
        max_rounds, loop ? 1 : 0, handle);
  else
    k_round_update<false><<<(B + kUpdateChains - 1) / kUpdateChains, 32 * kUpdateChains, 0, cs>>>(
        R.acc, R.yo, R.xd, R.scall, B, L, d, R.K, R.y, R.sc, R.kk, R.gam, R.rounds, R.tsum, R.ctl, R.seed,
        max_rounds, loop ? 1 : 0, handle);
  return launch_check();
}

// Rounds of every chain in one launch (rows of up to kRoundMaxD elements).
static RoundsArgs rounds_args(const SamplerRun& R) {
  RoundsArgs A{};
  A.y = R.y; A.sc = R.sc; A.rows = R.xd;   // the padded rows run on into the unused draft and target arrays
  A.kk = R.kk; A.gam = R.gam; A.rounds = R.rounds; A.tsum = R.tsum; A.ctl = R.ctl;
  A.B = R.B; A.L = R.L; A.d = R.d; A.S = R.S; A.G = R.G; A.seed = R.seed;
  A.mode = R.mode; A.frozen = R.drafter == SDV_DRAFTER_FROZEN;
  return A;
}

// Whether k_rounds runs the sampler (rows of up to kRoundMaxD elements) or one kernel per phase
// of a round does.  k_rounds' time grows by whole waves of CTAs and with the threads' groups,
// filled or not; the phases' with chains and elements, from a floor of five launches a round.
//  - All chains in one wave, or means too large for the phases' shared memory: k_rounds (0.25 to
//    0.99 of the phases' time over the sizes measured; but 1.06 for 152 chains of 2052 elements,
//    L = 32, and 1.07 for 1824 of 256, L = 4).
//  - Aligned rows of up to 1024 elements, more waves: phases (d = 1024, L = 8: 456 chains, one
//    wave, 46 us a round against 61, 608 chains 88 against 74, 1024 chains 119 against 107).
//  - Other rows: up to 7 (aligned) or 5 waves of full rows, fewer where a row leaves part of the
//    groups empty, and, over 1024 elements, where the window outgrows the noise that is drawn
//    ahead.  k_rounds over phases at L = 8 by waves: aligned 1028 1.2 at 7, 2048 0.90 at 7 and
//    1.07 at 27, 2052 1.31 at 7; else 513 0.94 at 2 and 1.09 at 4, 901 0.82 at 2 and 1.01 at 8,
//    1101 1.11 at 2 and 1.72 at 7, 2001 0.91 at 2 and 1.18 at 4, 3001 0.81 at 3.  At L = 16 and
//    2 waves: 1028 1.09, 2048 0.74, 2052 1.11.
static bool rounds_fit(const SamplerRun& R) {
  if (R.d > kRoundMaxD) return false;
  const RoundShape s = round_shape(R.d, R.gl.vec);
  const int64_t slots = (int64_t)sm_count() * s.per_sm, waves = (R.B + slots - 1) / slots;
  if (waves <= 1 || !R.gl.smem) return true;
  if (R.gl.vec && R.d <= 1024) return false;
  const float full = (float)R.d / (float)(4 * s.threads * s.groups);
  const float window = R.d > 1024 ? 8.0f / (float)std::max(8, R.L) : 1.0f;
  return (float)waves <= (R.gl.vec ? 7.0f : 5.0f) * full * window;
}

static int launch_rounds(const SamplerRun& R, const RoundsArgs& A, cudaStream_t s) {
  return R.gl.maxc == 8 ? launch_rounds_c<8>(A, R.gl.vec, s) : launch_rounds_c<16>(A, R.gl.vec, s);
}

// Rounds run (host, after a synchronisation) and the chains' outputs (device copies).
static int read_results(const SamplerRun& R, float* y_out, int32_t* k_out, int32_t* chain_rounds_out,
                        int32_t* tau_sum_out, int32_t* rounds_out, cudaStream_t s) {
  int r = 0;
  if (cudaMemcpyAsync(&r, &R.ctl->r, sizeof(r), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return launch_check(), SDV_ECUDA;
  *rounds_out = r;
  // outputs that the run wrote itself stay where they are
  auto copy = [&](void* out, const void* from, size_t bytes) {
    return out == nullptr || out == from || cudaMemcpyAsync(out, from, bytes, cudaMemcpyDeviceToDevice, s) == cudaSuccess;
  };
  const size_t n = (size_t)R.B * 4;
  if (!copy(y_out, R.y, n * (size_t)R.d) || !copy(k_out, R.kk, n) || !copy(chain_rounds_out, R.rounds, n) ||
      !copy(tau_sum_out, R.tsum, n))
    return launch_check(), SDV_ECUDA;
  return SDV_OK;
}

}  // namespace sdv

using namespace sdv;

extern "C" {

int sdv_gmm_target(const float* states, const int32_t* k, int n, int64_t d, const float* means,
                   const float* log_weights, int C, float comp_var, int K, float churn,
                   float beta_min, float beta_max, float t_floor, float* mq_out, float* score_out,
                   sdv_stream_t stream) {
  if (!states || !k || !means || !log_weights || (!mq_out && !score_out)) return SDV_EINVAL;
  if (n < 0 || d < 1 || C < 1 || C > kSdvMaxComponents || !(comp_var > 0.f)) return SDV_EINVAL;
  if (!valid_sched(K, churn, beta_min, beta_max, t_floor)) return SDV_EINVAL;
  if (n == 0) return SDV_OK;
  const Sched S = make_sched(K, churn, beta_min, beta_max, t_floor);
  const Gmm G{means, log_weights, C, comp_var};
  // float4 paths need 16-byte aligned rows in every array the kernel touches
  const bool al = ((reinterpret_cast<uintptr_t>(states) | reinterpret_cast<uintptr_t>(mq_out) |
                    reinterpret_cast<uintptr_t>(score_out)) % 16) == 0;
  const GmmLaunch gl = gmm_launch(C, d, means, al);
  SDV_GMM_DISPATCH(gl, k_gmm_rows, rows_grid(n), (cudaStream_t)stream, states, k, nullptr, n, d, S, G,
                   gl.smem, mq_out, score_out);
  return launch_check();
}

int sdv_free_draft(const float* y, const float* score, const int32_t* k, const int32_t* L_eff, int B,
                   int L, int64_t d, int K, float churn, float beta_min, float beta_max,
                   float t_floor, uint64_t seed, float* x_draft, float* mu_draft, float* sigma,
                   sdv_stream_t stream) {
  if (!y || !score || !k || !L_eff || !x_draft || !mu_draft || !sigma) return SDV_EINVAL;
  if (B < 1 || L < 1 || L > SDV_MAX_L || d < 1) return SDV_EINVAL;
  if (!valid_sched(K, churn, beta_min, beta_max, t_floor)) return SDV_EINVAL;
  const Sched S = make_sched(K, churn, beta_min, beta_max, t_floor);
  const int64_t n = (int64_t)B * ((d + 3) / 4);
  const bool vec = (d % 4 == 0) && ((reinterpret_cast<uintptr_t>(y) | reinterpret_cast<uintptr_t>(score) |
                                      reinterpret_cast<uintptr_t>(x_draft) |
                                      reinterpret_cast<uintptr_t>(mu_draft)) % 16 == 0);
  const unsigned grid = (unsigned)((n + 255) / 256);
  if (vec) k_draft<true><<<grid, 256, 0, (cudaStream_t)stream>>>(y, score, k, L_eff, B, L, d, S, seed, nullptr, x_draft, mu_draft, sigma);
  else k_draft<false><<<grid, 256, 0, (cudaStream_t)stream>>>(y, score, k, L_eff, B, L, d, S, seed, nullptr, x_draft, mu_draft, sigma);
  return launch_check();
}

size_t sdv_sampler_workspace_bytes(int B, int L, int64_t d) {
  if (B < 1 || L < 1 || L > SDV_MAX_L || d < 1) return 0;
  return sampler_layout(B, L, d).total;
}

int sdv_sampler_run(int B, int L, int64_t d, const float* means, const float* log_weights, int C,
                    float comp_var, int K, float churn, float beta_min, float beta_max,
                    float t_floor, uint64_t seed, int mode, int drafter, int max_rounds,
                    float* y_out, int32_t* k_out, int32_t* chain_rounds_out,
                    int32_t* tau_sum_out, int32_t* rounds_out, void* workspace,
                    size_t workspace_bytes, sdv_stream_t stream) {
  if (!y_out || !rounds_out) return SDV_EINVAL;
  if (max_rounds < 0) return SDV_EINVAL;
  SamplerRun R;
  int rc = sampler_setup(B, L, d, means, log_weights, C, comp_var, K, churn, beta_min, beta_max, t_floor, seed,
                         mode, drafter, workspace, workspace_bytes, &R);
  if (rc != SDV_OK) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  if (max_rounds > 0 && rounds_fit(R)) {
    // one kernel from Y_0 to the outputs, which it writes itself where they are aligned; the
    // workspace gets the state too, so that sdv_sampler_round can continue the run
    RoundsArgs A = rounds_args(R);
    A.fresh = 1;
    A.max_rounds = max_rounds;
    auto at = [](const void* p, size_t a) { return reinterpret_cast<uintptr_t>(p) % a == 0; };
    if (at(y_out, R.gl.vec ? 16 : 4)) A.y_out = R.y = y_out;
    if (k_out && at(k_out, 4)) A.k_out = R.kk = k_out;
    if (chain_rounds_out && at(chain_rounds_out, 4)) A.rounds_out = R.rounds = chain_rounds_out;
    if (tau_sum_out && at(tau_sum_out, 4)) A.tsum_out = R.tsum = tau_sum_out;
    if (cudaMemsetAsync(R.ctl, 0, sizeof(SamplerCtl), s) != cudaSuccess) return launch_check(), SDV_ECUDA;
    if ((rc = launch_rounds(R, A, s)) != SDV_OK) return rc;
    return read_results(R, y_out, k_out, chain_rounds_out, tau_sum_out, rounds_out, s);
  }
  if ((rc = enqueue_begin(R, s)) != SDV_OK) return rc;

  // A run too short for any chain to finish (a round advances L + 1 steps at most) needs no
  // condition: its rounds are enqueued as they are (building the graph takes 0.1 ms, eight
  // rounds of 1024 chains 0.9 ms).
  if (max_rounds > 0 && max_rounds <= kDirectRounds && (int64_t)(max_rounds - 1) * (L + 1) < K) {
    for (int r = 0; r < max_rounds; ++r)
      if ((rc = enqueue_round(R, s, 0, false, 0)) != SDV_OK) return rc;
    return read_results(R, y_out, k_out, chain_rounds_out, tau_sum_out, rounds_out, s);
  }
  // Otherwise the round loop is one CUDA graph: a while node whose body is one round, captured
  // once; the round's seed lives in device memory (SamplerCtl) and the round's last
  // update CTA ends the loop.  One graph launch runs every round with no host round trip.
  if (max_rounds > 0) {
    cudaGraph_t graph = nullptr, body = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaStream_t cs = nullptr;
    cudaGraphConditionalHandle handle = 0;
    cudaGraphNode_t loop = nullptr;
    bool ok = cudaGraphCreate(&graph, 0) == cudaSuccess &&
              cudaGraphConditionalHandleCreate(&handle, graph, 1u, cudaGraphCondAssignDefault) == cudaSuccess;
    if (ok) {
      cudaGraphNodeParams cp{};
      cp.type = cudaGraphNodeTypeConditional;
      cp.conditional.handle = handle;
      cp.conditional.type = cudaGraphCondTypeWhile;
      cp.conditional.size = 1;
      ok = cudaGraphAddNode(&loop, graph, nullptr, nullptr, 0, &cp) == cudaSuccess;
      if (ok) body = cp.conditional.phGraph_out[0];
    }
    ok = ok && cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) == cudaSuccess &&
         cudaStreamBeginCaptureToGraph(cs, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal) ==
             cudaSuccess;
    if (ok) {
      rc = enqueue_round(R, cs, max_rounds, true, handle);
      cudaGraph_t captured = nullptr;
      const bool ended = cudaStreamEndCapture(cs, &captured) == cudaSuccess;
      ok = rc == SDV_OK && ended && cudaGraphInstantiate(&exec, graph, 0) == cudaSuccess &&
           cudaGraphLaunch(exec, s) == cudaSuccess;
    }
    if (exec) cudaGraphExecDestroy(exec);
    if (graph) cudaGraphDestroy(graph);
    if (cs) cudaStreamDestroy(cs);
    if (!ok) {
      if (rc != SDV_OK) return rc;
      return launch_check(), SDV_ECUDA;
    }
  }
  return read_results(R, y_out, k_out, chain_rounds_out, tau_sum_out, rounds_out, s);
}

int sdv_sampler_begin(int B, int L, int64_t d, const float* means, const float* log_weights, int C,
                      float comp_var, int K, float churn, float beta_min, float beta_max, float t_floor,
                      uint64_t seed, void* workspace, size_t workspace_bytes, sdv_stream_t stream) {
  SamplerRun R;
  const int rc = sampler_setup(B, L, d, means, log_weights, C, comp_var, K, churn, beta_min, beta_max, t_floor,
                               seed, SDV_MODE_BLOCK, SDV_DRAFTER_FREE, workspace, workspace_bytes, &R);
  if (rc != SDV_OK) return rc;
  return enqueue_begin(R, (cudaStream_t)stream);
}

int sdv_sampler_round(int B, int L, int64_t d, const float* means, const float* log_weights, int C,
                      float comp_var, int K, float churn, float beta_min, float beta_max, float t_floor,
                      uint64_t seed, int mode, int drafter, void* workspace, size_t workspace_bytes,
                      sdv_stream_t stream) {
  SamplerRun R;
  const int rc = sampler_setup(B, L, d, means, log_weights, C, comp_var, K, churn, beta_min, beta_max, t_floor,
                               seed, mode, drafter, workspace, workspace_bytes, &R);
  if (rc != SDV_OK) return rc;
  if (rounds_fit(R)) {
    RoundsArgs A = rounds_args(R);
    A.max_rounds = A.one_round = 1;
    return launch_rounds(R, A, (cudaStream_t)stream);
  }
  return enqueue_round(R, (cudaStream_t)stream, 0, false, 0);
}

int sdv_sampler_end(int B, int L, int64_t d, void* workspace, size_t workspace_bytes, float* y_out,
                    int32_t* k_out, int32_t* chain_rounds_out, int32_t* tau_sum_out, int32_t* rounds_out,
                    sdv_stream_t stream) {
  if (!y_out || !rounds_out) return SDV_EINVAL;
  if (B < 1 || L < 1 || L > SDV_MAX_L || d < 1) return SDV_EINVAL;
  const SamplerLayout w = sampler_layout(B, L, d);
  if (!workspace || workspace_bytes < w.total) return SDV_ENOWORKSPACE;
  if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return SDV_EALIGN;
  SamplerRun R{};
  R.B = B; R.L = L; R.d = d;
  sampler_views(w, (char*)workspace, &R);
  return read_results(R, y_out, k_out, chain_rounds_out, tau_sum_out, rounds_out, (cudaStream_t)stream);
}

int sdv_em_sample(int B, int64_t d, const float* means, const float* log_weights, int C,
                  float comp_var, int K, float churn, float beta_min, float beta_max,
                  float t_floor, uint64_t seed, float* y_out, sdv_stream_t stream) {
  if (!means || !log_weights || !y_out) return SDV_EINVAL;
  if (B < 1 || d < 1 || C < 1 || C > kSdvMaxComponents || !(comp_var > 0.f)) return SDV_EINVAL;
  if (!valid_sched(K, churn, beta_min, beta_max, t_floor)) return SDV_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  const Sched S = make_sched(K, churn, beta_min, beta_max, t_floor);
  const Gmm G{means, log_weights, C, comp_var};
  // rows of up to 1024 elements fit the registers of a team; longer ones stay in memory
  if (d <= 1024)
    return C <= 8 ? launch_em<8>(B, d, S, G, seed, y_out, s) : launch_em<16>(B, d, S, G, seed, y_out, s);
  const int64_t ng = (int64_t)B * ((d + 3) / 4);
  // the initial state only needs y; the bookkeeping arrays of the init kernel are not used
  k_sampler_init<<<(unsigned)((ng + 255) / 256), 256, 0, s>>>(B, 1, d, K, seed, y_out, nullptr, nullptr,
                                                              nullptr, nullptr, nullptr);
  int rc = launch_check();
  if (rc != SDV_OK) return rc;
  const GmmLaunch gl = gmm_launch(C, d, means, reinterpret_cast<uintptr_t>(y_out) % 16 == 0);
  SDV_GMM_DISPATCH(gl, k_em_rows, rows_grid(B), s, y_out, B, d, S, G, gl.smem, seed);
  return launch_check();
}

}  // extern "C"
