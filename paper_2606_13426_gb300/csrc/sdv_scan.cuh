// sdv_scan.cuh - one chain's acceptance scan by one warp (sm_103a): log ratios and norms
// from the tile sums, sample and block verification (Algorithms token- /
// block-verification), and the residual's 1-D draw.  Used by the verification kernels
// and by the sampler's round kernel.
#pragma once

#include "sdv_device.cuh"
#include "sdv_host.h"

namespace sdv {

// The verification seed: by value, or from device memory (sampler rounds).
__device__ __forceinline__ uint64_t seed_of(const ScanArgs& A) { return A.seed_dev ? *A.seed_dev : A.seed; }

// ---------------------------------------------------------------- chain scan (one warp)
__device__ __forceinline__ ChainState inactive_state() {
  ChainState cs;
  cs.tau = 0; cs.row = -1; cs.U = NAN; cs.la_res = 0.f; cs.sigma = NAN; cs.dnorm = NAN;
  cs.inv_norm = 0.f; cs.refl = 0.f; cs.status = 0u; cs.kind = kKindInactive;
  cs.pad[0] = cs.pad[1] = 0;
  return cs;
}

struct ScanOut {
  ChainState cs;
  UParams P;   // residual parameters of row tau - 1 (block mode, cs.kind == kKindResid)
  bool have_P;
};

__device__ __forceinline__ UParams shfl_params(const UParams& P, int src) {
  const unsigned FULL = 0xffffffffu;
  UParams R;
  R.D = __shfl_sync(FULL, P.D, src);
  R.la = __shfl_sync(FULL, P.la, src);
  R.ap = __shfl_sync(FULL, P.ap, src);
  R.am = __shfl_sync(FULL, P.am, src);
  R.lv = __shfl_sync(FULL, P.lv, src);
  R.lvn = __shfl_sync(FULL, P.lvn, src);
  R.lnd_ap = __shfl_sync(FULL, P.lnd_ap, src);
  R.g_ap = __shfl_sync(FULL, P.g_ap, src);
  R.l1mx0 = __shfl_sync(FULL, P.l1mx0, src);
  return R;
}

// The slot of a tile's partial: S1 and S2, each in an 8-byte word below the tag of the call
// that stored it (words are read and written whole, so that a tag vouches for the sum beside
// it).  Its reader frees the slot by clearing both words, the second with release: a replayed
// call, whose tag is the one it was captured with, then finds no partial of an earlier replay
// there, and whoever sees the second word clear (acquire) may store.
__device__ __forceinline__ ulonglong2 slot_read(const uint64_t* p) {
  ulonglong2 v;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ bool slot_holds(const ulonglong2& v, uint32_t tag) {
  return (uint32_t)(v.x >> 32) == tag && (uint32_t)(v.y >> 32) == tag;
}
// (One word: asking for both by one 16-byte acquire made eight pipelined latent calls take
// 185.7 us, by two acquires 193; this way 172.6.)
__device__ __forceinline__ bool slot_is_free(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p + 1) : "memory");
  return (uint32_t)(v >> 32) == 0u;
}
__device__ __forceinline__ void slot_store(uint64_t* p, uint32_t tag, float2 s) {
  const unsigned long long t = (unsigned long long)tag << 32;
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(t | __float_as_uint(s.x)),
               "l"(t | __float_as_uint(s.y)) : "memory");
}
// Frees slots t0, t0 + dt, ... below n, once a barrier has shown that they are read.
__device__ __forceinline__ void slots_free(uint64_t* p, int t0, int dt, int n) {
  for (int t = t0; t < n; t += dt) asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p + 2 * t), "l"(0ull) : "memory");
  asm volatile("fence.acq_rel.gpu;" ::: "memory");
  for (int t = t0; t < n; t += dt) asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p + 2 * t + 1), "l"(0ull) : "memory");
}

// Per-lane values of one chain's window, held by one warp: step j in lane j & 31 of
// segment j >> 5 (L <= 64).
struct ScanRegs {
  float ell[2], dn[2], S1[2], S2[2], sg[2];
  int g;         // window length gamma_k, clamped to [0, L]
  bool any_bad;  // a non-finite ratio, norm or sigma
  bool stale;    // a k_tiles partial without this call's tag (not yet visible)
};

// ell_j and |Delta_j| of one step from its sums (S1, S2) and sigma into slot q of R;
// returns whether sigma is unusable.
__device__ __forceinline__ bool scan_step(ScanRegs& R, int q, float a1, float a2, float s) {
  R.S1[q] = a1; R.S2[q] = a2; R.sg[q] = s;
  const float rs = frcp_fast(s);
  R.ell[q] = -(a1 + 0.5f * a2) * (rs * rs);
  R.dn[q] = sqrtf(a2) * rs;
  return !(s > 0.f) || !isfinite(s);
}

// Loads chain b's ell_j and |Delta_j|: from the tile partials (S1, S2 of every tile of
// the row, read through L2; or `tiles`, the chain's [L, C] in shared memory) and sigma,
// or from given arrays.  With check_tags, R.stale reports a slot that does not hold this
// call's partial.  Called by a full warp; reads only.
__device__ __forceinline__ ScanRegs scan_load(const ScanArgs& A, int b, bool check_tags = true,
                                              const float2* tiles = nullptr) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int L = A.L;
  ScanRegs R;
  // window length gamma_k, clamped to [0, L] (device data the host cannot check)
  R.g = A.L_eff ? max(0, min(A.L_eff[b], L)) : L;
  const int nseg = (L + 31) >> 5;
  bool bad = false, stale = false;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int j = lane + 32 * q;
    R.ell[q] = 0.f; R.dn[q] = 0.f; R.S1[q] = 0.f; R.S2[q] = 0.f; R.sg[q] = 1.f;
    if (q < nseg && j < R.g) {
      if (tiles || A.tpart) {
        // partials written by other CTAs: read through L2, summed over the row's tiles
        // in tile order
        float a1 = 0.f, a2 = 0.f;
        if (tiles) {
          for (int c = 0; c < A.C; ++c) {
            a1 += tiles[j * A.C + c].x;
            a2 += tiles[j * A.C + c].y;
          }
        } else {
          const uint64_t* p = A.tpart + 2 * (((int64_t)b * L + j) * A.C);
          for (int c0 = 0; c0 < A.C; c0 += 4) {   // four loads in flight
            ulonglong2 t[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) t[u] = slot_read(p + 2 * min(c0 + u, A.C - 1));
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              if (c0 + u < A.C) {
                if (check_tags && !slot_holds(t[u], A.tag)) stale = true;
                a1 += __uint_as_float((uint32_t)t[u].x);
                a2 += __uint_as_float((uint32_t)t[u].y);
              }
            }
          }
        }
        bad |= scan_step(R, q, a1, a2, A.sigma[(int64_t)b * A.sstride + j]);
      } else {
        R.ell[q] = A.ell_in[(int64_t)b * L + j];
        R.dn[q] = A.dn_in[(int64_t)b * L + j];
      }
      if (!isfinite(R.ell[q]) || !isfinite(R.dn[q])) bad = true;
    }
  }
  R.any_bad = __any_sync(FULL, bad);
  R.stale = __any_sync(FULL, stale);
  return R;
}

// The per-step outputs (ell_j, |Delta_j|; zero outside the window) by the lanes of the warp
// that loaded R.
__device__ __forceinline__ void scan_write_steps(const ScanArgs& A, int b, const ScanRegs& R) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int j = lane + 32 * q;
    if (j < A.L) {
      if (A.ell_out) A.ell_out[(int64_t)b * A.L + j] = R.ell[q];
      if (A.dn_out) A.dn_out[(int64_t)b * A.L + j] = R.dn[q];
    }
  }
}

// The per-chain outputs known after the acceptance rule (accepted length, tau, log
// alpha_res), by one thread.
__device__ __forceinline__ void scan_write_chain(const ScanArgs& A, int b, const ChainState& cs) {
  if (A.accepted_len) A.accepted_len[b] = cs.tau > 0 ? cs.tau - 1 : 0;
  if (A.tau_out) A.tau_out[b] = cs.tau;
  if (A.la_res_out && cs.kind != kKindInactive) A.la_res_out[b] = cs.la_res;
}

// log eta_j of the lane's steps: coins from Philox (b, j, 0, 0), word 0.
__device__ __forceinline__ void scan_coins(const ScanArgs& A, int b, float (&leta)[2]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    leta[q] = 0.f;
    if (32 * q < A.L)
      leta[q] = log_uniform(philox_block(seed_of(A), (uint32_t)b, (uint32_t)(lane + 32 * q), kStreamCoin, 0u).x);
  }
}

// For chain b with loaded values R and coins log eta_j (compared in log space): the
// acceptance rule.  In block mode every
// candidate residual row j (lane j & 31 of segment j >> 5) also gets the U-sampler setup
// at (|Delta_j|, log alpha_{j-1}) (log alpha_{-1} = 0), whose log v is the residual mass
// that h_{j-1} needs: the scan evaluates it once for both.  Called by a full warp; every
// lane returns the result.  Writes nothing.
template <typename Coop>
static __device__ ScanOut scan_decide(const ScanArgs& A, int b, const ScanRegs& R, const float (&leta)[2], Coop& co) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int L = A.L;
  const int g = R.g;
  ScanOut out;
  out.have_P = false;
  if (g <= 0) {
    out.cs = inactive_state();
    return out;
  }
  const int nseg = (L + 31) >> 5;

  const float ellw[2] = {R.ell[0] * A.inv_omega2, R.ell[1] * A.inv_omega2};

  int tau;             // 1-based
  float la_res = 0.f;  // log alpha_{tau-1}
  if (A.mode == 0) {
    // sample verification: c_j = [eta_j < min{1, e^ell_j}]; tau = first failure
    unsigned fm[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int j = lane + 32 * q;
      const bool fail = (q < nseg && j < g) && !(leta[q] < fminf(0.f, ellw[q]));
      fm[q] = __ballot_sync(FULL, fail);
    }
    tau = fm[0] ? __ffs(fm[0]) : (fm[1] ? 32 + __ffs(fm[1]) : g + 1);
  } else {
    // block verification: log alpha_j = min{0, log alpha_{j-1} + ell_j}, evaluated in
    // step order by every lane on all tempered ell (gathered with independent
    // shuffles), lane j & 31 of segment j >> 5 keeping log alpha_j, so that a clamp
    // to alpha = 1 is exact exactly when the recursion reaches it
    float la[2] = {0.f, 0.f};
    float run = 0.f;
#pragma unroll 4
    for (int k = 0; k < g; ++k) {
      const float e = __shfl_sync(FULL, k < 32 ? ellw[0] : ellw[1], k & 31);
      run = fminf(0.f, run + e);
      if (k < 32) la[0] = (k == lane) ? run : la[0];
      else la[1] = (k - 32 == lane) ? run : la[1];
    }
    // log alpha_{j-1} of each candidate residual row, and its U-sampler setup
    float lap[2];
    {
      const float up0 = __shfl_up_sync(FULL, la[0], 1);
      const float last0 = __shfl_sync(FULL, la[0], 31);
      const float up1 = __shfl_up_sync(FULL, la[1], 1);
      lap[0] = (lane == 0) ? 0.f : up0;
      lap[1] = (lane == 0) ? last0 : up1;
    }
    UParams Pq[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if (q < nseg) {  // warp-uniform
        const bool ok = (R.dn[q] > 0.f) && isfinite(R.dn[q]) && isfinite(lap[q]);
        Pq[q] = usample_setup(ok ? R.dn[q] : 1.f, ok ? fminf(lap[q], 0.f) : -1.f, co);
      } else {
        Pq[q] = UParams{};
      }
    }
    // h_j (0-based j) uses |Delta| and log v of step j + 1 (the paper's D_{j+1})
    const float dnx0 = __shfl_down_sync(FULL, R.dn[0], 1);
    const float dnx1 = __shfl_down_sync(FULL, R.dn[1], 1);
    const float dnf1 = __shfl_sync(FULL, R.dn[1], 0);
    const float lvx0 = __shfl_down_sync(FULL, Pq[0].lv, 1);
    const float lvx1 = __shfl_down_sync(FULL, Pq[1].lv, 1);
    const float lvf1 = __shfl_sync(FULL, Pq[1].lv, 0);
    unsigned sm[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int j = lane + 32 * q;
      bool succ = false;
      if (q < nseg && j < g) {
        float lh;
        if (j == g - 1) {
          lh = la[q];  // h_gamma = alpha_gamma
        } else {
          const float Dn = (q == 0) ? (lane == 31 ? dnf1 : dnx0) : dnx1;
          const float lv = (q == 0) ? (lane == 31 ? lvf1 : lvx0) : lvx1;
          lh = block_log_h(la[q], Dn, lv);
        }
        succ = leta[q] < lh;
      }
      sm[q] = __ballot_sync(FULL, succ);
    }
    int last = -1;  // 0-based index of the last success
    if (sm[1]) last = 32 + 31 - __clz(sm[1]);
    else if (sm[0]) last = 31 - __clz(sm[0]);
    tau = last + 2;
    if (tau >= 2) {
      const int k = tau - 2;
      const float v0 = __shfl_sync(FULL, la[0], k & 31);
      const float v1 = __shfl_sync(FULL, la[1], k & 31);
      la_res = (k < 32) ? v0 : v1;
    }
    if (tau <= g) {  // residual parameters of row tau - 1
      const int rr = tau - 1;
      const UParams P0 = shfl_params(Pq[0], rr & 31);
      const UParams P1 = shfl_params(Pq[1], rr & 31);
      out.P = (rr >> 5) ? P1 : P0;
      out.have_P = true;
    }
  }

  // quantities of step tau (0-based row tau-1) when a residual is drawn
  const bool resid = tau <= g;
  const int rrow = resid ? tau - 1 : 0;
  const int rq = rrow >> 5, rl = rrow & 31;
  const float Dt = rq ? __shfl_sync(FULL, R.dn[1], rl) : __shfl_sync(FULL, R.dn[0], rl);
  const float st = rq ? __shfl_sync(FULL, R.sg[1], rl) : __shfl_sync(FULL, R.sg[0], rl);
  const float S1t = rq ? __shfl_sync(FULL, R.S1[1], rl) : __shfl_sync(FULL, R.S1[0], rl);
  const float S2t = rq ? __shfl_sync(FULL, R.S2[1], rl) : __shfl_sync(FULL, R.S2[0], rl);

  uint32_t status = R.any_bad ? 2u : 0u;
  int kind;
  if (!resid) {
    kind = A.has_bonus ? kKindBonus : kKindCopy;
  } else if (!(S2t > 0.f) || !(Dt > 0.f)) {
    kind = kKindZeroDelta;
    status |= 1u;
  } else if (A.residual_kind == 1) {
    kind = kKindReflect;
  } else {
    kind = kKindResid;
  }
  ChainState& cs = out.cs;
  cs.tau = tau;
  cs.row = resid ? rrow : g - 1;
  cs.U = NAN;
  cs.la_res = la_res;
  cs.sigma = resid ? st : NAN;
  cs.dnorm = resid ? Dt : NAN;
  cs.inv_norm = (S2t > 0.f) ? rsqrtf(S2t) : 0.f;
  cs.refl = (S2t > 0.f) ? 1.0f + 2.0f * S1t / S2t : 0.f;
  cs.status = status;
  cs.kind = kind;
  cs.pad[0] = cs.pad[1] = 0;
  return out;
}

// scan_load, the per-step outputs, scan_decide and the per-chain outputs in one go (the
// kernels whose writes need not wait for an earlier grid).
static __device__ ScanOut scan_warp(const ScanArgs& A, int b) {
  const ScanRegs R = scan_load(A, b);
  scan_write_steps(A, b, R);
  float leta[2];
  scan_coins(A, b, leta);
  OneWarp co;
  const ScanOut o = scan_decide(A, b, R, leta, co);
  if ((threadIdx.x & 31) == 0) scan_write_chain(A, b, o.cs);
  return o;
}

// Per-chain outputs that depend on U: status bits and (U, log alpha_res, |Delta_tau|,
// sigma_tau); written by one thread (leader).
__device__ __forceinline__ void report_chain(const ScanArgs& A, int b, const ChainState& cs, bool leader) {
  if (leader && cs.kind != kKindInactive) {
    if (A.status_out) A.status_out[b] = cs.status;
    if (A.aux_out) {
      float* a = A.aux_out + 4 * (int64_t)b;
      a[0] = cs.U;
      a[1] = cs.la_res;
      a[2] = cs.dnorm;
      a[3] = cs.sigma;
    }
  }
}

}  // namespace sdv
