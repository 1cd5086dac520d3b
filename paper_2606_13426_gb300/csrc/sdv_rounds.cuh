// sdv_rounds.cuh - rounds of the speculative sampler, one chain per CTA (sm_103a); included
// by sdv_rounds_c8.cu and sdv_rounds_c16.cu, which instantiate it for their component bound.
#pragma once

#include <algorithm>

#include "sdv_sampler.cuh"
#include "sdv_scan.cuh"

namespace sdv {

// ---------------------------------------------------------------- rounds, one chain per CTA
// A chain's whole rounds (Alg. full-block-verification) in one CTA: draft, target call,
// log ratios, acceptance, residual or bonus step and the next state, for as many rounds as
// asked for.  Chains never meet (their random numbers are keyed by chain and round), so
// nothing is exchanged between CTAs and one launch runs a whole sampling.  Thread t owns the
// groups of four t, t + NT, ... (NG of them) of every row: the state, the cached score and
// the draft stay in registers, the drafted rows also go to memory (each thread reads back
// only its own groups), and the target means and scores that a round needs again, one or two
// rows, are formed again from the row's responsibilities.  RB rows go through the target
// call together: RB x MAXC distances in one warp reduce-scatter and one pass over the warps.
// While the first warp runs a round's acceptance rule and U-draw, a chain of dependent
// evaluations, the others draw the next round's noise (it depends on chain, round and step
// only), the larger part of a round's instructions.  With few chains a round is bound by that
// chain's latency (d = 1024, L = 8, up to one chain per SM: 21 us a round, 40 us with five
// kernels a round in a graph and the windows in HBM); with many by the supply of instructions
// (65 thousand warp instructions a chain and round; 456 chains use 60 % of the issue slots, the
// rest goes to barriers and instruction fetches), see rounds_fit.
// Sums over the warp of N values per lane (N = 2, 4, .. 32): lane l returns the sum of
// value l / (32 / N), added over lanes in the order of an xor butterfly 16, 8, 4, 2, 1.
template <int N>
__device__ __forceinline__ float warp_sums(float (&v)[N]) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  int n = N;
#pragma unroll
  for (int h = 16; h >= 1; h >>= 1) {
    if (n > 1) {
      n >>= 1;
      const bool up = (lane & h) != 0;
#pragma unroll
      for (int k = 0; k < N / 2; ++k) {
        if (k < n) {
          const float send = up ? v[k] : v[k + n];
          const float keep = up ? v[k + n] : v[k];
          v[k] = keep + __shfl_xor_sync(FULL, send, h);
        }
      }
    } else {
      v[0] += __shfl_xor_sync(FULL, v[0], h);
    }
  }
  return v[0];
}

// RB: rows per pass, 32 / MAXC for aligned rows of up to 1024 elements (at 768 threads per SM),
// else one.
template <int MAXC, int NT, int NG, bool VEC, int RB>
__global__ void __launch_bounds__(NT, NG == 1 ? (RB == 1 ? 1024 : 768) / NT : 1) k_rounds(RoundsArgs A) {
  constexpr int NV = RB * MAXC;          // distances per pass
  constexpr int NW = NT / 32;
  constexpr int MAXR = SDV_MAX_L + 1;
  const unsigned FULL = 0xffffffffu;
  __shared__ float4 rc_s[MAXR];          // (sqrt(abar), 1/v, beta, sigma) of step k + j
  __shared__ float resp_s[MAXR][MAXC];   // responsibilities of the round's rows
  __shared__ float wsc_s[MAXR];          // sqrt(abar) / (their sum)
  __shared__ float red_s[2][NW][NV];
  __shared__ float rw_s[NW][NV], ww_s[NW][RB];        // this pass's ([c][row]), one copy per warp
  __shared__ float s12_s[SDV_MAX_L][2][NW];
  __shared__ float lg_s[MAXC];
  __shared__ float dot_s[NW];
  __shared__ ChainState cs_s;
  extern __shared__ float4 dyn_s[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = blockIdx.x;
  const int C = A.G.C, L = A.L, d = (int)A.d, ng = (d + 3) / 4;
  float4* row_s = dyn_s;                 // [ng]: the residual's G; the state (Frozen)
  float4* nz_s = dyn_s + ng;             // [pre][ng]: the draft's noise
  const Sched& S = A.S;
  const float cst = 0.5f * (1.0f + S.churn * S.churn);
  int k = 0, g = min(L, S.K), r0 = 0;
  if (!A.fresh) {
    k = A.kk[b];
    g = A.gam[b];
    r0 = A.ctl->r;
  }
  int lr = 0, tsum = 0;

  auto load4f = [&](const float* p, int gi) {   // group gi of an unpadded row; 0 past d
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (gi < ng) {
      if (VEC) {
        v = *reinterpret_cast<const float4*>(p + 4 * gi);
      } else {
        v.x = p[4 * gi];
        if (4 * gi + 1 < d) v.y = p[4 * gi + 1];
        if (4 * gi + 2 < d) v.z = p[4 * gi + 2];
        if (4 * gi + 3 < d) v.w = p[4 * gi + 3];
      }
    }
    return v;
  };
  auto store4f = [&](float* p, int gi, float4 v) {
    if (gi < ng) {
      if (VEC) {
        *reinterpret_cast<float4*>(p + 4 * gi) = v;
      } else {
        p[4 * gi] = v.x;
        if (4 * gi + 1 < d) p[4 * gi + 1] = v.y;
        if (4 * gi + 2 < d) p[4 * gi + 2] = v.z;
        if (4 * gi + 3 < d) p[4 * gi + 3] = v.w;
      }
    }
  };
  auto mean4 = [&](int c, int i) { return load4f(A.G.means + (int64_t)c * d, tid + NT * i); };
  // elements past d stay 0, so that they add nothing to any sum
  auto masked = [&](float4 v, int gi) {
    const int e = d - 4 * gi;
    if (VEC ? e <= 0 : e < 4) {
      if (e < 1) v.x = 0.f;
      if (e < 2) v.y = 0.f;
      if (e < 3) v.z = 0.f;
      v.w = 0.f;
    }
    return v;
  };
  auto drift1 = [&](float z, float be, float sc) { return z + S.delta * (0.5f * be * z + cst * be * sc); };
  auto drift = [&](float4 z, float be, float4 sc) {
    return make_float4(drift1(z.x, be, sc.x), drift1(z.y, be, sc.y), drift1(z.z, be, sc.z), drift1(z.w, be, sc.w));
  };
  // score of group i of a row from its responsibilities (r[c], w)
  auto score = [&](const float* r, float w, float inv_v, int i, float4 z) {
    float ws[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int c = 0; c < MAXC; ++c) {
      if (c < C) {
        const float4 m = mean4(c, i);
        const float rc = r[c];
        ws[0] = fmaf(rc, m.x, ws[0]);
        ws[1] = fmaf(rc, m.y, ws[1]);
        ws[2] = fmaf(rc, m.z, ws[2]);
        ws[3] = fmaf(rc, m.w, ws[3]);
      }
    }
    return make_float4((w * ws[0] - z.x) * inv_v, (w * ws[1] - z.y) * inv_v, (w * ws[2] - z.z) * inv_v,
                       (w * ws[3] - z.w) * inv_v);
  };
  auto dist = [&](float4 z, float4 m, float sab, float a) {
    const float zf[4] = {z.x, z.y, z.z, z.w}, mf[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float df = zf[e] - sab * mf[e];
      a = fmaf(df, df, a);
    }
    return a;
  };
  // responsibilities of the rows whose distances lie in red (values row * MAXC + c): lane
  // l of every warp gets exp(logit - max) of value l, with the normalised weight of its row
  auto softmax = [&](const float (*red)[NV], int row0, int nrows, float& wsc) {
    const int v = lane % NV, r = v / MAXC, c = v - r * MAXC;
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < NW; ++w) t += red[w][v];
    const float4 rc = rc_s[row0 + min(r, nrows - 1)];
    const float a = (c < C) ? __ldg(A.G.log_w + c) - 0.5f * t * rc.y : -INFINITY;
    float mx = a;
#pragma unroll
    for (int o = MAXC / 2; o >= 1; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(FULL, mx, o));
    const float ex = (c < C) ? expf(a - mx) : 0.f;
    float den = ex;
#pragma unroll
    for (int o = MAXC / 2; o >= 1; o >>= 1) den += __shfl_xor_sync(FULL, den, o);
    wsc = rc.x / den;
    return ex;
  };

  float* yrow = A.y + (int64_t)b * d;
  float* scrow = A.sc + (int64_t)b * d;
  const int64_t dp = 4 * (int64_t)ng;
  float* rows = A.rows + (int64_t)b * L * dp;
  auto row4 = [&](int j, int i) -> float4& {   // this thread's group i of drafted row j
    return *reinterpret_cast<float4*>(rows + (int64_t)j * dp + 4 * (tid + NT * i));
  };
  float4 y[NG], sc[NG];
#pragma unroll
  for (int i = 0; i < NG; ++i) {
    const int gi = tid + NT * i;
    y[i] = A.fresh ? masked(normals4_f(A.seed, (uint32_t)b, (uint32_t)gi, kStreamInit, 0u), gi) : load4f(yrow, gi);
    sc[i] = A.fresh ? make_float4(0.f, 0.f, 0.f, 0.f) : load4f(scrow, gi);
  }

  // noise of the first `pre` draft rows of round r0 + n, and (with_g) the residual's G of the
  // round before it, a group per lane, by warps w0, w0 + 1, ...
  auto draw_ahead = [&](int n, int w0, bool with_g) {
    const uint64_t sn = round_seed(A.seed, r0 + n), sp = round_seed(A.seed, r0 + n - 1);
    const int W = (ng + 31) / 32, items = W * (n < A.max_rounds ? A.pre : 0), all = items + (with_g ? W : 0);
#pragma unroll 1
    for (int it = warp - w0; it < all; it += NW - w0) {
      const int j = it / W, gi = (it - j * W) * 32 + lane;
      const bool res = it >= items;
      if (gi < ng) {
        const float4 v = normals4(res ? sp : sn, (uint32_t)b, (uint32_t)gi, res ? kStreamResid : kStreamDraft,
                                  res ? 0u : (uint32_t)j);
        if (res) row_s[gi] = v;
        else nz_s[j * ng + gi] = v;
      }
    }
  };
  if (g > 0) draw_ahead(0, 0, false);

  while (g > 0 && lr < A.max_rounds) {
    const uint64_t rs = round_seed(A.seed, r0 + lr);
    for (int j = tid; j <= g; j += NT) {
      const float tf = S.tfwd(k + j);
      const float ab = S.abar(tf);
      rc_s[j] = make_float4(sqrtf(ab), 1.0f / (ab * A.G.comp_var + 1.0f - ab), S.beta(tf), S.sigma(k + j));
    }
    // the start state's score: of every round (Frozen), or of a run's first (the only
    // explicit target call of the Free drafter)
    const bool score_now = A.frozen || (A.fresh && lr == 0);
    if (score_now) {
#pragma unroll
      for (int i = 0; i < NG; ++i)
        if (tid + NT * i < ng) row_s[tid + NT * i] = y[i];
    }
    __syncthreads();
    if (score_now) {
      // its distances summed as the target
      // call of single rows does (gmm_rows_warp): a warp takes whole components
      const float4 rc = rc_s[0];
      for (int c = warp; c < C; c += NW) {
        const float* mu = A.G.means + (int64_t)c * d;
        float a = 0.f;
#pragma unroll 2
        for (int gi = lane; gi < ng; gi += 32) a = dist(row_s[gi], load4f(mu, gi), rc.x, a);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(FULL, a, o);
        if (lane == 0) lg_s[c] = __ldg(A.G.log_w + c) - 0.5f * a * rc.y;
      }
      __syncthreads();
      float mx = -INFINITY, den = 0.f, r[MAXC];
#pragma unroll
      for (int c = 0; c < MAXC; ++c) {
        r[c] = (c < C) ? lg_s[c] : -INFINITY;
        mx = fmaxf(mx, r[c]);
      }
#pragma unroll
      for (int c = 0; c < MAXC; ++c) {
        r[c] = (c < C) ? expf(r[c] - mx) : 0.f;
        den += r[c];
      }
      const float w = rc.x / den;
#pragma unroll
      for (int i = 0; i < NG; ++i) sc[i] = masked(score(r, w, rc.y, i, y[i]), tid + NT * i);
    }

    // draft and target call, RB rows at a time
    float4 z[RB + 1][NG];
#pragma unroll
    for (int i = 0; i < NG; ++i) z[0][i] = y[i];
    int buf = 0;
#pragma unroll 1
    for (int j0 = 0; j0 < g; j0 += RB, buf ^= 1) {
      const int nr = min(RB, g - j0);
#pragma unroll
      for (int q = 0; q < RB; ++q) {
        if (q < nr) {
          const float4 rc = rc_s[j0 + q];
#pragma unroll
          for (int i = 0; i < NG; ++i) {
            const int gi = tid + NT * i;
            const float4 n = j0 + q < A.pre ? nz_s[(j0 + q) * ng + min(gi, ng - 1)]
                                            : normals4_f(rs, (uint32_t)b, (uint32_t)gi, kStreamDraft, (uint32_t)(j0 + q));
            const float4 m = drift(z[q][i], rc.z, sc[i]);
            z[q + 1][i] = masked(make_float4(m.x + rc.w * n.x, m.y + rc.w * n.y, m.z + rc.w * n.z, m.w + rc.w * n.w), gi);
            if (gi < ng) row4(j0 + q, i) = z[q + 1][i];
          }
        }
      }
      float v[NV];
#pragma unroll
      for (int q = 0; q < NV; ++q) v[q] = 0.f;
#pragma unroll
      for (int i = 0; i < NG; ++i) {
#pragma unroll
        for (int c = 0; c < MAXC; ++c) {
          if (c < C) {
            const float4 m = mean4(c, i);
#pragma unroll
            for (int q = 0; q < RB; ++q)
              if (q < nr) v[q * MAXC + c] = dist(z[q][i], m, rc_s[j0 + q].x, v[q * MAXC + c]);
          }
        }
      }
      const float vs = warp_sums<NV>(v);
      if (lane % (32 / NV) == 0) red_s[buf][warp][lane / (32 / NV)] = vs;
      __syncthreads();
      float wsc;
      const float ex = softmax(red_s[buf], j0, nr, wsc);
      if (lane < NV) {
        rw_s[warp][lane % MAXC * RB + lane / MAXC] = ex;
        if (lane % MAXC == 0) ww_s[warp][lane / MAXC] = wsc;
        if (warp == 0 && lane / MAXC < nr) {
          resp_s[j0 + lane / MAXC][lane % MAXC] = ex;
          if (lane % MAXC == 0) wsc_s[j0 + lane / MAXC] = wsc;
        }
      }
      __syncwarp();
      float ws[RB][NG][4];
#pragma unroll
      for (int q = 0; q < RB; ++q)
#pragma unroll
        for (int i = 0; i < NG; ++i) ws[q][i][0] = ws[q][i][1] = ws[q][i][2] = ws[q][i][3] = 0.f;
#pragma unroll
      for (int c = 0; c < MAXC; ++c) {
        if (c < C) {
          float rq[RB];
#pragma unroll
          for (int q = 0; q < RB; ++q) rq[q] = rw_s[warp][c * RB + q];
#pragma unroll
          for (int i = 0; i < NG; ++i) {
            const float4 m = mean4(c, i);
#pragma unroll
            for (int q = 0; q < RB; ++q) {
              ws[q][i][0] = fmaf(rq[q], m.x, ws[q][i][0]);
              ws[q][i][1] = fmaf(rq[q], m.y, ws[q][i][1]);
              ws[q][i][2] = fmaf(rq[q], m.z, ws[q][i][2]);
              ws[q][i][3] = fmaf(rq[q], m.w, ws[q][i][3]);
            }
          }
        }
      }
      float s12[2 * RB];
#pragma unroll
      for (int q = 0; q < 2 * RB; ++q) s12[q] = 0.f;
#pragma unroll
      for (int q = 0; q < RB; ++q) {
        if (q < nr) {
          const float4 rc = rc_s[j0 + q];
          const float w = ww_s[warp][q];
          float s1 = 0.f, s2 = 0.f;
#pragma unroll
          for (int i = 0; i < NG; ++i) {
            const float zf[4] = {z[q][i].x, z[q][i].y, z[q][i].z, z[q][i].w};
            const float cf[4] = {sc[i].x, sc[i].y, sc[i].z, sc[i].w};
            const float fx[4] = {z[q + 1][i].x, z[q + 1][i].y, z[q + 1][i].z, z[q + 1][i].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {   // elements past d: z = sc = 0 and zero means give 0
              const float fq = drift1(zf[e], rc.z, (w * ws[q][i][e] - zf[e]) * rc.y), fp = drift1(zf[e], rc.z, cf[e]);
              const float dl = fp - fq, a = fx[e] - fp;
              s1 = fmaf(a, dl, s1);
              s2 = fmaf(dl, dl, s2);
            }
          }
          s12[2 * q] = s1;
          s12[2 * q + 1] = s2;
        }
      }
      const float ss = warp_sums<2 * RB>(s12);
      const int si = lane / (16 / RB);   // 2 row + which sum
      if (lane % (16 / RB) == 0 && si / 2 < nr) s12_s[j0 + si / 2][si & 1][warp] = ss;
#pragma unroll
      for (int i = 0; i < NG; ++i) z[0][i] = z[RB][i];
    }
    __syncthreads();

    // acceptance and U by warp 0, while the other warps draw the residual's noise and the
    // next round's
    if (warp == 0) {
      ScanArgs SA{};
      SA.L = L; SA.seed = rs; SA.mode = A.mode; SA.inv_omega2 = 1.0f; SA.has_bonus = true;
      ScanRegs R;
      R.g = g;
      bool bad = false;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int j = lane + 32 * q;
        R.ell[q] = 0.f; R.dn[q] = 0.f; R.S1[q] = 0.f; R.S2[q] = 0.f; R.sg[q] = 1.f;
        if (j < g) {
          float t[2][8];
#pragma unroll
          for (int w = 0; w < 8; ++w) {
            t[0][w] = w < NW ? s12_s[j][0][w] : 0.f;
            t[1][w] = w < NW ? s12_s[j][1][w] : 0.f;
          }
          const float s1 = ((t[0][0] + t[0][4]) + (t[0][2] + t[0][6])) + ((t[0][1] + t[0][5]) + (t[0][3] + t[0][7]));
          const float s2 = ((t[1][0] + t[1][4]) + (t[1][2] + t[1][6])) + ((t[1][1] + t[1][5]) + (t[1][3] + t[1][7]));
          bad |= scan_step(R, q, s1, s2, rc_s[j].w);
          bad |= !isfinite(R.ell[q]) || !isfinite(R.dn[q]);
        }
      }
      R.any_bad = __any_sync(FULL, bad);
      R.stale = false;
      float leta[2];
      scan_coins(SA, b, leta);
      OneWarp co;
      const ScanOut so = scan_decide(SA, b, R, leta, co);
      ChainState cs = so.cs;
      if (cs.kind == kKindResid) {
        const uint32_t wbits = philox_block(rs, (uint32_t)b, 0u, kStreamUSample, 0u).x;
        uint32_t st = 0u;
        const UParams Q = so.have_P ? so.P : usample_setup(cs.dnorm, fminf(cs.la_res, 0.f), co);
        cs.U = usample_warp(Q, wbits, &st, co);
      }
      if (lane == 0) cs_s = cs;
      if (NW == 1) draw_ahead(lr + 1, 0, true);
    } else {
      draw_ahead(lr + 1, NW > 1 ? 1 : 0, true);
    }
    __syncthreads();
    const ChainState cs = cs_s;
    const int tau = cs.tau;
    if (tau >= g) {
      // the target call at the window's last state, which only these chains need
      float v[MAXC];
#pragma unroll
      for (int c = 0; c < MAXC; ++c) v[c] = 0.f;
#pragma unroll
      for (int i = 0; i < NG; ++i) {
        const float4 zg = tid + NT * i < ng ? row4(g - 1, i) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int c = 0; c < MAXC; ++c)
          if (c < C) v[c] = dist(zg, mean4(c, i), rc_s[g].x, v[c]);
      }
      const float vs = warp_sums<MAXC>(v);
      if (lane % (32 / MAXC) == 0) {
        const int c = lane / (32 / MAXC);
#pragma unroll
        for (int q = 0; q < RB; ++q) red_s[0][warp][q * MAXC + c] = vs;   // softmax reads every row
      }
      __syncthreads();
      float wsc;
      const float ex = softmax(red_s[0], g, 1, wsc);
      if (warp == 0 && lane < MAXC) {
        resp_s[g][lane] = ex;
        if (lane == 0) wsc_s[g] = wsc;
      }
    }
    float coef = 0.f;
    const int rr = tau - 1;   // rejected row
    float4 fq[NG], fp[NG], G[NG];
    float dot = 0.f;
    if (tau <= g) {
      const float4 rc = rc_s[rr];
#pragma unroll
      for (int i = 0; i < NG; ++i) {
        const int gi = tid + NT * i;
        const float4 zr = rr == 0 ? y[i] : (gi < ng ? row4(rr - 1, i) : make_float4(0.f, 0.f, 0.f, 0.f));
        fq[i] = drift(zr, rc.z, score(resp_s[rr], wsc_s[rr], rc.y, i, zr));
        fp[i] = drift(zr, rc.z, sc[i]);
        G[i] = row_s[min(gi, ng - 1)];
        dot = fmaf(fp[i].x - fq[i].x, G[i].x, dot);   // past d delta is 0
        dot = fmaf(fp[i].y - fq[i].y, G[i].y, dot);
        dot = fmaf(fp[i].z - fq[i].z, G[i].z, dot);
        dot = fmaf(fp[i].w - fq[i].w, G[i].w, dot);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(FULL, dot, o);
      if (lane == 0) dot_s[warp] = dot;
    }
    __syncthreads();
    if (tau <= g && cs.kind == kKindResid) {
      float t = dot_s[0];
#pragma unroll
      for (int w = 1; w < NW; ++w) t += dot_s[w];
      coef = cs.U - t * cs.inv_norm;   // U - e^T G
    }
    const bool end = tau > g && k + g >= S.K;   // no bonus step past the end of sampling
    const int st = min(tau, g);
#pragma unroll
    for (int i = 0; i < NG; ++i) {
      const int gi = tid + NT * i;
      const float4 zs = gi < ng ? row4(st - 1, i) : make_float4(0.f, 0.f, 0.f, 0.f);
      const float4 rc = rc_s[st];
      const float4 ns = score(resp_s[st], wsc_s[st], rc.y, i, zs);
      float4 ny;
      if (tau <= g) {
        const float q4[4] = {fq[i].x, fq[i].y, fq[i].z, fq[i].w}, p4[4] = {fp[i].x, fp[i].y, fp[i].z, fp[i].w};
        const float g4[4] = {G[i].x, G[i].y, G[i].z, G[i].w};
        float o[4];
#pragma unroll
        for (int e = 0; e < 4; ++e)
          o[e] = cs.kind == kKindResid ? q4[e] + cs.sigma * fmaf((p4[e] - q4[e]) * cs.inv_norm, coef, g4[e])
                                       : q4[e] + cs.sigma * g4[e];
        ny = make_float4(o[0], o[1], o[2], o[3]);
      } else if (end) {
        ny = zs;
      } else {
        const float4 n = normals4(rs, (uint32_t)b, (uint32_t)gi, kStreamBonus, 0u);
        const float4 mb = drift(zs, rc.z, ns);
        ny = make_float4(mb.x + rc.w * n.x, mb.y + rc.w * n.y, mb.z + rc.w * n.z, mb.w + rc.w * n.w);
      }
      y[i] = masked(ny, gi);
      sc[i] = masked(ns, gi);
    }
    k = min(k + tau, S.K);
    g = k < S.K ? min(L, S.K - k) : 0;
    tsum += tau;
    ++lr;
    __syncthreads();   // the shared arrays are read
  }

  if (lr > 0) {
#pragma unroll
    for (int i = 0; i < NG; ++i) {
      store4f(yrow, tid + NT * i, y[i]);
      store4f(scrow, tid + NT * i, sc[i]);
      if (A.y_out) store4f(A.y_out + (int64_t)b * d, tid + NT * i, y[i]);
    }
    if (tid == 0) {
      const int nr = A.fresh ? lr : A.rounds[b] + lr, nt = A.fresh ? tsum : A.tsum[b] + tsum;
      A.kk[b] = k;
      A.gam[b] = g;
      A.rounds[b] = nr;
      A.tsum[b] = nt;
      if (A.k_out) A.k_out[b] = k;
      if (A.rounds_out) A.rounds_out[b] = nr;
      if (A.tsum_out) A.tsum_out[b] = nt;
    }
  }
  if (tid == 0) {
    if (lr > 0) atomicMax(&A.ctl->active, (unsigned)lr);
    if (ticket_acq_rel(&A.ctl->done) == gridDim.x - 1) {
      // the last chain: every CTA has read the round counter
      const int r = r0 + (A.one_round ? 1 : (int)atomicAdd(&A.ctl->active, 0u));
      A.ctl->r = r;
      A.ctl->seed_r = round_seed(A.seed, r);
      A.ctl->active = 0u;
      A.ctl->done = 0u;
    }
  }
}


// `rounds` rounds of every chain in one launch (rows of up to kRoundMaxD elements).
template <int MAXC, int NT, int NG, bool VEC, int RB>
static int launch_rounds_t(RoundsArgs A, cudaStream_t s) {
  const size_t row = sizeof(float4) * (size_t)((A.d + 3) / 4);
  constexpr size_t kAhead = 32 * 1024;   // for noise drawn ahead: eight rows of 1024 elements
  A.pre = (int)std::min<size_t>((size_t)A.L, kAhead / row);
  const size_t smem = row * (size_t)(1 + A.pre);
  if (smem > 32 * 1024) {
    // the limit is shared by all host threads: that of this kernel's longest rows
    constexpr size_t kMost = sizeof(float4) * NT * NG + kAhead;
    const cudaError_t e = cudaFuncSetAttribute(k_rounds<MAXC, NT, NG, VEC, RB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMost);
    if (e != cudaSuccess) {
      set_last_cuda_error((int)e);
      cudaGetLastError();
      return SDV_ECUDA;
    }
  }
  k_rounds<MAXC, NT, NG, VEC, RB><<<(unsigned)A.B, NT, smem, s>>>(A);
  return launch_check();
}

template <int MAXC>
int launch_rounds_c(const RoundsArgs& A, bool vec, cudaStream_t s) {
  if (!vec) {
    if (A.d <= 256) return launch_rounds_t<MAXC, 64, 1, false, 1>(A, s);
    if (A.d <= 1024) return launch_rounds_t<MAXC, 256, 1, false, 1>(A, s);
    return launch_rounds_t<MAXC, 256, 4, false, 1>(A, s);
  }
  constexpr int RB = 32 / MAXC;
  if (A.d <= 128) return launch_rounds_t<MAXC, 32, 1, true, RB>(A, s);
  if (A.d <= 256) return launch_rounds_t<MAXC, 64, 1, true, RB>(A, s);
  if (A.d <= 512) return launch_rounds_t<MAXC, 128, 1, true, RB>(A, s);
  if (A.d <= 1024) return launch_rounds_t<MAXC, 256, 1, true, RB>(A, s);
  if (A.d <= 2048) return launch_rounds_t<MAXC, 256, 2, true, 1>(A, s);
  return launch_rounds_t<MAXC, 256, 4, true, 1>(A, s);
}

}  // namespace sdv
