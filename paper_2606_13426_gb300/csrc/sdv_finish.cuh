// sdv_finish.cuh - the output row of one chain, shared out over threads (sm_103a): the
// residual's noise, delta^T G over the rejected row, and the row itself (Algorithms
// decomposition-res and reflect-res, the bonus step, the last accepted draft).
#pragma once

#include "sdv_scan.cuh"
#include "sdv_tiles.cuh"

namespace sdv {

// Groups of four elements s0 + o, s0 + o + no, ... below s1 of the row belong to this
// thread, owner o of no.
struct RowSlice {
  int64_t s0, s1;
  int o, no;
};

// What of a slice waits between its phases.  kHoldAll: the noise in shared memory, and m^q
// and delta = m^p - m^q, of at most kOwn groups per owner, in registers; kHoldNoise: the
// noise only (the rows are read twice); kHoldNothing: the noise is drawn twice too.
// kHoldNoiseFar: kHoldNoise with longer sweeps.
enum : int { kHoldAll = 0, kHoldNoise = 1, kHoldNothing = 2, kHoldNoiseFar = 3 };

// Groups of an owner per sweep over its slice, their loads issued together: more where few
// CTAs read long rows.
constexpr int kOwn = 4;
__host__ __device__ constexpr int own_groups(int hold) { return hold == kHoldNoiseFar ? 2 * kOwn : kOwn; }
template <int OWN>
struct RowRegs {
  float fq[OWN][4], dl[OWN][4];
};

struct FinishShared {
  ChainState cs;
  float dot[32];    // delta^T G by warp
  float slice[8];   // delta^T G by CTA of a cluster
  float u;
  float leta[SDV_MAX_L];   // log eta_j
  float coop[2][kCoopPieces][32];
};

// The residual's G of the owner's groups (stream kStreamResid; it depends on the chain, not
// on the rejected step) to g_s, indexed from s0; only the owner reads it back.
template <int HOLD>
__device__ __forceinline__ void draw_noise(uint64_t seed, int b, const RowSlice& sl, float4* g_s) {
  if (HOLD == kHoldAll || HOLD == kHoldNoise || HOLD == kHoldNoiseFar) {
#pragma unroll 1
    for (int64_t gi = sl.s0 + sl.o; gi < sl.s1; gi += sl.no)
      g_s[gi - sl.s0] = normals4(seed, (uint32_t)b, (uint32_t)gi, kStreamResid, 0u);
  }
}

// The residual's noise of group gi.
template <int HOLD>
__device__ __forceinline__ float4 noise_of(uint64_t seed, int b, const RowSlice& sl, const float4* g_s, int64_t gi) {
  if (gi >= sl.s1) return make_float4(0.f, 0.f, 0.f, 0.f);
  return HOLD == kHoldNothing ? normals4_f(seed, (uint32_t)b, (uint32_t)gi, kStreamResid, 0u) : g_s[gi - sl.s0];
}

// m^q and m^p of OWN of the owner's groups from gi0 on (elements past the row's end load
// zeros, groups past the slice's end are zero), their loads issued together; rows_delta
// makes the latter delta.
template <typename T, bool VEC4, int OWN>
__device__ __forceinline__ void load_rows(const T* __restrict__ mq, const T* __restrict__ mp, int64_t d,
                                          const RowSlice& sl, int64_t gi0, float (&fq)[OWN][4], float (&fp)[OWN][4]) {
#pragma unroll
  for (int u = 0; u < OWN; ++u) {
    const int64_t gi = gi0 + (int64_t)u * sl.no;
    const int64_t i = gi < sl.s1 ? 4 * gi : d;   // d: loads nothing
    load4<T, VEC4>(mq, i, d, fq[u]);
    load4<T, VEC4>(mp, i, d, fp[u]);
  }
}

template <int OWN>
__device__ __forceinline__ void rows_delta(const float (&fq)[OWN][4], float (&dl)[OWN][4]) {
#pragma unroll
  for (int u = 0; u < OWN; ++u)
#pragma unroll
    for (int k = 0; k < 4; ++k) dl[u][k] -= fq[u][k];
}

// This thread's share of delta^T G over the slice (chain state kind kKindResid).  With
// kHoldAll the rows have been loaded (load_rows from s0 + o on).
template <typename T, bool VEC4, int HOLD>
__device__ __forceinline__ float slice_dot(const T* __restrict__ mq, const T* __restrict__ mp, int L, int64_t d,
                                           uint64_t seed, int b,
                                           const ChainState& cs, const RowSlice& sl, RowRegs<own_groups(HOLD)>& rg, const float4* g_s) {
  constexpr int OWN = own_groups(HOLD);
  const int64_t rbase = ((int64_t)b * L + cs.row) * d;
  float sp = 0.f;
  for (int64_t gi0 = sl.s0 + sl.o; gi0 < sl.s1 || HOLD == kHoldAll; gi0 += (int64_t)OWN * sl.no) {
    if (HOLD != kHoldAll) load_rows<T, VEC4>(mq + rbase, mp + rbase, d, sl, gi0, rg.fq, rg.dl);
    rows_delta(rg.fq, rg.dl);
#pragma unroll
    for (int u = 0; u < OWN; ++u) {
      const int64_t gi = gi0 + (int64_t)u * sl.no;
      const float4 G = noise_of<HOLD>(seed, b, sl, g_s, gi);
      sp = fmaf(rg.dl[u][0], G.x, sp);
      sp = fmaf(rg.dl[u][1], G.y, sp);
      sp = fmaf(rg.dl[u][2], G.z, sp);
      sp = fmaf(rg.dl[u][3], G.w, sp);
    }
    if (HOLD == kHoldAll) break;
  }
  return sp;
}

// Writes the owner's groups of y[b, :]: the decomposition residual m^q + sigma (G + e coef),
// e = delta inv_norm, coef = U - e^T G; the reflection x - delta (1 + 2 S1/S2); m^q + sigma G
// for a zero shift; the bonus step; or the last accepted draft.
template <typename T, bool VEC4, int HOLD>
__device__ __forceinline__ void slice_write(const T* __restrict__ x, const T* __restrict__ mq, const T* __restrict__ mp,
                                            const T* __restrict__ mq_bonus, const float* __restrict__ sigma_bonus, int L,
                                            int64_t d, uint64_t seed, int b, const ChainState& cs, float coef,
                                            T* __restrict__ y, const RowSlice& sl, RowRegs<own_groups(HOLD)>& rg, const float4* g_s) {
  constexpr int OWN = own_groups(HOLD);
  if (cs.kind == kKindInactive) return;
  const int64_t rbase = ((int64_t)b * L + cs.row) * d;
  const int64_t ybase = (int64_t)b * d;
  if (cs.kind == kKindResid) {
    for (int64_t gi0 = sl.s0 + sl.o; gi0 < sl.s1 || HOLD == kHoldAll; gi0 += (int64_t)OWN * sl.no) {
      if (HOLD != kHoldAll) {
        load_rows<T, VEC4>(mq + rbase, mp + rbase, d, sl, gi0, rg.fq, rg.dl);
        rows_delta(rg.fq, rg.dl);
      }
#pragma unroll
      for (int u = 0; u < OWN; ++u) {
        const int64_t gi = gi0 + (int64_t)u * sl.no;
        if (gi < sl.s1) {
          const float4 G = noise_of<HOLD>(seed, b, sl, g_s, gi);
          const float g4[4] = {G.x, G.y, G.z, G.w};
          float out[4];
#pragma unroll
          for (int k = 0; k < 4; ++k)
            out[k] = rg.fq[u][k] + cs.sigma * fmaf(rg.dl[u][k] * cs.inv_norm, coef, g4[k]);
          store4<T, VEC4>(y + ybase, 4 * gi, d, out);
        }
      }
      if (HOLD == kHoldAll) break;
    }
    return;
  }
  const bool bonus = cs.kind == kKindBonus, refl = cs.kind == kKindReflect, zero = cs.kind == kKindZeroDelta;
  const float sgm = bonus ? sigma_bonus[b] : cs.sigma;
  const T* src = bonus ? mq_bonus + ybase : (zero ? mq : x) + rbase;
  for (int64_t gi0 = sl.s0 + sl.o; gi0 < sl.s1; gi0 += (int64_t)OWN * sl.no) {
    float a[OWN][4];
#pragma unroll
    for (int u = 0; u < OWN; ++u) {
      const int64_t gi = gi0 + (int64_t)u * sl.no;
      load4<T, VEC4>(src, gi < sl.s1 ? 4 * gi : d, d, a[u]);
    }
    if (refl) {
      load_rows<T, VEC4>(mq + rbase, mp + rbase, d, sl, gi0, rg.fq, rg.dl);
      rows_delta(rg.fq, rg.dl);
    }
#pragma unroll
    for (int u = 0; u < OWN; ++u) {
      const int64_t gi = gi0 + (int64_t)u * sl.no;
      if (gi < sl.s1) {
        if (refl) {
#pragma unroll
          for (int k = 0; k < 4; ++k) a[u][k] -= rg.dl[u][k] * cs.refl;
        } else if (bonus || zero) {
          const float4 G = normals4_f(seed, (uint32_t)b, (uint32_t)gi, bonus ? kStreamBonus : kStreamResid, 0u);
          a[u][0] += sgm * G.x; a[u][1] += sgm * G.y; a[u][2] += sgm * G.z; a[u][3] += sgm * G.w;
        }
        store4<T, VEC4>(y + ybase, 4 * gi, d, a[u]);
      }
    }
  }
}

// Grid dependencies (programmatic dependent launch).  A kernel launched with the
// programmatic-serialisation attribute may start while the previous kernel on its
// stream is still running, as soon as every CTA of that kernel has called
// griddep_launch_dependents or exited; griddep_wait blocks until the previous kernel has
// completed and its writes are visible.  Without that attribute (or with no previous
// kernel) both are no-ops.
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void griddep_launch_dependents() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

}  // namespace sdv
