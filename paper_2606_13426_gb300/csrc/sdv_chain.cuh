// sdv_chain.cuh - one verification call of few chains as ONE kernel (sm_103a); included by
// sdv_chain_f32.cu and sdv_chain_bf16.cu, which instantiate it for their type.
//
// A cluster of CTAs takes a chain from its window to its output row: the CTAs stream the
// chain's tiles (App. "Density ratio calculations") and send each tile's (S1, S2) to the
// first CTA's shared memory; that CTA's first warp runs the acceptance rule (Algorithms
// token- / block-verification) while every other warp of the cluster draws the residual's
// Gaussian for its own slice of the row; the rejected step goes to all CTAs, which reduce
// delta^T G over their slices while the first warp draws U (Algorithm u-sample); then every
// CTA writes its slice of y (Algorithm decomposition-res, reflect-res, the bonus step or the
// last accepted draft).  Nothing passes through global memory between the phases, no
// counters have to be cleared, and the workspace is not used.
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <type_traits>

#include "sdv_device.cuh"
#include "sdv_host.h"
#include "sdv_scan.cuh"
#include "sdv_tiles.cuh"
#include "sdv_finish.cuh"
#include "sdv_chain.h"

namespace sdv {

// CTAs of k_chain per SM: up to 128 registers.  (Three, with 80 registers and a few of them
// spilled around the U-draw's calls: pixel batch 24.4 -> 28.7 us.)
constexpr int kChainPerSm = 2;

// ---------------------------------------------------------------- clusters
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// The two halves of a barrier that orders no memory: passing it shows that every CTA of the
// cluster has started, which remote stores need.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.aligned;" ::: "memory"); }
// Barrier over the cluster's threads; shared-memory writes before it, remote ones among
// them, are visible after it.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Stores a 32-bit word at shared-memory variable p of the cluster's CTA `rank`.
__device__ __forceinline__ void remote_store(void* p, uint32_t rank, uint32_t v) {
  uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(r), "r"(v) : "memory");
}

// Tiles whose loads a thread has in flight together (about twelve 16-byte loads).
__host__ __device__ constexpr int tiles_in_flight(int vpt) { return vpt == 1 ? 4 : (vpt == 2 ? 2 : 1); }

// The (S1, S2) share of this thread in NB consecutive tiles of this CTA's list (tile t of
// the chain is step t / C, chunk t % C), all loads issued before any sum; in_flight() runs
// while they are under way.
template <typename T, int VK, int VPT, int NB, typename Hook>
__device__ __forceinline__ void tiles_of(const VerifyArgs& A, int64_t row0, int t0, int dt, int nt, float2 (&s)[NB],
                                         const Hook& in_flight) {
  const T* x = (const T*)A.x;
  const T* mq = (const T*)A.mq;
  const T* mp = (const T*)A.mp;
  const int C = A.S.C;
  if (VK == kRowsAligned) {
    TileBuf<VPT> B[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int t = t0 + q * dt;
      const int j = C == 1 ? t : t / C, c = t - j * C;
      const int64_t e0 = (int64_t)c * A.chunk;
      const int64_t e1 = t < nt ? min(e0 + A.chunk, A.d) : e0;
      tile_issue<T, VPT>(x, mq, mp, (row0 + j) * A.d, e0, e1, B[q]);
    }
    in_flight();
#pragma unroll
    for (int q = 0; q < NB; ++q) s[q] = tile_fma<T, VPT>(B[q]);
  } else if (VK == kRowsUnaligned) {
    TileBuf<VPT> B[NB];
    EdgeBuf E[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int t = t0 + q * dt;
      const int j = C == 1 ? t : t / C, c = t - j * C;
      const bool in = t < nt;   // a tile past the list: an empty row
      unaligned_issue<T, VPT>(x, mq, mp, in ? (row0 + j) * A.d : 0, in ? A.d : 0, c, C, B[q], E[q]);
    }
    in_flight();
#pragma unroll
    for (int q = 0; q < NB; ++q) s[q] = unaligned_fma<T, VPT>(B[q], E[q]);
  } else if (A.d <= kElementMax) {  // short rows: a step each
    auto sums = [&](auto per) {
      constexpr int E = decltype(per)::value;
      float fx[NB][E], fq[NB][E], fp[NB][E];
#pragma unroll
      for (int q = 0; q < NB; ++q) {
        const int t = t0 + q * dt;
#pragma unroll
        for (int k = 0; k < E; ++k) {
          const int i = threadIdx.x + k * kK1Threads;
          const int64_t e = (row0 + t) * A.d + i;
          const bool in = t < nt && i < (int)A.d;
          fx[q][k] = in ? Elem<T>::load(x + e) : 0.f;
          fq[q][k] = in ? Elem<T>::load(mq + e) : 0.f;
          fp[q][k] = in ? Elem<T>::load(mp + e) : 0.f;
        }
      }
      in_flight();
#pragma unroll
      for (int q = 0; q < NB; ++q) {
        s[q] = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < E; ++k) {
          const float dl = fp[q][k] - fq[q][k], a = fx[q][k] - fp[q][k];
          s[q].x = fmaf(a, dl, s[q].x);
          s[q].y = fmaf(dl, dl, s[q].y);
        }
      }
    };
    if (A.d <= kK1Threads) sums(std::integral_constant<int, 1>());
    else sums(std::integral_constant<int, kElementsPerThread>());
  } else {
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int t = t0 + q * dt;
      const int j = C == 1 ? t : t / C, c = t - j * C;
      const int64_t e0 = (int64_t)c * A.chunk;
      s[q] = t < nt ? tile_sums<T>(x, mq, mp, (row0 + j) * A.d, e0, min(e0 + A.chunk, A.d)) : make_float2(0.f, 0.f);
    }
    in_flight();
  }
}

// Streams tiles t0, t0 + dt, ... below nt of the chain whose rows start at row0; this CTA's
// i-th tile leaves each warp's sums in warp_s[i][warp].  The warps go their own pace; once()
// runs behind the first tiles' loads, or without any.
template <typename T, int VK, int VPT, int NB, typename Hook>
__device__ __forceinline__ void stream_tiles(const VerifyArgs& A, int64_t row0, int t0, int dt, int nt, int most,
                                             float2* warp_s, const Hook& once) {
  constexpr int NW = kK1Threads / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (t0 >= nt) once();
  for (int i = 0; t0 + i * dt < nt; i += NB) {
    float2 s[NB];
    tiles_of<T, VK, VPT, NB>(A, row0, t0 + i * dt, dt, nt, s, [&] { if (i == 0) once(); });
#pragma unroll
    for (int q = 0; q < NB; ++q) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        s[q].x += __shfl_xor_sync(0xffffffffu, s[q].x, o);
        s[q].y += __shfl_xor_sync(0xffffffffu, s[q].y, o);
      }
      if (lane == 0 && i + q < most) warp_s[(size_t)(i + q) * NW + warp] = s[q];
    }
  }
}

// Sums this CTA's tiles over its warps in block_sum2's order (so that they equal k_tiles'
// partials) and puts them at their places rank, rank + cl, ... below n of the first CTA's
// tile_s.
__device__ __forceinline__ void send_tiles(const float2* warp_s, int rank, int cl, int n, float2* tile_s) {
  constexpr int NW = kK1Threads / 32;
  for (int tl = threadIdx.x; rank + tl * cl < n; tl += blockDim.x) {
    const float2* w = warp_s + (size_t)tl * NW;
    const float s1 = ((w[0].x + w[4].x) + (w[2].x + w[6].x)) + ((w[1].x + w[5].x) + (w[3].x + w[7].x));
    const float s2 = ((w[0].y + w[4].y) + (w[2].y + w[6].y)) + ((w[1].y + w[5].y) + (w[3].y + w[7].y));
    float2* dst = tile_s + rank + tl * cl;
    if (cl > 1) {
      remote_store(&dst->x, 0u, __float_as_uint(s1));
      remote_store(&dst->y, 0u, __float_as_uint(s2));
    } else {
      *dst = make_float2(s1, s2);
    }
  }
}

// The groups of the row that this thread owns: those of the CTA's slice, shared out over all
// warps but the first (which scans the chain in the first CTA).
__device__ __forceinline__ RowSlice cluster_slice(int64_t d, int cl, int rank) {
  const int64_t ng = (d + 3) / 4, per = (ng + cl - 1) / cl;
  return RowSlice{min(rank * per, ng), min((rank + 1) * per, ng), (int)threadIdx.x - 32, (int)blockDim.x - 32};
}

// What finishing can do before the chain's sums are known: the coins, by the first CTA's
// first warp, and the residual's noise, by all other warps.
template <int HOLD>
__device__ __forceinline__ void finish_ahead(const VerifyArgs& A, int b, int rank, const RowSlice& sl, float4* g_s,
                                             FinishShared& fs) {
  if (threadIdx.x >= 32) {
    draw_noise<HOLD>(seed_of(A.S), b, sl, g_s);
  } else if (rank == 0) {
    float leta[2];
    scan_coins(A.S, b, leta);
    fs.leta[threadIdx.x] = leta[0];
    fs.leta[threadIdx.x + 32] = leta[1];
  }
}

constexpr int kMaxScanners = 5;   // warps that share the scan's evaluations

// From the chain's tile sums (tile_s of the cluster's first CTA) to its outputs.  g > 0.
template <typename T, bool VEC4, int HOLD, int NT>
__device__ __forceinline__ void finish_cluster(const VerifyArgs& A, int b, int cl, int rank, const float2* tile_s,
                                               const RowSlice& sl, const float4* g_s, FinishShared& fs) {
  constexpr int NW = NT / 32;
  const int L = A.S.L;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint64_t seed = seed_of(A.S);
  // Several warps of the first CTA share the long evaluations of the scan and the U-draw: five
  // where CTAs have an SM to themselves, three where two share one and the rows wait in
  // registers (the others reduce delta^T G beside them), else its first warp alone.
  constexpr bool kAll = HOLD == kHoldAll;
  const int scanners = gridDim.x <= (unsigned)A.sms ? kMaxScanners : (kAll ? 3 : 1);
  CtaWarps co{fs.coop, 0, scanners};
  RowRegs<own_groups(HOLD)> rg;
  ScanRegs R;
  UParams P;
  bool have_P = false;
  // ---- acceptance (the first CTA)
  if (rank == 0 && warp < scanners) {
    // the coins, which warp 0 has drawn (k_finish_long comes here without a barrier since;
    // warps that decide differently would part for ever)
    if (scanners > 1) asm volatile("bar.sync 2, %0;" ::"r"(32 * scanners) : "memory");
    else __syncwarp();
    R = scan_load(A.S, b, false, tile_s);
    const float leta[2] = {fs.leta[lane], fs.leta[lane + 32]};
    const ScanOut so = scan_decide(A.S, b, R, leta, co);
    P = so.P;
    have_P = so.have_P;
    // the chain's state to every CTA of the cluster, one lane to each
    const uint32_t* w = reinterpret_cast<const uint32_t*>(&so.cs);
    uint32_t* dst = reinterpret_cast<uint32_t*>(&fs.cs);
    if (warp == 0 && lane < cl) {
#pragma unroll
      for (int i = 0; i < (int)(sizeof(ChainState) / 4); ++i) {
        if (cl > 1) remote_store(dst + i, (uint32_t)lane, w[i]);
        else dst[i] = w[i];
      }
    }
  }
  if (cl > 1) cluster_sync();
  else __syncthreads();

  // ---- U in the first CTA, delta^T G by all owners
  ChainState cs = fs.cs;
  float coef = 0.f;
  if (cs.kind == kKindResid) {
    const int64_t rbase = ((int64_t)b * L + cs.row) * A.d;
    if (kAll && warp > 0)   // in flight during the draw
      load_rows<T, VEC4>((const T*)A.mq + rbase, (const T*)A.mp + rbase, A.d, sl, sl.s0 + sl.o, rg.fq, rg.dl);
    if (rank == 0 && warp < scanners) {
      const uint32_t wbits = philox_block(seed, (uint32_t)b, 0u, kStreamUSample, 0u).x;
      uint32_t st = cs.status;
      const UParams Q = have_P ? P : usample_setup(cs.dnorm, fminf(cs.la_res, 0.f), co);
      cs.U = usample_warp(Q, wbits, &st, co);
      cs.status = st;
      if (warp == 0) {
        if (cl > 1) {
          if (lane < cl) remote_store(&fs.u, (uint32_t)lane, __float_as_uint(cs.U));
        } else if (lane == 0) {
          fs.u = cs.U;
        }
      }
    }
    if (warp > 0) {
      float dot = slice_dot<T, VEC4, HOLD>((const T*)A.mq, (const T*)A.mp, L, A.d, seed, b, cs, sl, rg, g_s);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
      if (lane == 0) fs.dot[warp] = dot;
    }
    __syncthreads();
    if (tid >= 32 && tid < 32 + cl) {        // the CTA's sum to every CTA
      float t = fs.dot[1];
#pragma unroll
      for (int w = 2; w < NW; ++w) t += fs.dot[w];
      if (cl > 1) remote_store(&fs.slice[rank], (uint32_t)(tid - 32), __float_as_uint(t));
      else fs.slice[0] = t;
    }
    if (cl > 1) cluster_sync();
    else __syncthreads();
    float t = 0.f;
    for (int r = 0; r < cl; ++r) t += fs.slice[r];
    coef = fs.u - t * cs.inv_norm;           // U - e^T G
  }
  // ---- outputs (of k_finish_long: once the stream and all before it have completed)
  griddep_wait();
  if (warp > 0) {
    slice_write<T, VEC4, HOLD>((const T*)A.x, (const T*)A.mq, (const T*)A.mp, (const T*)A.mq_bonus, A.sigma_bonus, L,
                                A.d, seed, b, cs, coef, (T*)A.y, sl, rg, g_s);
  } else if (rank == 0) {
    scan_write_steps(A.S, b, R);
    if (lane == 0) {
      scan_write_chain(A.S, b, cs);
      report_chain(A.S, b, cs, true);
    }
  }
}

// A finished chain's outputs (g = 0): zero per-step outputs, nothing else.
__device__ __forceinline__ void finish_inactive(const VerifyArgs& A, int b, int rank) {
  if (rank == 0 && threadIdx.x < 32) {
    griddep_wait();
    const ScanRegs R{};
    scan_write_steps(A.S, b, R);
    if (threadIdx.x == 0) scan_write_chain(A.S, b, inactive_state());
  }
}

// The whole call.  ROWS: how rows are read (kRows*).  cl: CTAs of a cluster.
template <typename T, int ROWS, int VPT, bool VEC4, int HOLD>
__global__ void __launch_bounds__(kK1Threads, kChainPerSm) k_chain(VerifyArgs A, int cl) {
  constexpr int NW = kK1Threads / 32;
  constexpr int NB = tiles_in_flight(VPT);
  extern __shared__ float4 dyn_s[];
  __shared__ FinishShared fs;
  const int L = A.S.L, C = A.S.C;
  const int b = blockIdx.x / cl;
  const int rank = cl > 1 ? (int)cluster_rank() : 0;
  // launched to overlap the end of the work before it, this kernel starts when that has
  // completed, and lets a kernel launched the same way get ready behind it
  griddep_wait();
  griddep_launch_dependents();
  const int g = A.S.L_eff ? max(0, min(A.S.L_eff[b], L)) : L;
  if (g == 0) {                                           // the whole cluster
    finish_inactive(A, b, rank);
    return;
  }
  if (cl > 1) cluster_arrive();
  const int nt = g * C;                                   // tiles of the chain
  const int most = (L * C + cl - 1) / cl;                 // of a CTA
  float2* warp_s = reinterpret_cast<float2*>(dyn_s);      // [most][NW] warp sums of this CTA's tiles
  float2* tile_s = warp_s + (size_t)most * NW;            // [L C] the chain's tiles (first CTA)
  float4* g_s = dyn_s + ((size_t)most * NW + L * C + 1) / 2;   // the slice's noise
  const RowSlice sl = cluster_slice(A.d, cl, rank);
  stream_tiles<T, ROWS, VPT, NB>(A, (int64_t)b * L, rank, cl, nt, most, warp_s,
                                 [&] { finish_ahead<HOLD>(A, b, rank, sl, g_s, fs); });
  __syncthreads();
  if (cl > 1) cluster_wait();
  send_tiles(warp_s, rank, cl, nt, tile_s);
  if (cl > 1) cluster_sync();
  else __syncthreads();
  finish_cluster<T, VEC4, HOLD, kK1Threads>(A, b, cl, rank, tile_s, sl, g_s, fs);
}

// Threads of k_finish_long: 512 where every CTA has an SM to itself, else 256.
constexpr int kLongThreads = 512, kLongThreadsMany = 256;
constexpr int64_t kLongPairGroups = 8192;   // see launch_finish_long

// The end of a call whose window k_tiles streams, for rows too long for one finishing CTA
// (k_finish): a cluster per chain.  Its first CTA reads the chain's partials with all its
// threads (the tags tell this call's; a stale one, or a fresh set, makes it wait for k_tiles)
// and frees their slots; the rest is k_chain's.  (stage = 0: sums of more tiles than shared memory
// holds are read by its first warp.)
template <typename T, bool VEC4, int HOLD, int NT>
__global__ void __launch_bounds__(NT) k_finish_long(VerifyArgs A, int cl, int stage) {
  extern __shared__ float4 dyn_s[];
  __shared__ FinishShared fs;
  const int L = A.S.L, C = A.S.C;
  const int b = blockIdx.x / cl;
  const int rank = cl > 1 ? (int)cluster_rank() : 0;
  const int g = A.S.L_eff ? max(0, min(A.S.L_eff[b], L)) : L;
  griddep_launch_dependents();
  if (g == 0) {
    finish_inactive(A, b, rank);
    return;
  }
  if (cl > 1) cluster_arrive();
  float2* tile_s = stage ? reinterpret_cast<float2*>(dyn_s) : nullptr;   // [L C]
  float4* g_s = dyn_s + (stage ? (L * C + 1) / 2 : 0);
  const RowSlice sl = cluster_slice(A.d, cl, rank);
  if (rank == 0 && !stage) griddep_wait();                // warp 0 reads the partials itself
  if (rank == 0 && stage) {
    uint64_t* const p = A.S.tpart + 2 * ((int64_t)b * L * C);
    auto fetch = [&](bool check) {
      int stale = check && A.S.fresh_set;   // any tag may be in its slots
#pragma unroll 4
      for (int t = threadIdx.x; t < g * C; t += NT) {
        const ulonglong2 v = slot_read(p + 2 * t);
        if (check && !slot_holds(v, A.S.tag)) stale = 1;
        tile_s[t] = make_float2(__uint_as_float((uint32_t)v.x), __uint_as_float((uint32_t)v.y));
      }
      return __syncthreads_or(stale);
    };
    if (fetch(true)) {
      griddep_wait();
      (void)fetch(false);
    }
    // by the warps that the scan does not wait for
    constexpr int kFirst = 32 * kMaxScanners;
    if (threadIdx.x >= kFirst) slots_free(p, (int)threadIdx.x - kFirst, NT - kFirst, g * C);
  }
  if (cl > 1) cluster_wait();
  finish_ahead<HOLD>(A, b, rank, sl, g_s, fs);
  finish_cluster<T, VEC4, HOLD, NT>(A, b, cl, rank, tile_s, sl, g_s, fs);
  if (rank == 0 && !stage) {
    __syncthreads();
    slots_free(A.S.tpart + 2 * ((int64_t)b * L * C), threadIdx.x, NT, g * C);
  }
}

// ---------------------------------------------------------------- log ratios alone
// One cluster of CTAs per row (chain b, step j): its tiles' sums meet in the first CTA, which
// adds them in tile order (as scan_load does, so that the ratios equal a whole call's) and
// writes ell_j and |Delta_j|.  Bound by HBM for long rows (64 chains x 16 steps x 16384 bf16
// elements, 100.7 MB: 26.7 us with ticket counters and their memset, 18.5 now), by the CTAs'
// latency for many short ones, hence six per SM where a row is one small tile (471 x 18 rows
// of 576 bf16 elements: 51 us with three per SM, 24.5 with six).
template <typename T, int ROWS, int VPT>
__global__ void __launch_bounds__(kK1Threads, VPT == 1 ? 6 : 3) k_ratios(VerifyArgs A, int cl, int span) {
  constexpr int NW = kK1Threads / 32;
  constexpr int NB = VPT == 1 ? 1 : tiles_in_flight(VPT);   // rows of one such tile are a tile each
  extern __shared__ float4 dyn_s[];
  const int L = A.S.L, C = A.S.C;
  const int64_t row = blockIdx.x / cl;
  const int b = (int)(row / L), j = (int)(row - (int64_t)b * L);
  const int rank = cl > 1 ? (int)cluster_rank() : 0;
  const int tid = threadIdx.x;
  griddep_wait();                  // as in k_chain
  griddep_launch_dependents();
  const int g = A.S.L_eff ? max(0, min(A.S.L_eff[b], L)) : L;
  if (j >= g) {                    // past the window: zeros
    if (rank == 0 && tid == 0) {
      A.S.ell_out[row] = 0.f;
      A.S.dn_out[row] = 0.f;
    }
    return;
  }
  if (cl > 1) cluster_arrive();
  const int most = (span + cl - 1) / cl;
  float2* warp_s = reinterpret_cast<float2*>(dyn_s);   // [most][NW]
  float2* tile_s = warp_s + (size_t)most * NW;         // [span] (first CTA)
  float a1 = 0.f, a2 = 0.f;
  for (int c0 = 0; c0 < C; c0 += span) {               // one span for any but enormous rows
    const int n = min(span, C - c0);
    stream_tiles<T, ROWS, VPT, NB>(A, (int64_t)b * L, j * C + c0 + rank, cl, j * C + c0 + n, most, warp_s, [] {});
    __syncthreads();
    if (cl > 1 && c0 == 0) cluster_wait();
    send_tiles(warp_s, rank, cl, n, tile_s);
    if (cl > 1) cluster_sync();
    else __syncthreads();
    if (rank == 0 && tid == 0) {
      for (int c = 0; c < n; ++c) {
        a1 += tile_s[c].x;
        a2 += tile_s[c].y;
      }
    }
    if (c0 + span < C) {           // tile_s is read before the next span's sums arrive
      if (cl > 1) cluster_sync();
      else __syncthreads();
    }
  }
  if (rank == 0 && tid == 0) {
    ScanRegs R;
    (void)scan_step(R, 0, a1, a2, A.S.sigma[(int64_t)b * A.S.sstride + j]);
    A.S.ell_out[row] = R.ell[0];
    A.S.dn_out[row] = R.dn[0];
  }
}

// ---------------------------------------------------------------- host side
constexpr size_t kChainSmemMax = 100 * 1024;   // kChainPerSm CTAs per SM
constexpr size_t kFinishSmemMax = 200 * 1024;  // k_finish_long: one

// Clusters of cl CTAs that the device holds at once, at per_sm CTAs per SM (a cluster needs
// its places within one GPC, so that some are left over).  Asked once per device.
static __global__ void __launch_bounds__(kK1Threads) k_place() {}
static int max_clusters(int cl, int per_sm) {
  static std::atomic<int> cache[64][9][3];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  std::atomic<int>& slot = cache[dev][cl][per_sm];
  int n = slot.load(std::memory_order_relaxed);
  if (n == 0) {
    // shared memory that only per_sm CTAs of an SM get
    const size_t smem = per_sm == 1 ? kFinishSmemMax : kChainSmemMax;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cl);
    cfg.blockDim = dim3(kK1Threads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaFuncSetAttribute(k_place, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFinishSmemMax) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, k_place, &cfg) != cudaSuccess || n < 1) {
      cudaGetLastError();
      return 0;
    }
    slot.store(n, std::memory_order_relaxed);
  }
  return n;
}


// CTAs per chain, or 0 when the call does not fit: as many (up to 8) as the chain has tiles
// and as leave every chain's cluster a place at once, kChainPerSm CTAs per SM, when each reads
// at most kChainBytes.  (A second wave of clusters doubles a call's time: B = 49, L = 7,
// d = 6336 took 25 us with six CTAs per chain, of which 46 fit.)  With more to read, k_tiles
// streams faster than the extra launch costs: 256 chains x 8 steps x 3072 fp32 elements, 288 KB
// a CTA, 24.5 us here and 25.2 split; 200 x 8 x 4096, 384 KB, 27.7 and 26.3; 100 x 8 x 10000,
// 313 KB, 34.6 and 29.0; 56 x 17 x 63432, 2.5 MB, 164 and 138.
constexpr int64_t kChainBytes = 300 * 1024;
// And at most 16 groups of four of the row for a thread: longer rows, of short windows, are
// finished by more threads (88 x 1 x 96920 fp32 112 us here, 62 by k_finish_long).
constexpr int64_t kChainGroups = 16 * (kK1Threads - 32);
constexpr size_t kChainTiles = 16;   // tiles of a CTA, of rows read as vectors
static int chain_cluster(int B, int L, int C, int64_t d, int es) {
  const int sms = sm_count();
  if (B > kChainPerSm * sms) return 0;
  int cl = std::min(8, L * C);
  while (cl > 1 && B > max_clusters(cl, kChainPerSm)) --cl;
  const int64_t bytes = 3 * (int64_t)L * d * es / cl;
  return bytes <= kChainBytes ? cl : 0;
}

template <typename Kern, typename... More>
static cudaError_t launch_cluster(Kern kern, const VerifyArgs& A, unsigned clusters, int cl, size_t smem, cudaStream_t s,
                                  unsigned threads, More... more) {
  if (smem > 40 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFinishSmemMax);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(clusters * (unsigned)cl);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  int n = 0;
  if (cl > 1) {
    at[n].id = cudaLaunchAttributeClusterDimension;
    at[n].val.clusterDim.x = (unsigned)cl;
    at[n].val.clusterDim.y = 1;
    at[n].val.clusterDim.z = 1;
    ++n;
  }
  {
    at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
  }
  cfg.attrs = at;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kern, A, cl, more...);
}

template <typename T, int HOLD>
static cudaError_t launch_t(const VerifyArgs& A, int B, int cl, int vpt, int rows, size_t smem, cudaStream_t s) {
  if (rows == kRowsElement)
    return launch_cluster(k_chain<T, kRowsElement, 1, false, HOLD>, A, B, cl, smem, s, kK1Threads);
#define SDV_VPT(V)                                                                                                     \
  return rows == kRowsAligned ? launch_cluster(k_chain<T, kRowsAligned, V, true, HOLD>, A, B, cl, smem, s, kK1Threads)  \
                              : launch_cluster(k_chain<T, kRowsUnaligned, V, false, HOLD>, A, B, cl, smem, s, kK1Threads)
  // rows whose noise outgrows the registers' share are long enough for full-sized tiles (bf16
  // tiles have at most two vectors)
  constexpr bool kSmall = HOLD == kHoldAll;
  if constexpr (kSmall) {
    if (vpt == 1) return launch_cluster(k_chain<T, kRowsAligned, 1, true, HOLD>, A, B, cl, smem, s, kK1Threads);
  }
  if constexpr (kSmall || sizeof(T) == 2) {
    if (vpt == 2) { SDV_VPT(2); }
  }
  if constexpr (sizeof(T) == 4) {
    if constexpr (kSmall) {
      if (vpt == 3) { SDV_VPT(3); }
    }
    if (vpt == 4) { SDV_VPT(4); }
  }
  return cudaErrorInvalidValue;   // not reached: ws_layout's tiles for these rows are listed
#undef SDV_VPT
}

template <typename T>
cudaError_t launch_chain(const VerifyArgs& A, int B, int L, int vpt, int rows, bool vec4, cudaStream_t s, bool* taken) {
  *taken = false;
  const int C = A.S.C;
  const int cl = chain_cluster(B, L, C, A.d, (int)sizeof(T));
  if (cl == 0 || (rows == kRowsAligned && !vec4)) return cudaSuccess;
  // one-vector tiles of rows off vector boundaries stream better spread over all SMs: 160 chains x
  // 25 steps x 1501 bf16 elements 38.0 us here, 23.4 by k_tiles, 4 x 16 x 1501 12.8 and 12.5
  // (but 300 x 12 x 901 fp32 19.3 and 20.6)
  if (rows == kRowsUnaligned && vpt == 1) return cudaSuccess;
  const size_t most = ((size_t)L * C + cl - 1) / cl;
  // nor many tiles of whole vectors one batch after another: 160 x 25 x 1024 bf16 elements 27.1 us
  // here, 21.0 by k_tiles, 160 x 25 x 512 fp32 22.9 and 19.9; twelve tiles, 300 x 12 x 1024 fp32,
  // 19.2 and 21.0; read by element, 160 x 25 x 256 fp32, 17.1 and 20.1
  if (rows == kRowsAligned && most > kChainTiles) return cudaSuccess;
  const int64_t ng = (A.d + 3) / 4, per = (ng + cl - 1) / cl;
  const size_t smem = 16 * ((most * (kK1Threads / 32) + (size_t)L * C + 1) / 2) + sizeof(float4) * (size_t)per;
  if (smem > kChainSmemMax || per > kChainGroups) return cudaSuccess;
  *taken = true;
  return per <= (int64_t)kOwn * (kK1Threads - 32) ? launch_t<T, kHoldAll>(A, B, cl, vpt, rows, smem, s)
                                                  : launch_t<T, kHoldNoise>(A, B, cl, vpt, rows, smem, s);
}

template <typename T, bool VEC4, int NT>
static cudaError_t launch_long_t(const VerifyArgs& A, int B, int cl, size_t tiles, size_t noise, cudaStream_t s) {
  const int stage = tiles <= kFinishSmemMax / 2;
  if (!stage) tiles = 0;
  // many CTAs: two per SM, as far as the noise allows
  if (A.S.residual_kind != SDV_RESIDUAL_REFLECTION &&   // which draws noise only where delta = 0
      tiles + noise <= (NT == kLongThreads ? kFinishSmemMax : kChainSmemMax))
    return launch_cluster(k_finish_long<T, VEC4, kHoldNoise, NT>, A, B, cl, tiles + noise, s, NT, stage);
  return launch_cluster(k_finish_long<T, VEC4, kHoldNothing, NT>, A, B, cl, tiles, s, NT, stage);
}

template <typename T>
cudaError_t launch_finish_long(const VerifyArgs& A, int B, int L, bool vec4, cudaStream_t s) {
  // Few chains: as many CTAs per chain, of 512 threads, as leave every cluster a place at once,
  // one CTA per SM.  Where that leaves a chain one CTA, or too little shared memory for its
  // noise, four CTAs of 256 threads, two to an SM, so that the last wave of them is short; or
  // eight, where only those hold the noise.  (88 chains of one step of 96919 bf16 elements: 66 us
  // with eight, 68 with four, 124 with one of 512 threads; 150 x 1 x 50000 fp32 56 with four, 69
  // with one; but 56 x 17 x 63432 140 with two of 512 threads, 168 with four of 256.)  Two for at
  // least a chain per SM of rows up to kLongPairGroups groups: every CTA of a chain holds its place
  // through the chain's scan and U-draw, and there are more CTAs than places.  (Two against four:
  // 512 chains of one step of 16388 fp32 elements 66 and 84 us, 505 x 1 x 30000 101 and 112, 152 x
  // 1 x 30000 39 and 40; but 100 x 1 x 30000 36 and 30, 512 x 1 x 36000 133 and 129, 250 x 1 x
  // 50000 106 and 88.)
  size_t tiles = 16 * (((size_t)L * A.S.C + 1) / 2);
  const auto noise = [&](int c) { return sizeof(float4) * (size_t)(((A.d + 3) / 4 + c - 1) / c); };
  const auto fits = [&](int c, size_t most) { return (tiles <= kFinishSmemMax / 2 ? tiles : 0) + noise(c) <= most; };
  int cl = B <= 8 ? 8 : 6;
  while (cl > 1 && B > max_clusters(cl, 1)) --cl;
  if (cl > 1 && (fits(cl, kFinishSmemMax) || !fits(8, kChainSmemMax)))
    return vec4 ? launch_long_t<T, true, kLongThreads>(A, B, cl, tiles, noise(cl), s)
                : launch_long_t<T, false, kLongThreads>(A, B, cl, tiles, noise(cl), s);
  if (B >= sm_count() && (A.d + 3) / 4 <= kLongPairGroups && fits(2, kChainSmemMax)) cl = 2;
  else cl = fits(4, kChainSmemMax) || !fits(8, kChainSmemMax) ? 4 : 8;
  return vec4 ? launch_long_t<T, true, kLongThreadsMany>(A, B, cl, tiles, noise(cl), s)
              : launch_long_t<T, false, kLongThreadsMany>(A, B, cl, tiles, noise(cl), s);
}

template <typename T>
static cudaError_t launch_ratios_t(const VerifyArgs& A, unsigned n, int cl, int span, int vpt, int rows, size_t smem,
                                   cudaStream_t s) {
  if (rows == kRowsElement) return launch_cluster(k_ratios<T, kRowsElement, 1>, A, n, cl, smem, s, kK1Threads, span);
#define SDV_VPT(V)                                                                                               \
  return rows == kRowsAligned ? launch_cluster(k_ratios<T, kRowsAligned, V>, A, n, cl, smem, s, kK1Threads, span)      \
                              : launch_cluster(k_ratios<T, kRowsUnaligned, V>, A, n, cl, smem, s, kK1Threads, span)
  if (vpt == 1) { SDV_VPT(1); }
  if (vpt == 2) { SDV_VPT(2); }
  if constexpr (sizeof(T) == 4) {
    if (vpt == 3) { SDV_VPT(3); }
    SDV_VPT(4);
  }
  return cudaErrorInvalidValue;
#undef SDV_VPT
}

template <typename T>
cudaError_t launch_ratios(const VerifyArgs& A, int B, int L, int vpt, int rows, cudaStream_t s) {
  const int C = A.S.C;
  const int64_t n = (int64_t)B * L;
  int cl = 1;
  while (cl < 8 && n * cl * 2 <= 3 * (int64_t)sm_count() && cl * 2 <= C) cl *= 2;
  const int span = std::min(C, 256 * cl);
  const size_t smem = sizeof(float2) * ((size_t)((span + cl - 1) / cl) * (kK1Threads / 32) + (size_t)span);
  return launch_ratios_t<T>(A, (unsigned)n, cl, span, vpt, rows, smem, s);
}

}  // namespace sdv
