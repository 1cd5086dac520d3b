// sdv_verify.cu - verification step of speculative diffusion sampling on sm_103a.
//
// A verification call runs one of two ways (enqueue_verify):
//   * a plain call of few chains as ONE kernel, k_chain (sdv_chain.cuh);
//   * many chains, few chains of long rows, and pipelined calls as two: k_tiles streams one
//     tile (chain b, step j, chunk c) of x, m^q and m^p per CTA, once, with 16-byte loads,
//     and reduces S1 = sum (x - m^p)(m^p - m^q) and S2 = sum (m^p - m^q)^2 (App. "Density
//     ratio calculations": Z^T Delta = S1/sigma^2, |Delta|^2 = S2/sigma^2), each partial
//     stored with the call's tag; then k_finish takes each chain from its partials to its
//     output: ell_j and |Delta_j|, the coins, sample or block acceptance (Algorithms
//     token-/block-verification), U (Algorithm u-sample) and the row (Algorithm
//     decomposition-res: y = m^q + sigma (U e + G - e e^T G); or reflect-res, the bonus
//     step, or the last accepted draft).  Rows too long for one CTA are finished by a
//     cluster of them, k_finish_long (sdv_chain.cuh).
// Both sum a tile, and a row's tiles, in the same order, so that the log ratios do not
// depend on the way.
#include <cuda_runtime.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

#include "sdv_device.cuh"
#include "sdv_host.h"
#include "sdv_scan.cuh"
#include "sdv_sets.h"
#include "sdv_tiles.cuh"
#include "sdv_finish.cuh"
#include "sdv_chain.h"

namespace sdv {

// ---------------------------------------------------------------- stream and finish
// The stream: one tile per CTA; its (S1, S2) is stored with the call's tag.  Bound by HBM
// (8 rows of 3072 floats for 256 chains, 75.5 MB, in about 11 us alone, 6.9 TB/s).  (Two or
// four software-pipelined tiles per CTA measured slower: 17.4 / 20.1 us against 16.5 us per
// pipelined pixel call.  Drawing the residual's noise of long rows behind the loads, into y,
// shortened their finishing but the whole call grew, 16 x 32 x 196608 fp32 198 -> 211 us.)
template <typename T, int ROWS, int VPT>
__global__ void __launch_bounds__(kK1Threads, tile_min_blocks(VPT)) k_tiles(VerifyArgs A) {
  __shared__ float2 red[kK1Threads / 32];
  const int L = A.S.L;
  const int C = A.S.C;
  const int64_t tile = blockIdx.x;
  const int64_t r = tile / C;
  const int c = (int)(tile - r * C);
  const int b = (int)(r / L), j = (int)(r - (int64_t)b * L);
  // a plain call's stream starts only when the work before it has completed (its launch, and
  // its CTAs' start, then overlap the end of that work)
  if (A.serial) griddep_wait();
  const int g = A.S.L_eff ? max(0, min(A.S.L_eff[b], L)) : L;
  if (j < g) {  // CTA-uniform
    const int64_t e0 = (int64_t)c * A.chunk;
    const int64_t e1 = min(e0 + A.chunk, A.d);
    // whether this CTA's slot is free, asked by thread 0 once its tile loads are in flight
    // (the acquire orders only what follows it)
    uint64_t* const slot = A.S.tpart + 2 * tile;
    bool is_free = false;
    float2 sm;
    if (ROWS == kRowsAligned) {
      TileBuf<VPT> B;
      tile_issue<T, VPT>((const T*)A.x, (const T*)A.mq, (const T*)A.mp, r * A.d, e0, e1, B);
      if (threadIdx.x == 0) is_free = slot_is_free(slot);
      sm = tile_fma<T, VPT>(B);
    } else if (ROWS == kRowsUnaligned) {
      TileBuf<VPT> B;
      EdgeBuf E;
      unaligned_issue<T, VPT>((const T*)A.x, (const T*)A.mq, (const T*)A.mp, r * A.d, A.d, c, C, B, E);
      if (threadIdx.x == 0) is_free = slot_is_free(slot);
      sm = unaligned_fma<T, VPT>(B, E);
    } else {
      if (threadIdx.x == 0) is_free = slot_is_free(slot);
      sm = tile_sums<T>((const T*)A.x, (const T*)A.mq, (const T*)A.mp, r * A.d, e0, e1);
    }
    const float2 t = block_sum2<kK1Threads>(sm.x, sm.y, red);
    if (threadIdx.x == 0) {
      // the slot's partial has not been read yet by the call that wrote it (which may
      // still be finishing, since calls overlap), or a call of another layout may have
      // written here: wait for the previous kernel, whose completion implies every
      // earlier call's (in practice the slot was read long ago)
      if (A.S.fresh_set || !is_free) griddep_wait();
      slot_store(slot, A.S.tag, t);
    }
  }
  if (blockIdx.x == 0) {
    // CTA 0 ties this grid's completion to the previous kernel's (so the next k_finish,
    // which writes its outputs after this grid has completed, writes after the previous
    // call's k_finish); it triggers first, its own tile done, so that k_finish can start
    __syncthreads();
    griddep_launch_dependents();
    if (threadIdx.x == 0) griddep_wait();
  }
}

// One CTA per chain: the CTA triggers its dependents at once (the next call's stream
// writes the other set of partials); warp 0 reads the chain's partials (k_finish starts
// only after every k_tiles CTA has stored its partial and exited or triggered; the tags
// confirm that each one read is this call's, else the warp waits for k_tiles to
// complete and reads them again) and scans the chain, while the other warps draw the
// residual's G into shared memory (dynamic, (d + 3)/4 float4) and warp 1 frees the
// chain's slots for the next call that writes this set; then warp 0 draws U while the
// others reduce delta^T G over the rejected row, and they write y.  Every output is written
// after griddep_wait.  Bound by the latency of one warp's evaluations (scan 4-5 us, U 4 us);
// what does not depend on them runs beside them: with 64 threads, the noise before the scan's
// end and delta^T G after the U-draw, one chain took 17-19 us.  128 threads for rows of up to
// 4096 elements (pipelined pixel calls, eight in a graph: 158 -> 143 us), 256 beyond.
template <typename T, bool VEC4, int NT>
__global__ void __launch_bounds__(NT) k_finish(VerifyArgs A) {
  __shared__ FinishShared fs;
  __shared__ float ell_s[SDV_MAX_L], dn_s[SDV_MAX_L];
  __shared__ float u_s;
  __shared__ int gw_s;             // the chain's window length (tiles written this call)
  extern __shared__ float4 g_s[];  // the residual's G, drawn once
  const int b = blockIdx.x;
  const int L = A.S.L;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const RowSlice sl{0, (A.d + 3) / 4, (int)threadIdx.x - 32, NT - 32};
  const uint64_t seed = seed_of(A.S);
  // 256 threads for long rows: few CTAs, their loads bound by latency (eight pipelined latent
  // calls 192 us with sweeps of four groups, 181 with eight; pixel rows 143 against 146)
  constexpr int HOLD = NT >= 256 && VEC4 ? kHoldNoiseFar : kHoldNoise;
  RowRegs<own_groups(HOLD)> rg;
  // the next kernel (the next call's stream) may start now: it writes the other set of
  // partials, and a slot of this set only once this call has read it
  griddep_launch_dependents();
  ScanOut so;
  OneWarp co;
  if (warp == 0) {
    float leta[2];
    scan_coins(A.S, b, leta);
    if (A.S.fresh_set) griddep_wait();   // any tag may be in its slots
    ScanRegs R = scan_load(A.S, b);
    if (R.stale) {
      // a partial of this call is not visible yet (k_finish starts once every k_tiles
      // CTA has stored its partial and exited or triggered, so in practice they all
      // are): wait for k_tiles to complete, which makes its writes visible, and read
      // them again
      griddep_wait();
      R = scan_load(A.S, b, false);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if (lane + 32 * q < L) {
        ell_s[lane + 32 * q] = R.ell[q];
        dn_s[lane + 32 * q] = R.dn[q];
      }
    }
    if (lane == 0) gw_s = R.g;
    __syncwarp();
    // warp 1 may free the slots (named barrier: this warp only arrives)
    asm volatile("bar.arrive 1, 64;" ::: "memory");
    so = scan_decide(A.S, b, R, leta, co);
    if (lane == 0) fs.cs = so.cs;
  } else {
    if (warp == 1) {
      asm volatile("bar.sync 1, 64;" ::: "memory");
      slots_free(A.S.tpart + 2 * ((int64_t)b * L * A.S.C), lane, 32, gw_s * A.S.C);
    }
    draw_noise<HOLD>(seed, b, sl, g_s);
  }
  __syncthreads();
  ChainState cs = fs.cs;
  float coef = 0.f;
  if (cs.kind == kKindResid) {
    if (warp == 0) {
      const uint32_t wbits = philox_block(seed, (uint32_t)b, 0u, kStreamUSample, 0u).x;
      uint32_t st = cs.status;
      const UParams Q = so.have_P ? so.P : usample_setup(cs.dnorm, fminf(cs.la_res, 0.f), co);
      cs.U = usample_warp(Q, wbits, &st, co);
      cs.status = st;
      if (lane == 0) u_s = cs.U;
    } else {
      float dot = slice_dot<T, VEC4, HOLD>((const T*)A.mq, (const T*)A.mp, L, A.d, seed, b, cs, sl, rg, g_s);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
      if (lane == 0) fs.dot[warp] = dot;
    }
    __syncthreads();
    float t = fs.dot[1];
#pragma unroll
    for (int w = 2; w < NT / 32; ++w) t += fs.dot[w];
    coef = u_s - t * cs.inv_norm;  // U - e^T G
  }
  // outputs: after k_tiles has completed, and with it the previous call (see k_tiles)
  griddep_wait();
  for (int i = threadIdx.x; i < L; i += NT) {
    if (A.S.ell_out) A.S.ell_out[(int64_t)b * L + i] = ell_s[i];
    if (A.S.dn_out) A.S.dn_out[(int64_t)b * L + i] = dn_s[i];
  }
  if (threadIdx.x == 0) {
    scan_write_chain(A.S, b, cs);
    report_chain(A.S, b, cs, true);
  }
  if (warp > 0)
    slice_write<T, VEC4, HOLD>((const T*)A.x, (const T*)A.mq, (const T*)A.mp, (const T*)A.mq_bonus, A.sigma_bonus, L,
                                A.d, seed, b, cs, coef, (T*)A.y, sl, rg, g_s);
}

// ---------------------------------------------------------------- acceptance scan only
__global__ void __launch_bounds__(kK2Threads) k_scan(ScanArgs A) {
  const int b = blockIdx.x * (kK2Threads / 32) + (threadIdx.x >> 5);
  if (b >= A.B) return;  // warp-uniform
  (void)scan_warp(A, b);
}

// ---------------------------------------------------------------- stand-alone pieces
__global__ void __launch_bounds__(kK2Threads)
k_usample(const float* __restrict__ D, const float* __restrict__ la, const uint32_t* __restrict__ w,
          int n, float* __restrict__ U, uint32_t* __restrict__ st) {
  const int i = blockIdx.x * (kK2Threads / 32) + (threadIdx.x >> 5);  // one warp per item
  if (i >= n) return;
  const float Dn = D[i];
  float l = la[i];
  uint32_t status = 0u;
  float u = NAN;
  if (isnan(Dn) || isnan(l)) {
    status = 2u;
  } else if (!(Dn > 0.f) || isinf(Dn)) {
    status = 1u;
  } else {
    l = fminf(l, 0.f);
    OneWarp co;
    u = usample_warp(usample_setup(Dn, l, co), w[i], &status, co);
  }
  if ((threadIdx.x & 31) == 0) {
    U[i] = u;
    if (st) st[i] = status;
  }
}

__global__ void k_philox(const uint4* __restrict__ ctr, uint64_t seed, int n, uint4* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = philox4x32_10(ctr[i], (uint32_t)seed, (uint32_t)(seed >> 32));
}

__global__ void k_special(int which, const float* __restrict__ z, int n, float* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float v = z[i];
  out[i] = which == 0 ? erfcx_any(v) : (which == 1 ? log_ndtr_g(v).x : (v < -4.0f ? gprime_cf(v) : gprime_ex(v)));
}

__global__ void k_normals(uint64_t seed, int B, int64_t d, uint32_t stream, uint32_t sub, float* out) {
  const int64_t ng = (d + 3) / 4;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)B * ng) return;
  const int b = (int)(t / ng);
  const int64_t gi = t - (int64_t)b * ng;
  const float4 G = normals4(seed, (uint32_t)b, (uint32_t)gi, stream, sub);
  const float g[4] = {G.x, G.y, G.z, G.w};
  for (int k = 0; k < 4; ++k)
    if (4 * gi + k < d) out[(int64_t)b * d + 4 * gi + k] = g[k];
}

// ---------------------------------------------------------------- host side
static thread_local int g_last_cuda_error = 0;

void set_last_cuda_error(int err) { g_last_cuda_error = err; }

int sm_count() {
  static std::atomic<int> cache[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 152;
  if (cache[dev].load() == 0) {
    int n = 0;
    cache[dev].store((cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0) ? n : 152);
  }
  return cache[dev].load();
}


static int check_launch() {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    g_last_cuda_error = (int)e;
    return SDV_ECUDA;
  }
  return SDV_OK;
}

static bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

// ---- per-thread timing ring (sdv_timing_enable / sdv_timing_read).  Records use
// cudaEventRecordExternal under stream capture, so that they become event-record
// nodes of the graph (a plain record there only expresses a dependency).
struct TimingRing {
  std::vector<cudaEvent_t> ev;  // slots x 3
  int slots = 0;
  long long next = 0;   // recorded calls
  int stride = 1;       // record one call in `stride`
  long long calls = 0;  // calls seen while enabled
};
static thread_local TimingRing g_timing;

static void timing_destroy() {
  for (cudaEvent_t e : g_timing.ev) cudaEventDestroy(e);
  g_timing.ev.clear();
  g_timing.slots = 0;
  g_timing.next = 0;
  g_timing.calls = 0;
}

static cudaEvent_t* timing_slot() {
  if (g_timing.slots == 0) return nullptr;
  if (g_timing.calls++ % g_timing.stride != 0) return nullptr;
  const int s = (int)(g_timing.next % g_timing.slots);
  ++g_timing.next;
  return &g_timing.ev[3 * (size_t)s];
}

static void timing_record(cudaEvent_t e, cudaStream_t s) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  cudaStreamIsCapturing(s, &cap);
  if (cap == cudaStreamCaptureStatusActive) cudaEventRecordWithFlags(e, s, cudaEventRecordExternal);
  else cudaEventRecord(e, s);
}

WsLayout ws_layout(int B, int L, int64_t d, int dtype) {
  WsLayout w{};
  const int es = dtype == SDV_BF16 ? 2 : 4;
  // vectors per thread: the smallest sweep that covers a row, capped at kK1Vpt (at 2
  // for bf16 rows, whose 16-byte vectors hold 8 elements: the 40-register tiles leave
  // room on an SM for the previous pipelined call's 256-thread finishing CTA; latent
  // rows 19.5 -> 19.0 us per pipelined call), so that common row lengths run whole,
  // unguarded sweeps
  const int64_t vec_per_row = (d * es + 15) / 16;
  const int64_t vpt_cap = es == 2 ? 2 : kK1Vpt;
  w.vpt1 = (int)std::min<int64_t>(vpt_cap, std::max<int64_t>(1, (vec_per_row + kK1Threads - 1) / kK1Threads));
  w.chunk1 = (int64_t)kK1Threads * w.vpt1 * (16 / es);
  w.C1 = (int)((d + w.chunk1 - 1) / w.chunk1);
  auto up = [](size_t v) { return (v + 255) & ~(size_t)255; };
  size_t off = 0;
  w.part_off = off;
  const size_t slots = (size_t)B * L * w.C1;
  // 4 bytes a slot are not used (see below)
  w.part_set_bytes = up(up(2 * sizeof(uint64_t) * slots) + sizeof(uint32_t) * slots);
  off = up(off + 2 * w.part_set_bytes);
  // Not used since slots are freed in place and finishing keeps its state on chip: a tag per
  // slot, a counter and a state per chain, and a sum per 1024 to 4096 elements of a row (about
  // 1024 in all).  The size stays, so that sizes that callers have stored, and sdv_verify_noalloc's limit, mean the same calls.
  int64_t chunk = 1024;
  while (chunk < 4096 && (int64_t)B * ((d + chunk - 1) / chunk) > 1024) chunk *= 2;
  off = up(off + 4 * (size_t)B);
  off = up(off + 48 * (size_t)B);
  off = up(off + 4 * (size_t)B * (size_t)((d + chunk - 1) / chunk));
  w.total = off;
  return w;
}

static int validate_window(const void* x, const void* mq, const void* mp, const float* sigma,
                           int64_t sstride, int B, int L, int64_t d, int dtype) {
  if (!x || !mq || !mp || !sigma) return SDV_EINVAL;
  if (B < 1 || L < 1 || L > SDV_MAX_L || d < 1) return SDV_EINVAL;
  if (dtype != SDV_F32 && dtype != SDV_BF16) return SDV_EINVAL;
  if (sstride < 0) return SDV_EINVAL;
  if ((double)B * L * (double)d > 9.0e18) return SDV_EINVAL;
  if (B > (1 << 30)) return SDV_EINVAL;
  const size_t es = dtype == SDV_BF16 ? 2 : 4;
  if (!aligned(x, es) || !aligned(mq, es) || !aligned(mp, es) || !aligned(sigma, 4)) return SDV_EALIGN;
  return SDV_OK;
}

// A launch through cudaLaunchKernelEx: dynamic shared memory (raising the kernel's limit when
// it passes 48 KB, to what the longest rows take: all host threads share the limit, so that a
// call must not set it to its own size) and programmatic stream serialisation (the kernels
// wait for the work before them where they need it).
constexpr size_t kLaunchSmemMax = sizeof(float4) * (size_t)kPipeMaxGroups;
template <typename Kern>
static cudaError_t launch_ex(Kern kern, unsigned grid, unsigned threads, size_t smem, const VerifyArgs& A,
                             cudaStream_t s) {
  // the kernels' static shared memory counts toward the 48 KB that need no permission
  if (smem > 40 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLaunchSmemMax);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, A);
}

template <typename T>
static cudaError_t launch_tiles(const VerifyArgs& A, int B, int L, int vpt, int rows, cudaStream_t s) {
  const unsigned tiles = (unsigned)((int64_t)B * L * A.S.C);
  if (rows == kRowsElement) return launch_ex(k_tiles<T, kRowsElement, 1>, tiles, kK1Threads, 0, A, s);
#define SDV_TILES(V)                                                                                          \
  return rows == kRowsAligned ? launch_ex(k_tiles<T, kRowsAligned, V>, tiles, kK1Threads, 0, A, s)    \
                              : launch_ex(k_tiles<T, kRowsUnaligned, V>, tiles, kK1Threads, 0, A, s)
  if (vpt == 1) { SDV_TILES(1); }
  if (vpt == 2) { SDV_TILES(2); }
  if constexpr (sizeof(T) == 4) {
    if (vpt == 3) { SDV_TILES(3); }
    SDV_TILES(4);
  }
  return cudaErrorInvalidValue;   // bf16 tiles have at most two vectors (ws_layout)
#undef SDV_TILES
}

// k_finish: kFinishThreads per chain (kFinishThreadsMany with many chains of short rows, whose
// latencies overlap, so that slots count more: 2000 chains x 6 steps x 512 bf16 elements, pipelined,
// 49.7 us a call with 128 threads, 46.3 with 64; but 512 x 8 x 3072 fp32 32.5 against 38.7), or kFinishWideThreads for rows longer than
// kFinishMaxGroups groups of four, whose residual passes and noise fewer threads would take
// too long over.
template <typename T>
static cudaError_t launch_finish(const VerifyArgs& A, int B, bool vec4, cudaStream_t s) {
  const int64_t ng = (A.d + 3) / 4;
  const size_t smem = sizeof(float4) * (size_t)ng;
  if (ng > kFinishMaxGroups) {
    if (vec4) return launch_ex(k_finish<T, true, kFinishWideThreads>, (unsigned)B, kFinishWideThreads, smem, A, s);
    return launch_ex(k_finish<T, false, kFinishWideThreads>, (unsigned)B, kFinishWideThreads, smem, A, s);
  }
  if (B >= kManyChainMin && ng <= kFinishManyMaxGroups) {
    if (vec4) return launch_ex(k_finish<T, true, kFinishThreadsMany>, (unsigned)B, kFinishThreadsMany, smem, A, s);
    return launch_ex(k_finish<T, false, kFinishThreadsMany>, (unsigned)B, kFinishThreadsMany, smem, A, s);
  }
  if (vec4) return launch_ex(k_finish<T, true, kFinishThreads>, (unsigned)B, kFinishThreads, smem, A, s);
  return launch_ex(k_finish<T, false, kFinishThreads>, (unsigned)B, kFinishThreads, smem, A, s);
}

// The tag of a call's k_tiles partials: a process-wide counter, never 0 (a free slot's),
// so consecutive calls on a workspace never share a tag.  A captured call keeps its tag at
// every replay of its graph; replays run one after another, and each leaves its slots free.
static std::atomic<uint32_t> g_partial_tag{0u};
static uint32_t next_partial_tag() {
  uint32_t t;
  do {
    t = g_partial_tag.fetch_add(1u, std::memory_order_relaxed) + 1u;
  } while (t == 0u);
  return t;
}

static PartialSets g_partial_sets;

// Enqueue the whole step (or, with ratios_only, the log-ratio pass) for validated args.
static int enqueue_verify(const void* x_draft, const void* mu_target, const void* mu_draft,
                          const float* sigma, int64_t sigma_stride_b, int B, int L, int64_t d,
                          int dtype, uint64_t seed, const uint64_t* seed_dev, int mode, const int32_t* L_eff,
                          const void* mu_target_bonus, const float* sigma_bonus,
                          int residual_kind, float omega, int32_t* accepted_len, void* y_out,
                          float* log_ratio_out, float* delta_norm_out, uint32_t* status_out,
                          float* chain_aux_out, bool ratios_only, bool timed, bool overlap,
                          void* workspace, cudaStream_t s) {
  const WsLayout w = ws_layout(B, L, d, dtype);
  char* ws = (char*)workspace;
  VerifyArgs A{};
  A.x = x_draft; A.mq = mu_target; A.mp = mu_draft;
  A.mq_bonus = mu_target_bonus; A.sigma_bonus = sigma_bonus;
  A.d = d; A.serial = !overlap; A.sms = sm_count(); A.chunk = w.chunk1; A.y = y_out;
  ScanArgs& S = A.S;
  S.C = w.C1; S.sigma = sigma; S.sstride = sigma_stride_b;
  S.B = B; S.L = L; S.L_eff = L_eff; S.seed = seed; S.seed_dev = seed_dev; S.mode = mode;
  S.inv_omega2 = 1.0f / (omega * omega); S.residual_kind = residual_kind;
  S.has_bonus = mu_target_bonus != nullptr;
  S.ell_out = log_ratio_out; S.dn_out = delta_norm_out; S.accepted_len = accepted_len;
  S.status_out = status_out; S.aux_out = chain_aux_out;

  cudaEvent_t* tev = (ratios_only || !timed) ? nullptr : timing_slot();
  if (tev) timing_record(tev[0], s);
  const int64_t ng = (d + 3) / 4;
  const bool f32 = dtype == SDV_F32;
  const int64_t V = f32 ? 4 : 8;
  // Rows of at most one element a thread are read by element (160 chains x 25 steps x 92 fp32,
  // plain: 16.7 us, by vectors 22.0), and so are rows that start anywhere within a vector as
  // long as vectors leave many threads idle: 701 fp32 elements 21.9 us against 29.7, but 1001
  // 26.3 against 21.4; 1001 bf16 elements 27.1 against 38.2.
  const bool aligned16 = aligned(x_draft, 16) && aligned(mu_target, 16) && aligned(mu_draft, 16);
  const int rows = !aligned16 || d <= kK1Threads           ? kRowsElement
                   : d % V == 0                            ? kRowsAligned
                   : d <= (f32 ? 3 * kK1Threads : kElementMax) ? kRowsElement
                                                           : kRowsUnaligned;
  const size_t a4 = f32 ? 16 : 8;   // groups of four elements load and store as one vector
  const bool vec4 = d % 4 == 0 && aligned(x_draft, a4) && aligned(mu_target, a4) && aligned(mu_draft, a4) &&
                    (y_out == nullptr || aligned(y_out, a4)) && (mu_target_bonus == nullptr || aligned(mu_target_bonus, a4));
  overlap = overlap && !ratios_only;
  cudaError_t e = cudaSuccess;
  int rc = SDV_OK;
  auto launched = [&](cudaError_t err) {
    if (err == cudaSuccess) return check_launch();
    g_last_cuda_error = (int)err;
    cudaGetLastError();
    return (int)SDV_ECUDA;
  };
  // Paths (rows in groups of four elements):
  //  - log ratios alone: k_ratios, one kernel;
  //  - a plain call of few chains: k_chain, one kernel (launch_chain's rule);
  //  - rows up to kPipeMaxGroups: k_tiles + k_finish;
  //  - longer: k_tiles + k_finish_long.
  // A pipelined call launches every one of its kernels to overlap its predecessor.
  if (ratios_only)
    return launched(f32 ? launch_ratios<float>(A, B, L, w.vpt1, rows, s)
                        : launch_ratios<__nv_bfloat16>(A, B, L, w.vpt1, rows, s));
  if (!overlap) {
    bool taken = false;
    e = f32 ? launch_chain<float>(A, B, L, w.vpt1, rows, vec4, s, &taken)
            : launch_chain<__nv_bfloat16>(A, B, L, w.vpt1, rows, vec4, s, &taken);
    if (taken || e != cudaSuccess) {
      rc = launched(e);
      if (tev) {
        timing_record(tev[1], s);
        timing_record(tev[2], s);
      }
      return rc;
    }
  }
  const bool long_rows = ng > kPipeMaxGroups;
  // k_tiles + k_finish: tagged partials in the set after the one this workspace's
  // previous call used, no counters
  const uint64_t layout = (uint64_t)B * L * w.C1;   // the slots of a set, which fix both sets' places
  bool fresh = true;
  char* set = ws + w.part_off + (size_t)g_partial_sets.next(workspace, layout, &fresh) * w.part_set_bytes;
  S.fresh_set = fresh;
  S.tpart = (uint64_t*)set;
  S.tag = next_partial_tag();
  e = f32 ? launch_tiles<float>(A, B, L, w.vpt1, rows, s)
          : launch_tiles<__nv_bfloat16>(A, B, L, w.vpt1, rows, s);
  if ((rc = launched(e)) != SDV_OK) return rc;
  if (tev) timing_record(tev[1], s);
  // The finishing kernel is always launched to overlap the stream within the call: it
  // starts once every k_tiles CTA has stored its partial (and checks their tags); only the
  // stream's overlap with the previous call needs the pipelined contract.
  if (long_rows)
    e = f32 ? launch_finish_long<float>(A, B, L, vec4, s) : launch_finish_long<__nv_bfloat16>(A, B, L, vec4, s);
  else
    e = f32 ? launch_finish<float>(A, B, vec4, s) : launch_finish<__nv_bfloat16>(A, B, vec4, s);
  rc = launched(e);
  if (tev) timing_record(tev[2], s);
  return rc;
}

int verify_ex_impl(const void* x_draft, const void* mu_target, const void* mu_draft,
                        const float* sigma, int64_t sigma_stride_b, int B, int L, int64_t d, int dtype,
                        uint64_t seed, const uint64_t* seed_dev, int mode, const int32_t* L_eff,
                        const void* mu_target_bonus, const float* sigma_bonus, int residual_kind,
                        float omega, int32_t* accepted_len, void* y_out, float* log_ratio_out,
                        float* delta_norm_out, uint32_t* status_out, float* chain_aux_out,
                        void* workspace, size_t workspace_bytes, bool timed, void* stream, bool overlap) {
  int rc = validate_window(x_draft, mu_target, mu_draft, sigma, sigma_stride_b, B, L, d, dtype);
  if (rc != SDV_OK) return rc;
  if (mode != SDV_MODE_SAMPLE && mode != SDV_MODE_BLOCK) return SDV_EINVAL;
  if (residual_kind != SDV_RESIDUAL_DECOMPOSITION && residual_kind != SDV_RESIDUAL_REFLECTION)
    return SDV_EINVAL;
  if (residual_kind == SDV_RESIDUAL_REFLECTION && mode != SDV_MODE_SAMPLE) return SDV_EINVAL;
  if (!(omega > 0.f) || !std::isfinite(omega)) return SDV_EINVAL;
  if (!accepted_len || !y_out) return SDV_EINVAL;
  if ((mu_target_bonus == nullptr) != (sigma_bonus == nullptr)) return SDV_EINVAL;
  const size_t es = dtype == SDV_BF16 ? 2 : 4;
  if (!aligned(y_out, es) || !aligned(accepted_len, 4) ||
      (mu_target_bonus && !aligned(mu_target_bonus, es)) || (sigma_bonus && !aligned(sigma_bonus, 4)) ||
      (L_eff && !aligned(L_eff, 4)) || (log_ratio_out && !aligned(log_ratio_out, 4)) ||
      (delta_norm_out && !aligned(delta_norm_out, 4)) || (status_out && !aligned(status_out, 4)) ||
      (chain_aux_out && !aligned(chain_aux_out, 4)) || (seed_dev && !aligned(seed_dev, 8)))
    return SDV_EALIGN;
  const WsLayout w = ws_layout(B, L, d, dtype);
  if (!workspace || workspace_bytes < w.total) return SDV_ENOWORKSPACE;
  if (!aligned(workspace, 256)) return SDV_EALIGN;
  return enqueue_verify(x_draft, mu_target, mu_draft, sigma, sigma_stride_b, B, L, d, dtype, seed,
                        seed_dev, mode, L_eff, mu_target_bonus, sigma_bonus, residual_kind, omega,
                        accepted_len, y_out, log_ratio_out, delta_norm_out, status_out,
                        chain_aux_out, false, timed, overlap, workspace, (cudaStream_t)stream);
}

}  // namespace sdv

using namespace sdv;

extern "C" {

const char* sdv_version(void) { return "specdiff-gb300 0.2 (sm_103a)"; }

const char* sdv_strerror(int code) {
  switch (code) {
    case SDV_OK: return "ok";
    case SDV_EINVAL: return "invalid argument";
    case SDV_EALIGN: return "misaligned pointer";
    case SDV_ECUDA: return "CUDA launch failure";
    case SDV_ENOWORKSPACE: return "workspace missing or too small";
    default: return "unknown error";
  }
}

int sdv_last_cuda_error(void) { return g_last_cuda_error; }

size_t sdv_workspace_bytes(int B, int L, int64_t d, int dtype) {
  if (B < 1 || L < 1 || L > SDV_MAX_L || d < 1 || (dtype != SDV_F32 && dtype != SDV_BF16)) return 0;
  return ws_layout(B, L, d, dtype).total;
}

int sdv_verify_ex(const void* x_draft, const void* mu_target, const void* mu_draft,
                  const float* sigma, int64_t sigma_stride_b, int B, int L, int64_t d, int dtype,
                  uint64_t seed, int mode, const int32_t* L_eff, const void* mu_target_bonus,
                  const float* sigma_bonus, int residual_kind, float omega,
                  int32_t* accepted_len, void* y_out, float* log_ratio_out,
                  float* delta_norm_out, uint32_t* status_out, float* chain_aux_out,
                  void* workspace, size_t workspace_bytes, sdv_stream_t stream) {
  return verify_ex_impl(x_draft, mu_target, mu_draft, sigma, sigma_stride_b, B, L, d, dtype, seed,
                        nullptr, mode, L_eff, mu_target_bonus, sigma_bonus, residual_kind, omega,
                        accepted_len, y_out, log_ratio_out, delta_norm_out, status_out,
                        chain_aux_out, workspace, workspace_bytes, true, stream, false);
}

int sdv_verify_pipelined(const void* x_draft, const void* mu_target, const void* mu_draft,
                         const float* sigma, int64_t sigma_stride_b, int B, int L, int64_t d, int dtype,
                         uint64_t seed, int mode, const int32_t* L_eff, const void* mu_target_bonus,
                         const float* sigma_bonus, int residual_kind, float omega,
                         int32_t* accepted_len, void* y_out, float* log_ratio_out,
                         float* delta_norm_out, uint32_t* status_out, float* chain_aux_out,
                         void* workspace, size_t workspace_bytes, sdv_stream_t stream) {
  return verify_ex_impl(x_draft, mu_target, mu_draft, sigma, sigma_stride_b, B, L, d, dtype, seed,
                        nullptr, mode, L_eff, mu_target_bonus, sigma_bonus, residual_kind, omega,
                        accepted_len, y_out, log_ratio_out, delta_norm_out, status_out,
                        chain_aux_out, workspace, workspace_bytes, true, stream, true);
}

int sdv_verify(const void* x_draft, const void* mu_target, const void* mu_draft,
               const float* sigma, int64_t sigma_stride_b, int B, int L, int64_t d, int dtype,
               uint64_t seed, int mode, int32_t* accepted_len, void* y_out,
               float* log_ratio_out, float* delta_norm_out, uint32_t* status_out,
               void* workspace, size_t workspace_bytes, sdv_stream_t stream) {
  return sdv_verify_ex(x_draft, mu_target, mu_draft, sigma, sigma_stride_b, B, L, d, dtype, seed,
                       mode, nullptr, nullptr, nullptr, SDV_RESIDUAL_DECOMPOSITION, 1.0f,
                       accepted_len, y_out, log_ratio_out, delta_norm_out, status_out, nullptr,
                       workspace, workspace_bytes, stream);
}

int sdv_log_ratios(const void* x_draft, const void* mu_target, const void* mu_draft,
                   const float* sigma, int64_t sigma_stride_b, int B, int L, int64_t d, int dtype,
                   const int32_t* L_eff, float* log_ratio_out, float* delta_norm_out,
                   void* workspace, size_t workspace_bytes, sdv_stream_t stream) {
  int rc = validate_window(x_draft, mu_target, mu_draft, sigma, sigma_stride_b, B, L, d, dtype);
  if (rc != SDV_OK) return rc;
  if (!log_ratio_out || !delta_norm_out) return SDV_EINVAL;
  if (!aligned(log_ratio_out, 4) || !aligned(delta_norm_out, 4) || (L_eff && !aligned(L_eff, 4)))
    return SDV_EALIGN;
  const WsLayout w = ws_layout(B, L, d, dtype);
  if (!workspace || workspace_bytes < w.total) return SDV_ENOWORKSPACE;
  if (!aligned(workspace, 256)) return SDV_EALIGN;
  return enqueue_verify(x_draft, mu_target, mu_draft, sigma, sigma_stride_b, B, L, d, dtype, 0,
                        nullptr, SDV_MODE_BLOCK, L_eff, nullptr, nullptr, SDV_RESIDUAL_DECOMPOSITION,
                        1.0f, nullptr, nullptr, log_ratio_out, delta_norm_out, nullptr, nullptr, true,
                        false, false, workspace, (cudaStream_t)stream);
}

int sdv_accept_scan(const float* log_ratio, const float* delta_norm, int B, int L,
                    const int32_t* L_eff, uint64_t seed, int mode, float omega, int32_t* tau_out,
                    float* log_alpha_res_out, sdv_stream_t stream) {
  if (!log_ratio || !delta_norm || !tau_out) return SDV_EINVAL;
  if (B < 1 || L < 1 || L > SDV_MAX_L || B > (1 << 30)) return SDV_EINVAL;
  if (mode != SDV_MODE_SAMPLE && mode != SDV_MODE_BLOCK) return SDV_EINVAL;
  if (!(omega > 0.f) || !std::isfinite(omega)) return SDV_EINVAL;
  if (!aligned(log_ratio, 4) || !aligned(delta_norm, 4) || !aligned(tau_out, 4) ||
      (log_alpha_res_out && !aligned(log_alpha_res_out, 4)) || (L_eff && !aligned(L_eff, 4)))
    return SDV_EALIGN;
  ScanArgs A{};
  A.ell_in = log_ratio; A.dn_in = delta_norm; A.B = B; A.L = L; A.L_eff = L_eff;
  A.seed = seed; A.mode = mode; A.inv_omega2 = 1.0f / (omega * omega);
  A.tau_out = tau_out; A.la_res_out = log_alpha_res_out;
  k_scan<<<(B + kK2Threads / 32 - 1) / (kK2Threads / 32), kK2Threads, 0, (cudaStream_t)stream>>>(A);
  return check_launch();
}

int sdv_usample(const float* delta_norm, const float* log_alpha, const uint32_t* w_bits, int n,
                float* U_out, uint32_t* status_out, sdv_stream_t stream) {
  if (!delta_norm || !log_alpha || !w_bits || !U_out || n < 0) return SDV_EINVAL;
  if (!aligned(delta_norm, 4) || !aligned(log_alpha, 4) || !aligned(w_bits, 4) ||
      !aligned(U_out, 4) || (status_out && !aligned(status_out, 4)))
    return SDV_EALIGN;
  if (n == 0) return SDV_OK;
  k_usample<<<(n + kK2Threads / 32 - 1) / (kK2Threads / 32), kK2Threads, 0, (cudaStream_t)stream>>>(delta_norm, log_alpha, w_bits, n, U_out, status_out);
  return check_launch();
}

int sdv_philox(const uint32_t* ctr, uint64_t seed, int n, uint32_t* out, sdv_stream_t stream) {
  if (!ctr || !out || n < 0) return SDV_EINVAL;
  if (!aligned(ctr, 16) || !aligned(out, 16)) return SDV_EALIGN;
  if (n == 0) return SDV_OK;
  k_philox<<<(n + 255) / 256, 256, 0, (cudaStream_t)stream>>>((const uint4*)ctr, seed, n, (uint4*)out);
  return check_launch();
}

int sdv_normals(uint64_t seed, int B, int64_t d, int stream_id, uint32_t sub, float* out,
                sdv_stream_t stream) {
  if (!out || B < 1 || d < 1 || stream_id < 0) return SDV_EINVAL;
  if (!aligned(out, 4)) return SDV_EALIGN;
  const int64_t n = (int64_t)B * ((d + 3) / 4);
  k_normals<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream>>>(seed, B, d, (uint32_t)stream_id, sub, out);
  return check_launch();
}

int sdv_special(int which, const float* z, int n, float* out, sdv_stream_t stream) {
  if (!z || !out || n < 0 || which < 0 || which > 2) return SDV_EINVAL;
  if (!aligned(z, 4) || !aligned(out, 4)) return SDV_EALIGN;
  if (n == 0) return SDV_OK;
  k_special<<<(n + 255) / 256, 256, 0, (cudaStream_t)stream>>>(which, z, n, out);
  return check_launch();
}

int sdv_timing_enable(int slots) {
  if (slots < 0 || slots > (1 << 20)) return SDV_EINVAL;
  timing_destroy();
  if (slots == 0) return SDV_OK;
  g_timing.ev.resize(3 * (size_t)slots);
  for (auto& e : g_timing.ev) {
    if (cudaEventCreate(&e) != cudaSuccess) {
      g_last_cuda_error = (int)cudaGetLastError();
      g_timing.ev.clear();
      return SDV_ECUDA;
    }
  }
  g_timing.slots = slots;
  return SDV_OK;
}

int sdv_timing_stride(int every) {
  if (every < 1) return SDV_EINVAL;
  g_timing.stride = every;
  g_timing.calls = 0;
  return SDV_OK;
}

int sdv_timing_read(int n_calls, float* ms3) {
  if (!ms3 || g_timing.slots == 0 || n_calls < 1 || n_calls > g_timing.slots ||
      n_calls > g_timing.next)
    return SDV_EINVAL;
  double acc[3] = {0, 0, 0};
  for (int i = 0; i < n_calls; ++i) {
    const int s = (int)((g_timing.next - 1 - i) % g_timing.slots);
    cudaEvent_t* e = &g_timing.ev[3 * (size_t)s];
    if (cudaEventSynchronize(e[2]) != cudaSuccess) {
      g_last_cuda_error = (int)cudaGetLastError();
      return SDV_ECUDA;
    }
    for (int k = 0; k < 2; ++k) {
      float ms = 0.f;
      if (cudaEventElapsedTime(&ms, e[k], e[k + 1]) != cudaSuccess) {
        g_last_cuda_error = (int)cudaGetLastError();
        return SDV_ECUDA;
      }
      acc[k] += ms;
    }
  }
  for (int k = 0; k < 3; ++k) ms3[k] = (float)acc[k];
  return SDV_OK;
}

}  // extern "C"
