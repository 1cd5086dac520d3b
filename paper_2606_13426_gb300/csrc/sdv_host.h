// sdv_host.h - internal launch parameters and workspace layout of libspecdiff.
#pragma once

#include <cstddef>
#include <cstdint>

#include "../../include/specdiff.h"

namespace sdv {

// Streaming kernels: threads per CTA and 16-byte vectors per thread per tensor of a tile.
constexpr int kK1Threads = 256;
constexpr int kK1Vpt = 4;
// With this many chains of at most kFinishManyMaxGroups groups of 4 elements, k_finish takes
// fewer threads each.
constexpr int kManyChainMin = 512;
constexpr int64_t kFinishManyMaxGroups = 256;
// Resident k_tiles CTAs per SM (its register budget).  Three vectors per thread fit 48
// registers, so that the stream still finds room beside the previous pipelined call's
// k_finish CTAs.
constexpr int tile_min_blocks(int vpt) { return vpt <= 1 ? 8 : (vpt == 2 ? 6 : (vpt == 3 ? 5 : 4)); }
constexpr int kFinishThreads = 128;
constexpr int kFinishThreadsMany = 64;
constexpr int kFinishWideThreads = 256;
// Rows of up to kElementMax elements have at most kElementsPerThread for a thread.
constexpr int kElementsPerThread = 4;
constexpr int64_t kElementMax = kElementsPerThread * kK1Threads;
// Stand-alone acceptance scan: one warp per chain.
constexpr int kK2Threads = 128;
// Rows of up to kFinishMaxGroups groups of 4 elements are finished by k_finish's
// kFinishThreads, up to kPipeMaxGroups by kFinishWideThreads (the residual's noise cached in
// dynamic shared memory, 16 KB or up to 64 KB); longer rows by k_finish_long.
constexpr int64_t kFinishMaxGroups = 1024;
constexpr int64_t kPipeMaxGroups = 4096;

// How the kernels read the rows of a window: element by element, as whole aligned 16-byte
// vectors, or as vectors over rows that start anywhere within one (arrays 16-byte aligned).
enum : int { kRowsElement = 0, kRowsAligned = 1, kRowsUnaligned = 2 };

enum : int32_t {
  kKindInactive = 0,
  kKindResid = 1,      // decomposition residual
  kKindReflect = 2,    // reflection residual
  kKindZeroDelta = 3,  // |Delta_tau| = 0: m^q + sigma G
  kKindCopy = 4,       // full accept, last draft row
  kKindBonus = 5,      // full accept, bonus step
};

// Per-chain result of the scan, consumed by the residual writer (48 bytes).
struct ChainState {
  int32_t tau;      // 1-based
  int32_t row;      // row of the window the residual writer reads (tau-1, or the last draft)
  float U;          // residual 1-D draw
  float la_res;     // log alpha_{tau-1}
  float sigma;      // sigma_tau
  float dnorm;      // |Delta_tau|
  float inv_norm;   // 1/|delta_tau|, delta = m^p - m^q
  float refl;       // 1 + 2 S1/S2 (reflection: y = x - delta * refl)
  uint32_t status;
  int32_t kind;
  int32_t pad[2];
};

struct ScanArgs {
  uint64_t* tpart;        // k_tiles' slots, [B, L, C] pairs of words (S1 | tag << 32, S2 | tag << 32)
  uint32_t tag;           // this call's tag of its k_tiles partials (never 0: a free slot's tag)
  bool fresh_set;         // the first call on the set since another layout (PartialSets): its contents are unknown
  int C;
  const float* sigma;
  int64_t sstride;
  const float* ell_in;
  const float* dn_in;
  int B, L;
  const int32_t* L_eff;
  uint64_t seed;
  const uint64_t* seed_dev;  // nullable: the seed is read from device memory instead
  int mode;
  float inv_omega2;
  int residual_kind;
  bool has_bonus;
  float* ell_out;
  float* dn_out;
  int32_t* accepted_len;
  int32_t* tau_out;
  float* la_res_out;
  uint32_t* status_out;
  float* aux_out;
};

// Arguments of the kernels that stream a window or finish its chains.
struct VerifyArgs {
  const void* x;
  const void* mq;
  const void* mp;
  const void* mq_bonus;
  const float* sigma_bonus;
  int64_t d;
  int64_t chunk;
  bool serial;           // a plain call: its stream waits for the work before it
  int sms;               // the device's SMs (k_chain)
  void* y;
  ScanArgs S;
};

struct WsLayout {
  int vpt1;        // K1 16-byte vectors per thread per tensor
  int64_t chunk1;  // elements of a row per K1 tile
  int C1;          // K1 tiles per row
  // two sets of k_tiles' slots [B, L, C1], 16 bytes each
  size_t part_off, part_set_bytes, total;
};

WsLayout ws_layout(int B, int L, int64_t d, int dtype);

// sdv_verify_ex with the seed taken from device memory when seed_dev is not null (it
// is read by the kernels, so a captured call follows the value at replay), event
// timing skipped when timed is false, and, with overlap, the permission to start
// before the previous kernel on the stream has finished (sdv_verify_pipelined).  Same
// validation and return codes.
int verify_ex_impl(const void* x_draft, const void* mu_target, const void* mu_draft,
                   const float* sigma, int64_t sigma_stride_b, int B, int L, int64_t d, int dtype,
                   uint64_t seed, const uint64_t* seed_dev, int mode, const int32_t* L_eff,
                   const void* mu_target_bonus, const float* sigma_bonus, int residual_kind,
                   float omega, int32_t* accepted_len, void* y_out, float* log_ratio_out,
                   float* delta_norm_out, uint32_t* status_out, float* chain_aux_out,
                   void* workspace, size_t workspace_bytes, bool timed, void* stream,
                   bool overlap = false);

// Records a cudaError_t for sdv_last_cuda_error() (this host thread).
void set_last_cuda_error(int err);

// SMs of the current device (152 if it cannot be asked).
int sm_count();

// Largest number of mixture components of the analytic target.
constexpr int kSdvMaxComponents = SDV_MAX_COMPONENTS;

}  // namespace sdv
