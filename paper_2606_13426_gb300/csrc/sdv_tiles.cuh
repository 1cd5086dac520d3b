// sdv_tiles.cuh - reading a window: 16-byte streaming loads, the (S1, S2) sums of one tile
// of a row (App. "Density ratio calculations"), and group-of-four loads and stores of the
// residual row (sm_103a).
#pragma once

#include <cstring>

#include "sdv_device.cuh"
#include "sdv_host.h"

namespace sdv {

// ---------------------------------------------------------------- small helpers
template <int NT>
__device__ __forceinline__ float2 block_sum2(float a, float b, float2* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) red[w] = make_float2(a, b);
  __syncthreads();
  float2 r = make_float2(0.f, 0.f);
  if (w == 0) {
    r = (lane < NT / 32) ? red[lane] : make_float2(0.f, 0.f);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      r.x += __shfl_xor_sync(0xffffffffu, r.x, o);
      r.y += __shfl_xor_sync(0xffffffffu, r.y, o);
    }
  }
  return r;  // valid in thread 0
}

__device__ __forceinline__ void unpack(const uint4& v, float (&f)[4]) {
  f[0] = __uint_as_float(v.x);
  f[1] = __uint_as_float(v.y);
  f[2] = __uint_as_float(v.z);
  f[3] = __uint_as_float(v.w);
}
__device__ __forceinline__ void unpack(const uint4& v, float (&f)[8]) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    f[2 * i] = __uint_as_float(w[i] << 16);
    f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
  }
}

// Read-once streaming load: no L1 allocation.
__device__ __forceinline__ uint4 ldg_stream(const uint4* p) {
  uint4 r;
  asm("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
      : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
      : "l"(p));
  return r;
}

// Elements i .. i + 3 of a row of d (zeros past its end).  VEC4: d is a multiple of four and
// rows are aligned to four elements, so a group lies whole within the row or past it.
template <typename T, bool VEC4>
__device__ __forceinline__ void load4(const T* p, int64_t i, int64_t d, float (&f)[4]) {
  if (VEC4) {
    // a group past the end loads the row's first (no branch between the loads of several)
    const bool in = i < d;
    const T* q = in ? p + i : p;
    if (sizeof(T) == 4) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(q));
      f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w;
    } else {
      const uint2 v = __ldg(reinterpret_cast<const uint2*>(q));
      f[0] = __uint_as_float(v.x << 16); f[1] = __uint_as_float(v.x & 0xffff0000u);
      f[2] = __uint_as_float(v.y << 16); f[3] = __uint_as_float(v.y & 0xffff0000u);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) f[k] = in ? f[k] : 0.f;
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) f[k] = (i + k < d) ? Elem<T>::load(p + i + k) : 0.f;
  }
}

// Stores a group that starts within the row (i < d).
template <typename T, bool VEC4>
__device__ __forceinline__ void store4(T* p, int64_t i, int64_t d, const float (&f)[4]) {
  if (VEC4) {
    if (sizeof(T) == 4) {
      *reinterpret_cast<float4*>(p + i) = make_float4(f[0], f[1], f[2], f[3]);
    } else {
      __nv_bfloat162 lo = __floats2bfloat162_rn(f[0], f[1]);
      __nv_bfloat162 hi = __floats2bfloat162_rn(f[2], f[3]);
      uint2 v;
      memcpy(&v.x, &lo, 4);
      memcpy(&v.y, &hi, 4);
      *reinterpret_cast<uint2*>(p + i) = v;
    }
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (i + k < d) Elem<T>::store(p + i + k, f[k]);
  }
}

// ---------------------------------------------------------------- tile reduction
// (S1, S2) share of this thread in elements [e0, e1) of the row starting at element `base`,
// read one by one (arrays that do not start on a 16-byte boundary, and short rows of a length
// that is no multiple of a vector).
template <typename T>
__device__ __forceinline__ float2 tile_sums(const T* __restrict__ x, const T* __restrict__ mq,
                                            const T* __restrict__ mp, int64_t base, int64_t e0, int64_t e1) {
  float s1 = 0.f, s2 = 0.f;
  for (int64_t e = e0 + threadIdx.x; e < e1; e += kK1Threads) {
    const float fx = Elem<T>::load(x + base + e);
    const float fq = Elem<T>::load(mq + base + e);
    const float fp = Elem<T>::load(mp + base + e);
    const float dl = fp - fq, a = fx - fp;  // m^p - m^q, yhat - m^p
    s1 = fmaf(a, dl, s1);
    s2 = fmaf(dl, dl, s2);
  }
  return make_float2(s1, s2);
}

// One tile's 3 VPT 16-byte vectors per thread (a tile is one full sweep: VPT vectors
// per thread and tensor), issued together with guarded loads, and its (S1, S2)
// contribution.
template <int VPT>
struct TileBuf {
  uint4 x[VPT], q[VPT], p[VPT];
};

template <typename T, int VPT>
__device__ __forceinline__ void tile_issue(const T* __restrict__ x, const T* __restrict__ mq,
                                           const T* __restrict__ mp, int64_t base, int64_t e0, int64_t e1,
                                           TileBuf<VPT>& B) {
  constexpr int V = 16 / (int)sizeof(T);
  const int64_t v0 = (base + e0) / V;
  const int nv = (int)((e1 - e0) / V);
  const uint4* X = reinterpret_cast<const uint4*>(x) + v0;
  const uint4* Q = reinterpret_cast<const uint4*>(mq) + v0;
  const uint4* P = reinterpret_cast<const uint4*>(mp) + v0;
  const uint4 z = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
  for (int u = 0; u < VPT; ++u) {
    const int vv = threadIdx.x + u * kK1Threads;
    B.x[u] = vv < nv ? ldg_stream(X + vv) : z;
  }
#pragma unroll
  for (int u = 0; u < VPT; ++u) {
    const int vv = threadIdx.x + u * kK1Threads;
    B.q[u] = vv < nv ? ldg_stream(Q + vv) : z;
  }
#pragma unroll
  for (int u = 0; u < VPT; ++u) {
    const int vv = threadIdx.x + u * kK1Threads;
    B.p[u] = vv < nv ? ldg_stream(P + vv) : z;
  }
}

template <typename T, int VPT>
__device__ __forceinline__ float2 tile_fma(const TileBuf<VPT>& B) {
  constexpr int V = 16 / (int)sizeof(T);
  float s1 = 0.f, s2 = 0.f;
#pragma unroll
  for (int u = 0; u < VPT; ++u) {
    float fx[V], fq[V], fp[V];
    unpack(B.x[u], fx);
    unpack(B.q[u], fq);
    unpack(B.p[u], fp);
#pragma unroll
    for (int k = 0; k < V; ++k) {
      const float dl = fp[k] - fq[k];  // m^p - m^q (zero-filled vectors contribute 0)
      const float a = fx[k] - fp[k];   // yhat - m^p
      s1 = fmaf(a, dl, s1);
      s2 = fmaf(dl, dl, s2);
    }
  }
  return make_float2(s1, s2);
}

// ---------------------------------------------------------------- rows off 16-byte boundaries
// Tile c of a row whose length is no multiple of a 16-byte vector's V elements (so that rows
// start anywhere within a vector), the arrays themselves being 16-byte aligned: the vectors
// that lie whole within the row, 256 VPT to a tile, and its first and last few elements, less
// than a vector each, one to a thread of the first and of the last tile.  One vector load
// replaces V element loads: 75 x 75 x 3 bf16 rows, 24 chains x 7 steps, streamed in 22 us
// with element loads.
struct EdgeBuf {
  float x, q, p;
};

template <typename T, int VPT>
__device__ __forceinline__ void unaligned_issue(const T* __restrict__ x, const T* __restrict__ mq,
                                                const T* __restrict__ mp, int64_t base, int64_t d, int c, int C,
                                                TileBuf<VPT>& B, EdgeBuf& E) {
  constexpr int V = 16 / (int)sizeof(T);
  const int64_t v0 = base / V * V;                 // the row's first vector, in elements
  const int64_t m = base - v0, end = m + d;        // the row's start and end from there
  const int64_t f = m > 0 ? V : 0;                 // the whole vectors, in elements from v0 on
  const int64_t l = end / V * V;
  const int64_t e0 = f + (int64_t)c * kK1Threads * VPT * V;
  tile_issue<T, VPT>(x, mq, mp, v0, e0, max(e0, min(e0 + kK1Threads * VPT * V, l)), B);
  const int t = threadIdx.x;
  const bool head = t < V;
  const int64_t e = head ? m + t : max(l, f) + (t - V);
  const bool in = head ? c == 0 && m > 0 && e < min((int64_t)V, end) : t < 2 * V && c == C - 1 && e < end;
  E.x = in ? Elem<T>::load(x + v0 + e) : 0.f;
  E.q = in ? Elem<T>::load(mq + v0 + e) : 0.f;
  E.p = in ? Elem<T>::load(mp + v0 + e) : 0.f;
}

template <typename T, int VPT>
__device__ __forceinline__ float2 unaligned_fma(const TileBuf<VPT>& B, const EdgeBuf& E) {
  const float2 s = tile_fma<T, VPT>(B);
  const float dl = E.p - E.q, a = E.x - E.p;
  return make_float2(fmaf(a, dl, s.x), fmaf(dl, dl, s.y));
}

}  // namespace sdv
