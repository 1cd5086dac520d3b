// sdv_device.cuh - device-side building blocks of the verification step (sm_103a).
//
//  * Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11) and the uniform /
//    Box-Muller transforms of the counter layout documented in specdiff.h.
//  * log Phi and the scaled log-CDF g(a) = log Phi(a) + a^2/2, its derivative
//    g'(s) = lambda(s) + s (lambda = phi/Phi, the inverse Mills ratio), and
//    differences g(hi) - g(hi - h) by 8-point Gauss-Legendre quadrature.
//  * The block-verification acceptance probability h_j (Algorithm
//    block-verification) in log form (App. "Density ratio calculations"), from
//    the same residual mass log v that the U-sampler's setup computes.
//  * The residual's 1-D draw U = Psi_alpha^{-1}(w) (Prop. decomposition,
//    Eq. u-cdf, Algorithm u-sample) as a one-warp multisection.
//
// Everything is fp32: GB300's fp64 rate is a small fraction of its fp32 rate.
// The special-function helpers are __noinline__: inlined at every call site they
// made the acceptance-scan kernel's code too large for the instruction cache.
// The forms below avoid the cancellations that fp32 would otherwise suffer:
//  - v = alpha Phi(a+) - Phi(a-) is written as alpha Phi(a+) (1 - e^{x0}) with
//    x0 = log(Phi(a-)/(alpha Phi(a+))) = g(a-) - g(a+), exact because
//    log alpha + a-^2/2 = a+^2/2 (a+- = log alpha / D +- D/2);
//  - Psi near its upper end a+ (where its density vanishes) is evaluated as a
//    complement, 1 - Psi(a+ - t) = int_0^t phi(a- - s) expm1(D s) ds / v,
//    which has a positive integrand (alpha phi(u) - phi(u - D) =
//    phi(u - D) expm1(D (a+ - u)));
//  - for s < -4, lambda(s) + s = 1/(x + 2/(x + 3/(x + ...))), x = -s, which is
//    Laplace's continued fraction for the Mills ratio with its first term
//    cancelled analytically.
// The quadratures' node pairs are not unrolled.  The code runs on one warp per chain, mostly
// from a cold instruction cache: rolled, a pair's two nodes still overlap, and the smaller
// code (gdiff 19 KB unrolled, of 130 KB in a finishing kernel) measured faster (pixel batch
// 25.1 -> 23.9 us, tiny call 13.3 -> 12.7).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>
#include <cuda_bf16.h>

namespace sdv {

// ---------------------------------------------------------------- Philox
constexpr float kLn2Hi = 0.69314718055994531f;  // log 2 (fp32)
constexpr uint32_t kPhiloxM0 = 0xD2511F53u;
constexpr uint32_t kPhiloxM1 = 0xCD9E8D57u;
constexpr uint32_t kPhiloxW0 = 0x9E3779B9u;
constexpr uint32_t kPhiloxW1 = 0xBB67AE85u;

enum : uint32_t {
  kStreamCoin = 0,
  kStreamUSample = 1,
  kStreamResid = 2,
  kStreamBonus = 3,
  kStreamDraft = 4,
  kStreamInit = 5,
  kStreamEM = 6,
};

// Ten rounds of the Philox4x32 S-box: (c0,c1,c2,c3) -> (hi(M1 c2)^c1^k0,
// lo(M1 c2), hi(M0 c0)^c3^k1, lo(M0 c0)); the key is bumped by the Weyl
// constants between rounds.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) {
      k0 += kPhiloxW0;
      k1 += kPhiloxW1;
    }
    const uint32_t lo0 = kPhiloxM0 * c.x;
    const uint32_t hi0 = __umulhi(kPhiloxM0, c.x);
    const uint32_t lo1 = kPhiloxM1 * c.z;
    const uint32_t hi1 = __umulhi(kPhiloxM1, c.z);
    c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
  }
  return c;
}

__device__ __forceinline__ uint4 philox_block(uint64_t seed, uint32_t c0, uint32_t c1,
                                              uint32_t c2, uint32_t c3) {
  return philox4x32_10(make_uint4(c0, c1, c2, c3), (uint32_t)seed, (uint32_t)(seed >> 32));
}

// log u for u = (x + 1/2) 2^-32 with one logarithm: in the lower half, u = m 2^e with
// m in [1/2, 1) split off the exponent bits, so log u = (e - 1) log 2 + log1p(2m - 1),
// 2m - 1 exact; the upper half goes through 1 - u, exact in the integer domain, as
// log1p(-(1 - u)), so log u keeps full relative accuracy near 1.  The argument and the
// offset are selected first (no divergence between lanes), then one log1pf.
__device__ __forceinline__ float log_uniform(uint32_t x) {
  const float u = ((float)x + 0.5f) * 0x1p-32f;
  const uint32_t ub = __float_as_uint(u);
  const float m2 = __uint_as_float((ub & 0x007fffffu) | 0x3f800000u);   // 2m in [1, 2)
  const float e1 = (float)((int)(ub >> 23) - 127);                      // e - 1
  const float v = ((float)(0xFFFFFFFFu - x) + 0.5f) * 0x1p-32f;          // 1 - u
  const bool lower = x < 0x80000000u;
  const float arg = lower ? m2 - 1.0f : -v;
  const float base = lower ? e1 * kLn2Hi : 0.0f;
  return base + log1pf(arg);
}

// Box-Muller on two words: (r cos 2 pi u1, r sin 2 pi u1), r = sqrt(-2 ln u0).
__device__ __forceinline__ float2 box_muller(uint32_t w0, uint32_t w1) {
  const float r = sqrtf(-2.0f * log_uniform(w0));
  float s, c;
  sincospif(((float)w1 + 0.5f) * 0x1p-31f, &s, &c);
  return make_float2(r * c, r * s);
}

// Four normals of Philox block (b, blk, stream, sub): elements 4 blk .. 4 blk + 3.
__device__ __forceinline__ float4 normals4(uint64_t seed, uint32_t b, uint32_t blk,
                                           uint32_t stream, uint32_t sub) {
  const uint4 w = philox_block(seed, b, blk, stream, sub);
  const float2 z01 = box_muller(w.x, w.y);
  const float2 z23 = box_muller(w.z, w.w);
  return make_float4(z01.x, z01.y, z23.x, z23.y);
}

// normals4 as one shared copy, for the residual paths that run once per chain.
static __device__ __noinline__ float4 normals4_f(uint64_t seed, uint32_t b, uint32_t blk, uint32_t stream,
                                               uint32_t sub) {
  return normals4(seed, b, blk, stream, sub);
}

// ---------------------------------------------------------------- normal CDF helpers
constexpr float kSqrtHalf = 0.70710678118654752f;
constexpr float kHalfLog2Pi = 0.91893853320467274f;  // log(2 pi) / 2
constexpr float kLn2 = 0.69314718055994531f;

// Reciprocal without the IEEE slow path: the hardware approximation refined by one
// Newton step (about 1 ulp for finite non-zero x; +-inf gives 0 and 0 gives inf).
// IEEE division and __frcp_rn branch to a slow path, which keeps independent
// evaluations from overlapping; this form does not.
__device__ __forceinline__ float frcp_fast(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  const float e = fmaf(-x, r, 1.0f);
  return (r != 0.0f && isfinite(r)) ? fmaf(r, e, r) : r;
}

// 8-point Gauss-Legendre nodes / weights on [-1, 1] (positive half).
static __constant__ float kGLx[4] = {0.18343464249564978f, 0.52553240991632899f,
                                          0.79666647741362673f, 0.96028985649753618f};
static __constant__ float kGLw[4] = {0.36268378337836166f, 0.31370664587788688f,
                                          0.22238103445337443f, 0.10122853629037706f};

// The scaled complementary error function erfcx(z) = exp(z^2) erfc(z), branch-free and
// inline so that independent evaluations (the quadrature nodes below) overlap.  For
// z >= 0: erfcx(z) = t exp(f(t)), t = 1/(1 + z/2), with f(t) = log(erfcx(z)/t) a
// degree-11 polynomial in x = 2t - 1 (a Chebyshev fit of f, generated by
// gen_erfcx_coeffs.py; max relative error 1.4e-7 in fp32).  z = +inf gives t = 0 and 0.
__device__ __forceinline__ float erfcx_pos(float z) {
  const float t = frcp_fast(fmaf(0.5f, z, 1.0f));
  const float x = fmaf(2.0f, t, -1.0f);
  // f(t) = log(erfcx(z)/t) in the power basis of x = 2t - 1, degree 11 (Horner)
  float f = -8.728381024e-05f;
  f = fmaf(f, x, 8.000738166e-06f);
  f = fmaf(f, x, 5.737663720e-04f);
  f = fmaf(f, x, -2.279109660e-04f);
  f = fmaf(f, x, -2.288765239e-03f);
  f = fmaf(f, x, 1.794066250e-03f);
  f = fmaf(f, x, 8.808825369e-03f);
  f = fmaf(f, x, -9.880019324e-03f);
  f = fmaf(f, x, -4.689364056e-02f);
  f = fmaf(f, x, 4.734388761e-02f);
  f = fmaf(f, x, 6.726431548e-01f);
  f = fmaf(f, x, -6.717940917e-01f);
  return t * expf(f);
}

// erfcx of any sign: erfcx(-a) = 2 exp(a^2) - erfcx(a) (no cancellation: the first
// term is at least 2, the second at most 1), with a^2 split exactly (hi + lo) so that
// exp(a^2) keeps full relative accuracy; overflows to +inf for a above ~9.4.
__device__ __forceinline__ float erfcx_any(float z) {
  const float a = fabsf(z);
  const float e = erfcx_pos(a);
  const float hi = a * a, lo = fmaf(a, a, -hi);
  const float big = 2.0f * expf(hi) * (1.0f + lo);
  return (z >= 0.0f) ? e : big - e;
}

// (log Phi(a), g(a)) from one scaled complement E = erfcx(|a|/sqrt 2)/2 =
// Phi(-|a|) e^{a^2/2}: for a <= 0, log Phi(a) = log E - a^2/2 (no underflow); for
// a > 0, log Phi(a) = log(1 - E e^{-a^2/2}).  Both branches are computed and one is
// selected, so that lanes with different arguments do not diverge.
__device__ __forceinline__ float2 log_ndtr_g(float a) {
  const float E = 0.5f * erfcx_pos(fabsf(a) * kSqrtHalf);
  const float h = 0.5f * a * a;
  const float lneg = logf(E);                  // log Phi(-|a|) + a^2/2
  const float lpos = log1pf(-E * expf(-h));    // log Phi(|a|)
  return (a <= 0.0f) ? make_float2(lneg - h, lneg) : make_float2(lpos, lpos + h);
}

// log Phi(a).
static __device__ __noinline__ float log_ndtr(float a) { return log_ndtr_g(a).x; }

// g(a) = log Phi(a) + a^2/2 (moderate for a <= 0).
static __device__ __noinline__ float gfun(float a) { return log_ndtr_g(a).y; }

// g'(s) = lambda(s) + s > 0 in its two forms.  For s < -4 (x = -s) Laplace's
// continued fraction for the Mills ratio with its first term cancelled,
// lambda(s) + s = 1/(x + 2/(x + 3/(x + ... 16/x))), written as 1/(x c) with
// c = 1 + 2u/(1 + 3u/(1 + ... 16u)), u = 1/x^2 <= 1/16, and c evaluated by the
// forward three-term recurrence (fused multiply-adds on positive terms, one
// division); 15 levels give ~5e-10 relative at x = 4 and less beyond.  Elsewhere
// sqrt(2/pi)/erfcx(-s/sqrt 2) + s, which tends to s for large s as erfcx overflows.
__device__ __forceinline__ float gprime_cf(float s) {
  const float x = fmaxf(-s, 4.0f);
  const float u = frcp_fast(x * x);
  float a0 = 1.0f, a1 = 1.0f, b0 = 0.0f, b1 = 1.0f;  // A_{n-2}, A_{n-1}, B_{n-2}, B_{n-1}
#pragma unroll
  for (int n = 2; n <= 16; ++n) {
    const float an = (float)n * u;
    const float a2 = fmaf(an, a0, a1), b2 = fmaf(an, b0, b1);
    a0 = a1; a1 = a2; b0 = b1; b1 = b2;
  }
  return b1 * frcp_fast(x * a1);
}
__device__ __forceinline__ float gprime_ex(float s) {
  // lambda(s) = sqrt(2/pi) / erfcx(-s/sqrt 2); erfcx = +inf (s above ~13) gives 0
  const float e = erfcx_any(-s * kSqrtHalf);
  return (isinf(e) ? 0.0f : __fdividef(0.79788456080286536f, e)) + s;
}

// g(hi) - g(hi - h) for h >= 0; the interval length is exactly h.  The direct
// difference of two g values is accurate to a few 1e-7 absolute (|g| <= ~3 for
// arguments above -8); it is replaced by 8-point Gauss-Legendre quadrature of g'
// where the difference itself is small: short intervals and the deep left tail
// (g' ~ 1/|s| there).  The choice of form (and, inside the quadrature, of the
// form of g') is voted over the converged lanes, and every form that some lane
// needs is evaluated by all of them as straight-line code (the eight nodes
// interleave); lanes with different arguments therefore never diverge.
//
// Coop: how the pieces of an evaluation (the quadrature's node pairs, the direct form) are
// shared out.  OneWarp computes them all.  With CtaWarps the first `warps` warps of a CTA
// make the same call with the same arguments, each computes the pieces that fall to it and
// reads the others from shared memory: the chain of dependent instructions gets shorter, the
// result is the same to the last bit.  What is not a piece is computed by every one of them,
// so that more warps than help the pieces cost issue slots.
struct OneWarp {
  static constexpr bool kShared = false;
};
constexpr int kCoopPieces = 6;
struct CtaWarps {
  static constexpr bool kShared = true;
  float (*buf)[kCoopPieces][32];   // [2]: a set is written again two exchanges later
  int flip, warps;
  __device__ __forceinline__ bool mine(int piece) const { return (int)(threadIdx.x >> 5) == piece % warps; }
  __device__ __forceinline__ void put(int piece, float v) { buf[flip][piece][threadIdx.x & 31] = v; }
  // all pieces are in place; at(p) reads them until the next but one exchange
  __device__ __forceinline__ void exchange() {
    asm volatile("bar.sync 2, %0;" ::"r"(32 * warps) : "memory");
    flip ^= 1;
  }
  __device__ __forceinline__ float at(int piece) const { return buf[flip ^ 1][piece][threadIdx.x & 31]; }
};

// Node pair i of the quadrature over [hi - h, hi]: its weight times g' at both nodes.
__device__ __forceinline__ float gdiff_pair(int i, float m, float r, bool need_ex, bool need_cf) {
  const float s1 = m + r * kGLx[i], s2 = m - r * kGLx[i];
  float g1 = 0.0f, g2 = 0.0f;
  if (need_ex) {
    g1 = gprime_ex(s1);
    g2 = gprime_ex(s2);
  }
  if (need_cf) {
    const float c1 = gprime_cf(s1), c2 = gprime_cf(s2);
    g1 = (s1 < -4.0f) ? c1 : g1;
    g2 = (s2 < -4.0f) ? c2 : g2;
  }
  return kGLw[i] * (g1 + g2);
}

__device__ __forceinline__ float gdiff_direct(float hi, float h) {
  const float2 ph = log_ndtr_g(hi), pl = log_ndtr_g(hi - h);
  return (hi <= 0.0f) ? ph.y - pl.y : (ph.x - pl.x) + h * (hi - 0.5f * h);
}

template <typename Coop>
static __device__ __noinline__ float gdiff(float hi, float h, Coop& co) {
  const unsigned act = __activemask();
  const bool careful = ((h < 0.5f) || (hi < -2.0f)) && (h <= fmaxf(2.0f, 0.5f * fabsf(hi)));
  const bool any_quad = __any_sync(act, careful), any_direct = __any_sync(act, !careful);
  const float r = 0.5f * h, m = hi - r;
  // nodes lie in [hi - h, hi]
  const bool need_cf = __any_sync(act, careful && hi - h < -4.0f);
  const bool need_ex = __any_sync(act, careful && hi >= -4.0f);
  float acc = 0.0f, direct = 0.0f;
  if constexpr (Coop::kShared) {
    if (any_quad) {
#pragma unroll 1
      for (int i = (int)(threadIdx.x >> 5); i < 4; i += co.warps) co.put(i, gdiff_pair(i, m, r, need_ex, need_cf));
    }
    if (any_direct && co.mine(4)) co.put(4, gdiff_direct(hi, h));
    co.exchange();
    if (any_quad) acc = ((co.at(0) + co.at(1)) + co.at(2)) + co.at(3);
    if (any_direct) direct = co.at(4);
  } else {
    if (any_quad) {
#pragma unroll 1
      for (int i = 0; i < 4; ++i) acc += gdiff_pair(i, m, r, need_ex, need_cf);
    }
    if (any_direct) direct = gdiff_direct(hi, h);
  }
  return careful ? r * acc : direct;
}

// log(1 - e^x), x <= 0 (both forms evaluated, one selected).
__device__ __forceinline__ float log1mexp(float x) {
  x = fminf(x, 0.0f);
  const float near0 = logf(-expm1f(x));
  const float far = log1pf(-expf(x));
  return (x > -kLn2) ? near0 : far;
}

// log(e^y - 1), y >= 0 (both forms evaluated, one selected).
__device__ __forceinline__ float logexpm1(float y) {
  const float big = y + log1pf(-expf(-y));
  const float small = logf(expm1f(fminf(y, 15.0f)));
  return (y > 15.0f) ? big : small;
}

__device__ __forceinline__ float logaddexp(float a, float b) {
  const float m = fmaxf(a, b);
  if (m == -INFINITY) return -INFINITY;
  return m + log1pf(expf(-fabsf(a - b)));
}

// log(Phi(b) - Phi(a)) for a < b.
static __device__ __noinline__ float log_ndtr_interval(float a, float b) {
  if (b <= 0.0f) return log_ndtr(b) + log1mexp(log_ndtr(a) - log_ndtr(b));
  if (a >= 0.0f) return log_ndtr(-a) + log1mexp(log_ndtr(-b) - log_ndtr(-a));
  return log1pf(-(expf(log_ndtr(a)) + expf(log_ndtr(-b))));
}

// ---------------------------------------------------------------- block verification
// log h_j, h_j = v_j / (v_j + 1 - alpha_j), from log alpha_j (<= 0), |Delta_{j+1}| and
// log v_j, the residual mass of step j + 1 at alpha_j (usample_setup(|Delta_{j+1}|,
// log alpha_j).lv).  Limits: alpha_j = 1 -> h = 1; alpha_j = 0 or |Delta_{j+1}| = 0
// (alpha_j < 1) -> h = 0.
__device__ __forceinline__ float block_log_h(float la, float Dn, float lv) {
  if (isnan(la) || isnan(Dn)) return -INFINITY;
  if (!(la < 0.0f)) return 0.0f;
  if (la == -INFINITY || !(Dn > 0.0f)) return -INFINITY;
  return lv - logaddexp(lv, log1mexp(la));
}

// ---------------------------------------------------------------- residual U-sampler
struct UParams {
  float D, la, ap, am;
  float lv;      // log v
  float lvn;     // log v - log phi(a-)
  float lnd_ap;  // log Phi(a+)
  float g_ap;    // g(a+)
  float l1mx0;   // log(1 - e^{x0}) = log(v / (alpha Phi(a+)))
};

template <typename Coop>
static __device__ __noinline__ UParams usample_setup(float D, float la, Coop& co) {
  UParams P;
  P.D = D;
  P.la = la;
  P.ap = la * frcp_fast(D) + 0.5f * D;
  P.am = P.ap - D;
  const float x0 = -gdiff(P.ap, D, co);
  const float2 lg = log_ndtr_g(P.ap);
  P.lnd_ap = lg.x;
  P.g_ap = lg.y;
  P.l1mx0 = log1mexp(x0);
  P.lv = la + P.lnd_ap + P.l1mx0;
  P.lvn = gfun(P.am) + kHalfLog2Pi + logexpm1(-x0);
  return P;
}

// log Psi(a+ - t), t > 0, as [log Phi(u) - log Phi(a+)] + log(1 - e^x) - log(1 - e^{x0}),
// u = a+ - t: Psi(u) = alpha Phi(u) (1 - e^x) / v and v = alpha Phi(a+) (1 - e^{x0}).
// The first bracket is g(u) - g(a+) + t (a+ + u)/2 for a+ <= 0 (no term larger than
// the result grows with |a+|) and a plain difference of log Phi otherwise.
template <typename Coop>
static __device__ __noinline__ float usample_log_psi(float t, const UParams& P, Coop& co) {
  const float u = P.ap - t;
  const float x = -gdiff(u, P.D, co) - P.D * t;     // log(Phi(u - D) / (alpha Phi(u)))
  const float2 lg = log_ndtr_g(u);
  const float dl = (P.ap <= 0.0f) ? (lg.y - P.g_ap) + 0.5f * t * (P.ap + u) : lg.x - P.lnd_ap;
  return dl + log1mexp(x) - P.l1mx0;
}

// log(1 - Psi(a+ - t)), t > 0: the integral by 8-point Gauss-Legendre quadrature near the
// upper end, the difference of two intervals' masses elsewhere (which a warp evaluates is
// voted over its lanes).
__device__ __forceinline__ float usample_near_pair(int i, float r, const UParams& P) {
  const float s1 = r * (1.0f + kGLx[i]), s2 = r * (1.0f - kGLx[i]);
  return kGLw[i] * (expf(P.am * s1 - 0.5f * s1 * s1) * expm1f(P.D * s1) +
                    expf(P.am * s2 - 0.5f * s2 * s2) * expm1f(P.D * s2));
}

template <typename Coop>
static __device__ __noinline__ float usample_log_1mpsi(float t, const UParams& P, Coop& co) {
  const unsigned act = __activemask();
  const bool near = P.D * t <= 1.0f && -P.am * t <= 4.0f;
  const bool any_near = __any_sync(act, near), any_far = __any_sync(act, !near);
  // a lane's form is evaluated at a point of its own range, whichever it uses
  const float tn = near ? t : 0.0f, tf = near ? 1.0f : t;
  const float r = 0.5f * tn, u = P.ap - tf;
  float acc = 0.0f, lA = 0.0f, lB = 0.0f;
  if constexpr (Coop::kShared) {
    if (any_near) {
#pragma unroll 1
      for (int i = (int)(threadIdx.x >> 5); i < 4; i += co.warps) co.put(i, usample_near_pair(i, r, P));
    }
    if (any_far && co.mine(4)) co.put(4, P.la + log_ndtr_interval(u, P.ap));
    if (any_far && co.mine(5)) co.put(5, log_ndtr_interval(u - P.D, P.am));
    co.exchange();
    if (any_near) acc = ((co.at(0) + co.at(1)) + co.at(2)) + co.at(3);
    if (any_far) {
      lA = co.at(4);
      lB = co.at(5);
    }
  } else {
    if (any_near) {
#pragma unroll 1
      for (int i = 0; i < 4; ++i) acc += usample_near_pair(i, r, P);
    }
    if (any_far) {
      lA = P.la + log_ndtr_interval(u, P.ap);
      lB = log_ndtr_interval(u - P.D, P.am);
    }
  }
  const float vn = logf(r * acc) - P.lvn;
  if (!any_far) return vn;
  return near ? vn : lA + log1mexp(lB - lA) - P.lv;
}

// log psi(a+ - t) (the residual's density at u = a+ - t), in the form whose terms do
// not cancel: a- t - t^2/2 + log expm1(D t) - (log v - log phi(a-)) keeps every term
// small when t is small (the deep left tail), while log alpha + log phi(u) +
// log(1 - e^{-D t}) - log v does when u is moderate and D t is large (large |Delta|,
// where the first form cancels terms of size D^2/2).
__device__ __forceinline__ float usample_log_density(float t, const UParams& P) {
  const float u = P.ap - t;
  const float mag1 = fmaxf(fabsf(P.am * t), fmaxf(0.5f * t * t, P.D * t));
  const float mag2 = fmaxf(0.5f * u * u, fmaxf(fabsf(P.la), fabsf(P.lv)));
  if (mag1 <= mag2) return P.am * t - 0.5f * t * t + logexpm1(P.D * t) - P.lvn;
  return P.la - 0.5f * u * u - kHalfLog2Pi + log1mexp(-P.D * t) - P.lv;
}

// U = Psi_alpha^{-1}(w), w = (wbits + 1/2) 2^-32, by one converged warp: every lane
// passes the same P (from usample_setup) and wbits and returns U.  Work in
// t = a+ - u (Psi decreases in t) with the gap g(t) = log w - log Psi (lower half
// of w) or log(1 - Psi) - log(1 - w) (upper half), increasing in t and >= 0
// exactly when Psi(a+ - t) <= w:
//  1. bracket: the 32 candidates t_k = s0 2^(k/2 - 11) (the paper's doubling of the
//     bracket, two steps per octave, all at once), s0 = 1/max(1, |a-|) the residual's scale;
//     where the root lies outside them, once more with 32 further up (to s0 2^24) or down;
//  2. rounds of 32-point multisection, the bracket's ends among the points, until it is at
//     most kUHermiteWidth wide: one round for t up to 4.5;
//  3. the root of the cubic that interpolates t(g) at both ends with its slopes, 1/g' with
//     g' = psi / Psi (or psi / (1 - Psi)), the density in closed form (usample_log_density).
// The cubic's error falls with the fourth power of the width: at 0.05 it is below 6e-8 over
// |Delta| in [1e-2, 40], log alpha in [-20, 0] (against bisection in 64 bits), less than
// fp32 log Psi itself gives; at 0.1 up to 8e-7.  Each evaluation of the gap is a chain of
// about a microsecond: three 32-point rounds and a Newton step took 4.9 us a draw.
constexpr float kUHermiteWidth = 0.05f;
constexpr int kUMaxRounds = 8;

template <typename Coop>
__device__ __forceinline__ float usample_warp(const UParams& P, uint32_t wbits, uint32_t* status, Coop& co) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const bool upper = wbits >= 0x80000000u;
  const float target = upper ? logf(((float)(0xFFFFFFFFu - wbits) + 0.5f) * 0x1p-32f)
                             : logf(((float)wbits + 0.5f) * 0x1p-32f);
  auto gap = [&](float t) -> float {
    if (upper) return usample_log_1mpsi(t, P, co) - target;
    return target - usample_log_psi(t, P, co);
  };
  const float s0 = frcp_fast(fmaxf(1.0f, fabsf(P.am)));
  float t = s0 * exp2f(0.5f * (float)lane - 11.0f);
  float gt = gap(t);
  unsigned m = __ballot_sync(FULL, gt >= 0.0f);
  if (m == 0u) {                              // lane 0 is the highest candidate so far
    t = s0 * exp2f(fmaf((float)lane, 19.5f / 31.0f, 4.5f));
    gt = gap(t);
    m = __ballot_sync(FULL, gt >= 0.0f) & ~1u;
    if (m == 0u) {
      *status |= 4u;  // SDV_STATUS_USAMPLE_RANGE
      return P.ap - s0 * exp2f(24.0f);
    }
  } else if (m & 1u) {                        // lane 31 is the lowest candidate so far
    t = s0 * exp2f((float)lane - 42.0f);
    gt = gap(t);
    m = __ballot_sync(FULL, gt >= 0.0f) | 0x80000000u;
    if (m & 1u) return P.ap;                  // t below 2^-42 of the scale
  }
  float lo, hi, glo, ghi;
  auto narrow = [&] {                         // to the points around the first t with gap >= 0
    const int f = __ffs(m) - 1;
    hi = __shfl_sync(FULL, t, f);
    ghi = __shfl_sync(FULL, gt, f);
    lo = __shfl_sync(FULL, t, f - 1);
    glo = __shfl_sync(FULL, gt, f - 1);
  };
  narrow();
#pragma unroll 1
  for (int r = 0; r < kUMaxRounds; ++r) {
    t = lane == 31 ? hi : fmaf((float)lane * (1.0f / 31.0f), hi - lo, lo);
    gt = gap(t);                              // every lane evaluates (converged votes)
    if (lane == 0) gt = glo;                  // the ends keep their known values
    if (lane == 31) gt = ghi;
    m = __ballot_sync(FULL, gt >= 0.0f && lane > 0) | 0x80000000u;
    narrow();
    if (hi - lo <= kUHermiteWidth) break;
  }
  // slopes at both ends: log psi at every lane's own point, taken from the ends' lanes
  const float lpsi = usample_log_density(t, P);
  const int f = __ffs(m) - 1;
  const float l0 = __shfl_sync(FULL, lpsi, f - 1), l1 = __shfl_sync(FULL, lpsi, f);
  const float d0 = expf(l0 - (upper ? glo + target : target - glo));
  const float d1 = expf(l1 - (upper ? ghi + target : target - ghi));
  const float T = hi - lo, dg = ghi - glo;
  const float x = fminf(fmaxf(__fdividef(-glo, dg), 0.0f), 1.0f);
  const float m0 = __fdividef(dg, d0), m1 = __fdividef(dg, d1);
  float o = x * (m0 + x * ((3.0f * T - 2.0f * m0 - m1) + x * (m0 + m1 - 2.0f * T)));
  o = isfinite(o) ? fminf(fmaxf(o, 0.0f), T) : x * T;
  // u = a+ - t from the end that was evaluated, so that U's rounding stays relative to |U|
  return (P.ap - lo) - o;
}

// ---------------------------------------------------------------- tickets
// Fetch-and-add of 1 with acquire-release semantics at GPU scope: the release
// publishes this thread's earlier writes, and the holder of the last ticket
// acquires every write released before it.
__device__ __forceinline__ unsigned int ticket_acq_rel(unsigned int* p) {
  unsigned int old;
  asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(old) : "l"(p) : "memory");
  return old;
}

// ---------------------------------------------------------------- element access
template <typename T> struct Elem;
template <> struct Elem<float> {
  static __device__ __forceinline__ float load(const float* p) { return __ldg(p); }
  static __device__ __forceinline__ void store(float* p, float v) { *p = v; }
};
template <> struct Elem<__nv_bfloat16> {
  static __device__ __forceinline__ float load(const __nv_bfloat16* p) {
    return __bfloat162float(__ldg(p));
  }
  static __device__ __forceinline__ void store(__nv_bfloat16* p, float v) {
    *p = __float2bfloat16_rn(v);
  }
};

}  // namespace sdv
