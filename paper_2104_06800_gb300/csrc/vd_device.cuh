// Device-side building blocks of the dense-indirect EM: the Philox counter
// RNG, the Fisk residual energy, bilinear flow sampling and the per-pixel
// energy E_j(rho) of the depth M-step (Eq. 5 of VOLDOR+, Sec. III-A).
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "vd_internal.h"

#define VD_LN2 0.69314718055994530942f

// ---------------------------------------------------------------------------
// Checked build (-DVD_CHECKED; the stand-in for a memory checker): every
// index a kernel forms from data is checked against its buffer; the first
// index out of range is recorded (site, index, bound) with a count of all,
// and the index is clamped into range so that the access stays inside its
// buffer (the results are then wrong and the call reports it).  Each
// translation unit has its own record; vd_check_report gathers them.
// Without the flag VD_CHK is the index itself.
// ---------------------------------------------------------------------------
#ifdef VD_CHECKED
static __device__ unsigned long long g_vd_check[4];
__device__ __forceinline__ long long vd_checked(int site, long long i, long long n) {
  if (i >= 0 && i < n) return i;
  if (atomicCAS(&g_vd_check[0], 0ull, (unsigned long long)site) == 0ull) {
    g_vd_check[1] = (unsigned long long)i;
    g_vd_check[2] = (unsigned long long)n;
  }
  atomicAdd(&g_vd_check[3], 1ull);
  return i < 0 ? 0 : (n > 0 ? n - 1 : 0);
}
#define VD_CHK(site, i, n) vd_checked((site), (long long)(i), (long long)(n))
// host accessor of this unit's record: copies it to out[4] and clears it
#define VD_CHECK_ACCESSOR(name)                                                  \
  cudaError_t vd_check_take_##name(unsigned long long* out) {                    \
    cudaError_t e = cudaMemcpyFromSymbol(out, g_vd_check, 4 * sizeof(unsigned long long)); \
    const unsigned long long z[4] = {0, 0, 0, 0};                                \
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_vd_check, z, sizeof z);       \
    return e;                                                                    \
  }
#else
#define VD_CHK(site, i, n) (i)
#define VD_CHECK_ACCESSOR(name)                                                  \
  cudaError_t vd_check_take_##name(unsigned long long* out) {                    \
    for (int i = 0; i < 4; ++i) out[i] = 0;                                      \
    return cudaSuccess;                                                          \
  }
#endif
// sites of the checked build
enum { VD_SITE_BILINEAR = 1, VD_SITE_P3P_TAPS = 2, VD_SITE_SCATTER = 3, VD_SITE_PICK = 4,
       VD_SITE_VC_CELL = 5, VD_SITE_CHAIN = 6 };

// First statement of every kernel launched with vd_launch: waits for the
// kernel before it (at once when the launch did not overlap it), then lets
// the next one be placed.  An overlapped kernel exists while its predecessor
// still writes, so its inputs are not read-only for its lifetime, which is
// what `const __restrict__` tells the compiler: it may then load them by the
// non-coherent path and before the wait.  Every such parameter is therefore
// passed here, and its value comes out of the wait as one the compiler knows
// nothing about.  Explicit __ldg stay for the flows, priors and rigidness: a
// launch that does not overlap (the E-step's confidence, a copy) stands between
// their writer and every reader.
template <typename T>
__device__ __forceinline__ void vd_pdl_hide(T& p) {
  size_t a = __cvta_generic_to_global(p);
  asm volatile("" : "+l"(a));
  p = reinterpret_cast<T>(__cvta_global_to_generic(a));
}
template <typename... T>
__device__ __forceinline__ void vd_pdl_begin(T&... inputs) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  (vd_pdl_hide(inputs), ...);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon et al., SC'11): ten rounds of two 32x32->64 bit
// multiplies, mixing with the key, key advanced by the Weyl constants.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 vd_philox(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint64_t p0 = (uint64_t)0xD2511F53u * c.x;   // one wide multiply per product
    const uint64_t p1 = (uint64_t)0xCD9E8D57u * c.z;
    const uint32_t hi0 = (uint32_t)(p0 >> 32), lo0 = (uint32_t)p0;
    const uint32_t hi1 = (uint32_t)(p1 >> 32), lo1 = (uint32_t)p1;
    c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return c;
}

__device__ __forceinline__ uint32_t vd_word(const uint4& w, int i) {
  return i == 0 ? w.x : (i == 1 ? w.y : (i == 2 ? w.z : w.w));
}

// (x >> 8) * 2^-24 as float (exact).
__device__ __forceinline__ float vd_u24(uint32_t x) {
  return __fmul_rn(__uint2float_rn(x >> 8), 5.9604644775390625e-8f);
}

// Hypothesis values, each operation rounded once (no contraction), so the
// float32 values are reproducible bit for bit.
__device__ __forceinline__ float vd_cand_uniform(uint32_t x, float rmin, float range) {
  return __fadd_rn(rmin, __fmul_rn(vd_u24(x), range));
}
__device__ __forceinline__ float vd_cand_perturb(uint32_t x, float rho, float s) {
  const float a = __fsub_rn(__fmul_rn(2.0f, vd_u24(x)), 1.0f);
  return __fmul_rn(rho, __fadd_rn(1.0f, __fmul_rn(s, a)));
}
__device__ __forceinline__ float vd_clamp(float c, float lo, float hi) {
  return fminf(fmaxf(c, lo), hi);
}

// ---------------------------------------------------------------------------
// Residual energy l = log(1 + P0 / p1(r)), p1 = density of a 2-D residual
// vector whose length is Fisk(alpha, beta) distributed and whose direction is
// uniform.  Returned in log2 units (multiply by ln 2).  Also returns
// y = P0 / p1 (the outlier-to-rigid likelihood ratio) for the E-step.
// ---------------------------------------------------------------------------
// 1 / x and log2 x of the special-function unit for x in float32's normal
// range: __fdividef and __log2f less the instructions that rescale subnormals
// (the same bits; three to four instructions fewer per call).
__device__ __forceinline__ float vd_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float vd_ex2(float x) {   // 0 below 2^-126
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float vd_lg2(float x) {
  float r;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Two float32 values in one 64-bit register pair.  The packed instructions
// round each half exactly as the scalar ones do, and cost one issue slot for
// both: what the issue-bound kernels (depth sampling, pose scoring) use them
// for.
typedef unsigned long long vd_f2;
__device__ __forceinline__ vd_f2 vd_pack(float lo, float hi) {
  vd_f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void vd_unpack(vd_f2 a, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a));
}
__device__ __forceinline__ vd_f2 vd_fma2(vd_f2 a, vd_f2 b, vd_f2 c) {
  vd_f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ vd_f2 vd_mul2(vd_f2 a, vd_f2 b) {
  vd_f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ vd_f2 vd_add2(vd_f2 a, vd_f2 b) {
  vd_f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ vd_f2 vd_sub2(vd_f2 a, vd_f2 b) {
  vd_f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// a / b of each half from ib = 1 / b rounded and nb = -b: the first quotient and
// its remainder (P. Markstein, IBM J. Res. Dev. 34(1), 1990).  The bits of a
// division, but for exact quotients within 2^-23 of a last place of a rounding
// boundary, in three packed operations.
__device__ __forceinline__ vd_f2 vd_div2(vd_f2 a, vd_f2 nb, vd_f2 ib) {
  const vd_f2 q = vd_mul2(a, ib);
  return vd_fma2(vd_fma2(q, nb, a), ib, q);
}

__device__ __forceinline__ float vd_lo(vd_f2 a) { return __uint_as_float((unsigned)a); }
__device__ __forceinline__ float vd_hi(vd_f2 a) { return __uint_as_float((unsigned)(a >> 32)); }

__device__ __forceinline__ float vd_ratio_general(const DevParams& P, float r2, float alpha) {
  float r = sqrtf(r2);
  if (P.beta != 2.0f) r = fmaxf(r, VD_R_FLOOR);
  const float s = r / alpha;
  const float ls = __log2f(s);
  const float sb = exp2f(P.beta * ls);
  // s^(2 - beta); with beta = 2 it is 1 at s = 0 and s = inf too (0 * inf is not)
  const float lsz = P.beta == 2.0f ? 0.0f : ls;
  const float s2b = exp2f((2.0f - P.beta) * lsz);
  const float one = 1.0f + sb;
  return P.cgen * alpha * alpha * s2b * one * one;
}

__device__ __forceinline__ float vd_ratio_y(const DevParams& P, float r2, float fmag2) {
  if (P.fast_beta2) {
    // beta = 2: P0 / p1 = P0 pi alpha^2 (1 + r^2 / alpha^2)^2
    const float s = fmaf(r2, P.inv_a2, 1.0f);
    return P.c0 * s * s;
  }
  return vd_ratio_general(P, r2, fmaf(P.alpha1, sqrtf(fmag2), P.alpha0));
}

// log2(1 + y).  Near the optimum y = P0 pi alpha^2 (1 + s^2)^2 is ~1e-3 and
// the MUFU log2 of 1 + y (absolute error ~2^-22) would lose most digits of
// the residual-dependent part, so small y uses the series
// ln(1 + y) = y - y^2/2 + y^3/3 - y^4/4 + y^5/5 (truncation < y^6/6).
__device__ __forceinline__ float vd_ell2(float y) {
  const float big = vd_lg2(1.0f + y);
  const float ser =
      y * fmaf(y, fmaf(y, fmaf(y, fmaf(y, 0.2f, -0.25f), 0.33333334f), -0.5f), 1.0f) *
      1.44269504f;
  return y < 0.03125f ? ser : big;
}

// log2(1 + P0 / p1) of a residual with r2 = r^2 and Fisk scale alpha.  Where
// the ratio y = P0 / p1 would overflow float32 (a residual of ~1e10 px and
// beyond), log2(1 + y) equals log2 y to float32 precision and is taken in the
// log domain; below that the value is vd_ell2(y).
__device__ __forceinline__ float vd_l2_general(const DevParams& P, float r2, float alpha) {
  float r = sqrtf(r2);
  if (P.beta != 2.0f) r = fmaxf(r, VD_R_FLOOR);
  const float s = r / alpha;
  const float ls = __log2f(s);
  const float sb = exp2f(P.beta * ls);
  // s^(2 - beta); with beta = 2 it is 1 at s = 0 and s = inf too (0 * inf is not)
  const float lsz = P.beta == 2.0f ? 0.0f : ls;
  const float s2b = exp2f((2.0f - P.beta) * lsz);
  const float one = 1.0f + sb;
  const float y = P.cgen * alpha * alpha * s2b * one * one;
  if (y < 1e30f) return vd_ell2(y);
  const float l1 = sb < 1e30f ? __log2f(one) : P.beta * ls;   // log2(1 + s^beta)
  return __log2f(P.cgen * alpha * alpha) + (2.0f - P.beta) * lsz + 2.0f * l1;
}

__device__ __forceinline__ float vd_l2_beta2(const DevParams& P, float r2) {
  // beta = 2: P0 / p1 = P0 pi alpha^2 (1 + r^2 / alpha^2)^2
  const float s = fmaf(r2, P.inv_a2, 1.0f);
  const float y = __fmul_rn(__fmul_rn(P.c0, s), s);
  // one logarithm and no branch: of 1 + y, or of s where y would overflow
  const bool mid = y < 1e30f;
  const float L = vd_lg2(mid ? __fadd_rn(1.0f, y) : s);
  const float ser =
      y * fmaf(y, fmaf(y, fmaf(y, fmaf(y, 0.2f, -0.25f), 0.33333334f), -0.5f), 1.0f) *
      1.44269504f;
  return y < 0.03125f ? ser : (mid ? L : fmaf(2.0f, L, P.log2c0));
}

// The flow term's log2(1 + P0 / p1): alpha = alpha0 + alpha1 |X_t(x)|.
__device__ __forceinline__ float vd_l2_flow(const DevParams& P, float r2, float fmag2) {
  if (P.fast_beta2) return vd_l2_beta2(P, r2);
  return vd_l2_general(P, r2, fmaf(P.alpha1, sqrtf(fmag2), P.alpha0));
}

// ---------------------------------------------------------------------------
// Entry i of a frame's rows K [R | tau] from its float64 value: float32 for
// the depth and pose kernels, and as a double-float pair (hi, lo; hi + lo is
// the float64 value to 48 bits) for the rigidness emissions.  Every writer
// of the pose rows stores both.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void vd_store_pose_entry(float* __restrict__ pf, float2* __restrict__ pd,
                                                    int i, double v) {
  const float hi = (float)v;
  pf[i] = hi;
  pd[i] = make_float2(hi, (float)(v - (double)hi));
}

// ---------------------------------------------------------------------------
// Bilinear sample of one flow field at (x, y), which must be inside the image.
// Taps (x0, y0)..(x0+1, y0+1) with x0 = min(floor(x), W-2).
// ---------------------------------------------------------------------------
//
// Both components go through packed arithmetic (vd_f2).  The floors come from
// one packed addition of 2^23 rounded towards zero, which leaves floor(x) in
// the low bits of each half for 0 <= x < 2^23 (images are at most 16384 wide
// and high), in place of two conversions to integer and two back.
__device__ __forceinline__ vd_f2 vd_bilinear2(const float2* __restrict__ F, int W, int H,
                                              vd_f2 xy) {
  const unsigned B = 0x4b000000u;                  // the bits of 2^23
  const float two23 = 8388608.0f;
  vd_f2 fl;
  asm("add.rz.f32x2 %0, %1, %2;" : "=l"(fl) : "l"(xy), "l"(vd_pack(two23, two23)));
  const unsigned x0 = min((unsigned)fl, B + (unsigned)(W - 2));
  const unsigned y0 = min((unsigned)(fl >> 32), B + (unsigned)(H - 2));
  const vd_f2 a = vd_sub2(xy, vd_sub2(vd_pack(__uint_as_float(x0), __uint_as_float(y0)),
                                      vd_pack(two23, two23)));
  // y0 W + x0 without the two 2^23 patterns, modulo 2^32
  const unsigned i = y0 * (unsigned)W + (x0 - B * ((unsigned)W + 1u));
  const float2* p = F + VD_CHK(VD_SITE_BILINEAR, (long long)i, (long long)W * H - W - 1);
  const vd_f2* p0 = reinterpret_cast<const vd_f2*>(p);
  const vd_f2* p1 = reinterpret_cast<const vd_f2*>(p + W);
  const vd_f2 f00 = __ldg(p0), f01 = __ldg(p0 + 1);
  const vd_f2 f10 = __ldg(p1), f11 = __ldg(p1 + 1);
  const vd_f2 ax = vd_pack(vd_lo(a), vd_lo(a)), ay = vd_pack(vd_hi(a), vd_hi(a));
  const vd_f2 t = vd_fma2(ax, vd_sub2(f01, f00), f00);
  const vd_f2 b = vd_fma2(ax, vd_sub2(f11, f10), f10);
  return vd_fma2(ay, vd_sub2(b, t), t);
}
__device__ __forceinline__ float2 vd_bilinear(const float2* __restrict__ F, int W, int H, float x,
                                              float y) {
  const vd_f2 r = vd_bilinear2(F, W, H, vd_pack(x, y));
  return make_float2(vd_lo(r), vd_hi(r));
}

__device__ __forceinline__ bool vd_inside(float x, float y, int W, int H) {
  return x >= 0.0f && x <= (float)(W - 1) && y >= 0.0f && y <= (float)(H - 1);
}

// ---------------------------------------------------------------------------
// Per-pixel constant part of the energy.  A_t = K R_t r_j (homogeneous image
// point of the ray), B_t = K tau_t is shared by all pixels (shared memory).
// ---------------------------------------------------------------------------
template <int NF>
struct VdPixel {
  float ax[NF], ay[NF], az[NF];
  float wl[NF];           // q_t * ln 2
  float f1x, f1y;         // X_1 at the pixel (x_0 = j exactly)
  float u, v;
  float pv;               // prior value (disparity or rho_hat)
  float pw;               // prior weight q_hat * conf (0 at holes / no prior)
};

// posef layout per frame t (0..N): 9 floats K R_t (row-major), 3 floats K tau_t.
template <int NF>
__device__ __forceinline__ void vd_pixel_setup(VdPixel<NF>& px, const DevParams& P,
                                               const float* __restrict__ sPose, int u, int v,
                                               const float* __restrict__ q, size_t npix, size_t j,
                                               const float2* __restrict__ flow,
                                               const float* __restrict__ prior_val,
                                               const float* __restrict__ qhat,
                                               const float* __restrict__ pconf) {
  const float rx = ((float)u - P.cx) / P.fx;
  const float ry = ((float)v - P.cy) / P.fy;
#pragma unroll
  for (int t = 0; t < NF; ++t) {
    const float* M = sPose + 12 * (t + 1);
    px.ax[t] = fmaf(M[0], rx, fmaf(M[1], ry, M[2]));
    px.ay[t] = fmaf(M[3], rx, fmaf(M[4], ry, M[5]));
    px.az[t] = fmaf(M[6], rx, fmaf(M[7], ry, M[8]));
    px.wl[t] = __ldg(q + (size_t)t * npix + j) * VD_LN2;
  }
  const float2 f1 = __ldg(flow + j);
  px.f1x = f1.x;
  px.f1y = f1.y;
  px.u = (float)u;
  px.v = (float)v;
  px.pw = 0.0f;
  px.pv = 0.0f;
  if (P.prior_kind != VD_PRIOR_NONE) {
    const float pvv = __ldg(prior_val + j);
    if (isfinite(pvv)) {
      px.pv = pvv;
      px.pw = __ldg(qhat + j) * __ldg(pconf + j);
    }
  }
}

// Prior term w_hat l_hat(c) of E_j (0 where the pixel has no prior).
template <int NF>
__device__ __forceinline__ float vd_prior_energy(const VdPixel<NF>& px, const DevParams& P,
                                                 float c) {
  if (!(px.pw > 0.0f)) return 0.0f;
  if (P.prior_kind == VD_PRIOR_STEREO) {
    const float d = px.pv - P.fxb * c;
    const float l2 = P.beta == 2.0f ? vd_l2_beta2(P, d * d) : vd_l2_general(P, d * d, P.alpha0);
    return px.pw * VD_LN2 * l2;
  }
  const float res = px.pv - c;
  const float sig = P.c_sigma * px.pv;
  const float z = fmaf(res * res, 0.5f / (sig * sig), P.logk);
  return px.pw * (z > 20.0f ? z : VD_LN2 * vd_ell2(__expf(z)));
}

// One flow term in log2 units.  (h, hz): homogeneous image point of the
// candidate in frame t, x and y packed; xyp: its image point in frame t-1,
// where the flow F was read; obs: the point is in front of camera t-1 and
// inside image t-1.  Writes the image point in frame t and whether it is in
// front of camera t.  Without a branch: a term is almost always observed, and
// what is not is discarded.  FAST: the launch's constants (beta = 2, one
// scale for all pixels).  POS: the window's last flow has an image point that
// nothing else reads; its products are scalar, since the compiler fuses a
// packed product into the packed difference that alone uses it.  The only flow
// of a window (and of the bootstrap's own depth) has that displacement in one
// multiply-add.
enum { VD_TERM_INNER = 0, VD_TERM_LAST = 1, VD_TERM_ONLY = 2 };
template <bool FAST, int POS>
__device__ __forceinline__ float vd_flow_term2(const DevParams& P, vd_f2 h, float hz, bool obs,
                                               vd_f2 F, vd_f2 xyp, vd_f2* xy_out,
                                               bool* front_out) {
  const bool front = hz > VD_Z_EPS;
  const float r = vd_rcp(hz);
  *xy_out = POS == VD_TERM_LAST ? vd_pack(__fmul_rn(vd_lo(h), r), __fmul_rn(vd_hi(h), r))
                                : vd_mul2(h, vd_pack(r, r));
  *front_out = front;
  const vd_f2 d =
      vd_sub2(F, POS == VD_TERM_ONLY
                     ? vd_fma2(h, vd_pack(r, r), vd_pack(-vd_lo(xyp), -vd_hi(xyp)))
                     : vd_sub2(*xy_out, xyp));
  const float dx = vd_lo(d), dy = vd_hi(d);
  const float r2 = fmaf(dx, dx, dy * dy);
  float l2;
  if (FAST) {
    l2 = vd_l2_beta2(P, r2);
  } else {
    const float Fx = vd_lo(F), Fy = vd_hi(F);
    l2 = vd_l2_general(P, r2, fmaf(P.alpha1, sqrtf(fmaf(Fx, Fx, Fy * Fy)), P.alpha0));
  }
  return obs ? (front ? l2 : VD_L_BEHIND / VD_LN2) : 0.0f;
}

// E_j(c) in full, for latency-bound callers (the chain propagation): every
// frame's projection first, then every gathered flow's taps (all loads in
// flight together), then the terms in the order and arithmetic of
// vd_energy, so the value is vd_energy's without a bound.  A caller that
// compares the result with a bound gets vd_energy's decision (an early
// exit there returns a partial sum already at or above it).
template <int NF>
__device__ __forceinline__ float vd_energy_full(const VdPixel<NF>& px, const DevParams& P,
                                                const float* __restrict__ sPose,
                                                const float2* __restrict__ flow, size_t npix,
                                                float c) {
  float xs[NF], ys[NF];
  bool fr[NF];
#pragma unroll
  for (int t = 0; t < NF; ++t) {   // projection into frame t + 1 (as vd_flow_term2 forms it)
    const float* M = sPose + 12 * (t + 1);
    const float hx = fmaf(c, M[9], px.ax[t]);
    const float hy = fmaf(c, M[10], px.ay[t]);
    const float hz = fmaf(c, M[11], px.az[t]);
    fr[t] = hz > VD_Z_EPS;
    const float iz = __fdividef(1.0f, hz);
    xs[t] = hx * iz;
    ys[t] = hy * iz;
  }
  // flow t is read at the pixel's position in frame t; every position is
  // bounded first and every tap loaded without a branch (a branch per flow
  // would wait for its loads before it issues the next flow's)
  float2 f00[NF], f01[NF], f10[NF], f11[NF];
  float wx[NF], wy[NF];
  bool ob[NF];
  ob[0] = true;
#pragma unroll
  for (int t = 1; t < NF; ++t) {
    ob[t] = fr[t - 1] && vd_inside(xs[t - 1], ys[t - 1], P.W, P.H);
    const float x = ob[t] ? xs[t - 1] : 0.0f, y = ob[t] ? ys[t - 1] : 0.0f;
    const int x0 = min(__float2int_rd(x), P.W - 2);
    const int y0 = min(__float2int_rd(y), P.H - 2);
    wx[t] = x - (float)x0;
    wy[t] = y - (float)y0;
    const float2* p = flow + (size_t)t * npix +
                      VD_CHK(VD_SITE_BILINEAR, (long long)y0 * P.W + x0,
                             (long long)P.W * P.H - P.W - 1);
    f00[t] = __ldg(p);
    f01[t] = __ldg(p + 1);
    f10[t] = __ldg(p + P.W);
    f11[t] = __ldg(p + P.W + 1);
  }
  float E = vd_prior_energy<NF>(px, P, c);
#pragma unroll
  for (int t = 0; t < NF; ++t) {
    const float xp = t == 0 ? px.u : xs[t - 1], yp = t == 0 ? px.v : ys[t - 1];
    float2 F = make_float2(px.f1x, px.f1y);
    if (t > 0) {
      const float tx = fmaf(wx[t], f01[t].x - f00[t].x, f00[t].x);
      const float ty = fmaf(wx[t], f01[t].y - f00[t].y, f00[t].y);
      const float bx = fmaf(wx[t], f11[t].x - f10[t].x, f10[t].x);
      const float by = fmaf(wx[t], f11[t].y - f10[t].y, f10[t].y);
      F = make_float2(fmaf(wy[t], bx - tx, tx), fmaf(wy[t], by - ty, ty));
    }
    const float dx = F.x - (xs[t] - xp);
    const float dy = F.y - (ys[t] - yp);
    const float r2 = fmaf(dx, dx, dy * dy);
    const float l = vd_l2_flow(P, r2, fmaf(F.x, F.x, F.y * F.y));
    E = fmaf(px.wl[t], ob[t] && fr[t] ? l : (ob[t] ? (VD_L_BEHIND / VD_LN2) : 0.0f), E);
  }
  return E;
}

// E_j(c): sum_t q_t l_t(c) + w_hat l_hat(c) in natural-log units.
// Every term is non-negative, so once the partial sum reaches `bound` the
// candidate cannot beat an energy of `bound`: the sum stops there and the
// partial value (>= bound) is returned.  The cheap terms come first: the
// prior, then X_1 (read at the pixel itself), then the gathered flows.
template <int NF>
__device__ __forceinline__ float vd_energy(const VdPixel<NF>& px, const DevParams& P,
                                           const float* __restrict__ sPose,
                                           const float2* __restrict__ flow, size_t npix,
                                           float c, float bound = INFINITY) {
  float E = vd_prior_energy<NF>(px, P, c);
  vd_f2 xyp = vd_pack(px.u, px.v);
  bool front_prev = true;
#pragma unroll
  for (int t = 0; t < NF; ++t) {
    if (E >= bound) return E;
    const float* M = sPose + 12 * (t + 1);
    const vd_f2 h = vd_pack(fmaf(c, M[9], px.ax[t]), fmaf(c, M[10], px.ay[t]));
    const float hz = fmaf(c, M[11], px.az[t]);
    bool obs = true;
    vd_f2 F = vd_pack(px.f1x, px.f1y);
    if (t > 0) {
      obs = front_prev && vd_inside(vd_lo(xyp), vd_hi(xyp), P.W, P.H);
      F = 0;
      if (obs) F = vd_bilinear2(flow + (size_t)t * npix, P.W, P.H, xyp);
    }
    vd_f2 xy;
    bool front;
    float l2;
    constexpr int END = NF == 1 ? VD_TERM_ONLY : VD_TERM_LAST;
    if (t == NF - 1)
      l2 = P.fast_beta2 ? vd_flow_term2<true, END>(P, h, hz, obs, F, xyp, &xy, &front)
                        : vd_flow_term2<false, END>(P, h, hz, obs, F, xyp, &xy, &front);
    else
      l2 = P.fast_beta2 ? vd_flow_term2<true, VD_TERM_INNER>(P, h, hz, obs, F, xyp, &xy, &front)
                        : vd_flow_term2<false, VD_TERM_INNER>(P, h, hz, obs, F, xyp, &xy, &front);
    E = fmaf(px.wl[t], l2, E);
    xyp = xy;
    front_prev = front;
  }
  return E;
}
