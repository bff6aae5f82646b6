// Adjoint of the GPP sum in FP64 (gpp_sigma_backward).
//
// The loss seen by the adjoint is L with dL = Re(sum_iw conj(g_ach[iw]) d achtemp[iw] +
// conj(g_asx[iw]) d asxtemp[iw]) (PyTorch's convention for complex outputs). With
// c_a = conj(g_ach), c_s = conj(g_asx) and the per-term weight M = am * aqsntemp (am =
// conj(aqsmtemp[b][g]) vcoul[g]), every (b, p, ig) contributes M Q to L, where
//   Q   = I w GI,   GI = sum_iw  c_a [b1] u  +  c_s occ (b1 ? w u v : -v/2)
//   dQ/dw-part:     GW = sum_iw  c_a [b1] x u^2  +  c_s occ (b1 ? 2 x^2 w (u v)^2 : -x v^2 / 2)
// with u = 1/(x - w), v = 1/(x + w) (so w u = delw, w^2 u v = w^2/(x^2 - w^2)); these are the
// derivatives of the branch formulas (the branch predicates are locally constant). Then
//   grad wtilde[p][ig]   = conj( sum_b M I GW )         (holomorphic input)
//   grad I_eps[p][ig]    = conj( sum_b M w GI )
//   grad aqsntemp[b][ig] = conj( sum_p am Q )
//   grad aqsmtemp[b][g]  = vcoul[g] sum_{p: g(p) = g} sum_ig aqsntemp[b][ig] Q   (enters
//                          through its conjugate, so no outer conj)
// Terms are recomputed, not stored. One reciprocal r = 1/(|x-w|^2 |x+w|^2) per term gives
// u = conj(x-w)|x+w|^2 r, v = conj(x+w)|x-w|^2 r and u v = conj(x^2-w^2) r.
//
// Decomposition: a CTA owns a tile of 8 columns (one per warp) x 32 G-vectors (one per lane),
// one (p, ig) pair per thread, and walks every band. wtilde / I_eps gradients stay in
// registers. Every kRedBands bands, the CTA sums am Q over its 8 columns and aqsntemp Q over
// its 32 G-vectors from shared memory in a fixed order and writes one partial per tile; columns
// are processed in batches of column groups per launch, and a finishing kernel adds each
// batch's partials into the outputs in a fixed order. No atomics: results are deterministic.
//
// Split-integer form. Warps in the range of the forward's split-integer form
// (gpp_terms_fix.cuh) take u and v from there (U + gamma), with the cotangent products as
// 31-bit integers and remainders. With x u = 1 + w u and x v = 1 - w v, on the fast path
//   GI = sum_iw cap u + csh v,   GW = GI + w H,   H = sum_iw cap u^2 - csh v^2
// (cap = c_a + c_s/2, csh = -c_s/2; the bands outside asxtemp: c_a and no v), so a term adds
// u and u^2 (squared in 64 bits) to 62-bit sums GI and H, which are multiplied by M and summed
// over the bands as in the forward:
//   grad I_eps = conj(w sum_b M GI),   grad wtilde = conj(I (sum_b M GI + w sum_b M H)).
// Q and its two weighted sums stay FP64 (21 FP64 instructions per unit, which run beside the
// integer work; the FP64 form has 141). Bound: dispatch of the integer and FP32 instructions
// (ALU 315, FMA pipe 665 per unit and 32 lanes), with the FP64 pipe 56% busy and its latency on
// top. B = 128, P = 410, G = 8192, nw = 3: 26.0 ms (FP64 form 108.3; 25.6 without the tests that
// send entries far below their scale to FP64, see kWeakBand).

#include <cuda_runtime.h>

#include "gpp_device.cuh"
#include "gpp_internal.h"
#include "gpp_terms_fix.cuh"

namespace gpp {

namespace {

constexpr int kTX = 32;  // G-vectors per tile
constexpr int kTY = 8;   // columns per tile (one column group)

// One (band, iw) entry for the adjoint: x, x^2 and the cotangent products that do not
// depend on (p, ig): c_a + c_s / 2 and its product with x (the fast path's partial
// fractions), c_a, c_s, c_a x, -c_s / 2, -x c_s / 2.
struct alignas(32) BwdBand {
  double2 lo;     // x, x^2
  double2 cap;    // c_a + c_s / 2
  double2 ca;     // c_a
  double2 cs;     // c_s
  double2 cax;    // c_a x
  double2 capx;   // (c_a + c_s / 2) x
  double2 csh;    // -c_s / 2
  double2 csxh;   // -x c_s / 2
};

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
// acc += a * b
__device__ __forceinline__ void cmac(double2& acc, double2 a, double2 b) {
  acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
  acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
}
__device__ __forceinline__ double2 csel(bool c, double2 a, double2 b) { return c ? a : b; }

template <bool V>
struct BoolTag {
  static constexpr bool value = V;
};

// A cotangent product for the split-integer form: c = (r1 + r0, i1 + i0) 2^(ec - 31), with
// the negatives and the FP32 value of the integer part.
struct alignas(16) FixC {
  int r1, i1, nr1, ni1;
  float r0, i0, r1f, i1f;
};
// The cotangent products of every frequency; ok: finite and of ordinary exponent. The bands of
// asxtemp (0: cap and csh) and the others (1: ca) have a scale each, since rows of the gradients
// belong to one of them alone: the sums of the moduli, sum_c of cap or ca and sum_s of csh, over
// 2^ec, add up to less than 1 - 2^-21.
// cap2, csh2, ca2: their squared moduli over 2^(2 ec), above zero for one that is not zero; spread:
// branch 2 may leave a band with far smaller ones than the scale is for (csh never drops out).
struct FixBwd {
  int ok, ec[2], spread[2];
  float sum_c[2], sum_s;
  float cap2[kMaxNw], csh2[kMaxNw], ca2[kMaxNw];
  FixC cap[kMaxNw], csh[kMaxNw], ca[kMaxNw];
};
static_assert(sizeof(FixBwd) <= 1024, "workspace segment of the cotangent products");

__device__ inline FixC fix_c(double2 c, int ec) {
  const double sr = c.x * exp2i(31 - ec), si = c.y * exp2i(31 - ec);
  const double rr = rint(sr), ri = rint(si);
  FixC o;
  o.r1 = static_cast<int>(rr);
  o.i1 = static_cast<int>(ri);
  o.nr1 = -o.r1;
  o.ni1 = -o.i1;
  o.r0 = static_cast<float>(sr - rr);
  o.i0 = static_cast<float>(si - ri);
  o.r1f = static_cast<float>(rr);
  o.i1f = static_cast<float>(ri);
  return o;
}

__device__ inline float fix_c2(double2 c, int ec) {
  const float r = static_cast<float>(c.x * exp2i(-ec)), i = static_cast<float>(c.y * exp2i(-ec));
  return c.x == 0.0 && c.y == 0.0 ? 0.0f : fmaxf(fmaf(r, r, i * i), 1e-37f);
}

// One warp, a lane per frequency: the split-integer form's cotangent products.
__device__ inline void fix_cotangents(int W, const double2* g_ach, const double2* g_asx,
                                      double ach_scale, FixBwd* out) {
  const int iw = threadIdx.x;
  const double2 zero = make_double2(0.0, 0.0);
  const double2 ga = iw < W ? g_ach[iw] : zero, gs = iw < W ? g_asx[iw] : zero;
  const double2 ca = make_double2(ach_scale * ga.x, -ach_scale * ga.y);
  const double2 csh = make_double2(-0.5 * gs.x, 0.5 * gs.y);
  const double2 cap = make_double2(ca.x - csh.x, ca.y - csh.y);
  // (not from the squares: those of cotangents below 1e-162 are zero)
  auto total = [](double2 c) { return warp_sum(hypot(c.x, c.y)); };
  const double sa = total(ca), sc = total(cap), ss = total(csh);
  const double m[2] = {(sc + ss) * (1.0 + 0x1p-20), sa * (1.0 + 0x1p-20)};
  bool ok = true;
  int ec[2];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    ok = ok && (m[c] == 0.0 || (m[c] > 1e-90 && m[c] < 1e90));   // false for NaN
    ec[c] = m[c] == 0.0 ? 0 : ((__double2hiint(m[c]) >> 20) & 0x7ff) - 1022;
  }
  if (iw == 0) {
    out->ok = ok;
    out->ec[0] = ec[0];
    out->ec[1] = ec[1];
    out->sum_c[0] = ok ? static_cast<float>(sc * exp2i(-ec[0])) : 0.0f;
    out->sum_c[1] = ok ? static_cast<float>(sa * exp2i(-ec[1])) : 0.0f;
    out->sum_s = ok ? static_cast<float>(ss * exp2i(-ec[0])) : 0.0f;
  }
  // per frequency's share: the least squared modulus that is not zero against the sum of them all
  auto spread_of = [&](double2 c, double2 s, int e) {
    float least = fix_c2(c, e), all = 0.0f, never = fix_c2(s, e);
    least = least == 0.0f ? 3.0e38f : least;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      least = fminf(least, __shfl_xor_sync(0xffffffffu, least, o));
      never += __shfl_xor_sync(0xffffffffu, never, o);
    }
    all = warp_sumf(fix_c2(c, e)) + never;
    // (a small csh is what is left where branch 2 takes every cap; no csh leaves nothing)
    return ok && never < all * 0x1p-8f && (never > 0.0f || least < all * 0x1p-8f);
  };
  const bool spread0 = spread_of(cap, csh, ec[0]), spread1 = spread_of(ca, zero, ec[1]);
  if (iw == 0) {
    out->spread[0] = spread0;
    out->spread[1] = spread1;
  }
  if (ok && iw < W) {
    out->cap[iw] = fix_c(cap, ec[0]);
    out->csh[iw] = fix_c(csh, ec[0]);
    out->ca[iw] = fix_c(ca, ec[1]);
    out->cap2[iw] = fix_c2(cap, ec[0]);
    out->csh2[iw] = fix_c2(csh, ec[0]);
    out->ca2[iw] = fix_c2(ca, ec[1]);
  }
}

// ach_scale: 1/2 with the half Coulomb-hole factor (it scales every achtemp cotangent).
__global__ void gpp_bwd_prep_kernel(int64_t B, int W, const double* __restrict__ wx,
                                    const double2* __restrict__ g_ach,
                                    const double2* __restrict__ g_asx, double ach_scale,
                                    BwdBand* bt, FixBwd* fixc) {
  if (blockIdx.x == gridDim.x - 1) {   // a block of its own for the split-integer products
    if (threadIdx.x < 32) fix_cotangents(W, g_ach, g_asx, ach_scale, fixc);
    return;
  }
  const int64_t stride = static_cast<int64_t>(gridDim.x - 1) * blockDim.x;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < B * W;
       i += stride) {
    const int iw = static_cast<int>(i % W);
    const double x = wx[i];
    const double2 ga = g_ach[iw], gs = g_asx[iw];
    const double2 ca = make_double2(ach_scale * ga.x, -ach_scale * ga.y);
    const double2 cs = make_double2(gs.x, -gs.y);
    BwdBand e;
    e.lo = make_double2(x, x * x);
    e.cap = make_double2(ca.x + 0.5 * cs.x, ca.y + 0.5 * cs.y);
    e.ca = ca;
    e.cs = cs;
    e.cax = make_double2(ca.x * x, ca.y * x);
    e.capx = make_double2(e.cap.x * x, e.cap.y * x);
    e.csh = make_double2(-0.5 * cs.x, -0.5 * cs.y);
    e.csxh = make_double2(-0.5 * x * cs.x, -0.5 * x * cs.y);
    bt[i] = e;
  }
}

// z^2 for a complex z, with the doubling of the imaginary part on the integer pipe.
__device__ __forceinline__ double2 csq(double2 z) {
  return make_double2(fma(z.x, z.x, -z.y * z.y), twice_alu(z.x * z.y));
}

// Per-term work for one band, all frequencies, on the fast path (every lane of the warp has
// 1e-12 < |w|^2 < 62499 and Re w >= 0, every wx >= 0: branch 1 is exactly |x - w|^2 > 1/4,
// branch 3 and the screened-exchange cutoff cannot occur). In partial fractions, with
// u = 1/(x - w), v = 1/(x + w) and b1 the branch-1 predicate, the asxtemp parts are
// w u v = (u - v)/2 and -v/2 in GI, 2 x^2 w (u v)^2 = x (u^2 - v^2)/2 and -x v^2/2 in GW, so
//   GI = sum_iw (c_a + c_s/2) b1 u - (c_s/2) v,   GW = sum_iw (c_a + c_s/2) b1 x u^2 - (c_s/2) x v^2
// on occupied bands (c_a b1 u and c_a b1 x u^2 on the others): two reciprocals per term and
// a select on u only.
template <int W, bool OCC>
__device__ __forceinline__ void bwd_terms_fast(const BwdBand* __restrict__ e, double wr,
                                               double wi, double wi2, double2& GI,
                                               double2& GW) {
#pragma unroll
  for (int iw = 0; iw < W; ++iw) {
    const double x = __ldg(&e[iw].lo.x);
    const double Ar = x - wr;
    const double A2 = fma(Ar, Ar, wi2);
    const double ra = rcp_refined(A2);
    const bool c1 = gt_nonneg(A2, kLimitTwo);
    const double2 u = c1 ? make_double2(Ar * ra, wi * ra) : make_double2(0.0, 0.0);
    const double2 uu = csq(u);
    if (OCC) {
      const double Sr = x + wr;
      const double S2 = fma(Sr, Sr, wi2);        // >= |w|^2 > 1e-12
      const double rs = rcp_refined(S2);
      const double2 v = make_double2(Sr * rs, -wi * rs);
      cmac(GI, __ldg(&e[iw].cap), u);
      cmac(GI, __ldg(&e[iw].csh), v);
      cmac(GW, __ldg(&e[iw].capx), uu);
      cmac(GW, __ldg(&e[iw].csxh), csq(v));
    } else {
      cmac(GI, __ldg(&e[iw].ca), u);
      cmac(GW, __ldg(&e[iw].cax), uu);
    }
  }
}

// Per-term work for one band, all frequencies, in the general form: accumulates GI and GW.
// sx2: sexcut^2 of the screened-exchange cutoff, 0 = off; where it drops ssx (x < 0 and
// |ssx| / |I| > sexcut, tested as in the forward) the ssx derivatives are zero.
template <int W, bool OCC>
__device__ __forceinline__ void bwd_terms(const BwdBand* __restrict__ e, double wr,
                                          double wi, double wi2, double wabs2, double mw2r,
                                          double w2i, double2 w, double sx2, double2& GI,
                                          double2& GW) {
#pragma unroll
  for (int iw = 0; iw < W; ++iw) {
    const double2 lo = __ldg(&e[iw].lo);
    const double x = lo.x, x2 = lo.y;
    const double Ar = x - wr;
    const double A2 = fma(Ar, Ar, wi2);
    const double Sr = x + wr;
    const double S2 = fma(Sr, Sr, wi2);
    const bool c1 = gt_nonneg(A2, kLimitTwo) && lt_nonneg(wabs2, kLimitOne * A2);
    const bool c2 = gt_nonneg(wabs2, kTolZero * A2);
    const double r = rcp_refined(A2 * S2);
    const double a1 = c1 ? S2 * r : 0.0;
    const double2 u = make_double2(Ar * a1, wi * a1);          // 1/(x - w) on branch 1
    cmac(GI, __ldg(&e[iw].ca), u);
    cmac(GW, __ldg(&e[iw].cax), cmul(u, u));
    if (OCC) {
      const double b2 = A2 * r;
      const double2 v = make_double2(Sr * b2, -wi * b2);       // 1/(x + w)
      const double2 uv = make_double2((x2 + mw2r) * r, w2i * r);  // 1/(x^2 - w^2)
      const double2 wuv = cmul(w, uv);
      const double2 h = csel(c1, wuv, v);
      const double2 T = cmul(h, csel(c1, uv, v));   // w (uv)^2 or v^2
      const double2 zero = make_double2(0.0, 0.0);
      const bool keep = !(sx2 > 0.0 && x < 0.0 &&
                          (c1 ? gt_nonneg(wabs2 * wabs2 * r, sx2)
                              : gt_nonneg(wabs2, 4.0 * sx2 * S2)));
      const double2 cs = __ldg(&e[iw].cs);
      const double tx2 = 2.0 * x2;
      const double2 cs2x2 = make_double2(tx2 * cs.x, tx2 * cs.y);   // 2 x^2 c_s
      const double2 ch = !keep ? zero : c1 ? cs : (c2 ? __ldg(&e[iw].csh) : zero);
      const double2 cT = !keep ? zero : c1 ? cs2x2 : (c2 ? __ldg(&e[iw].csxh) : zero);
      cmac(GI, ch, h);
      cmac(GW, cT, T);
    }
  }
}

// u^2 of u = U + gamma, in units of 2^31 of U^2's: V + its remainder and FP32 value, laid out as
// a FixU.
__device__ __forceinline__ FixU fix_square(const FixU& u) {
  const long long pr = mad_wide(u.Ur, u.Ur, mad_wide(-u.Ui, u.Ui, 0));
  const long long pi = mad_wide(u.Ur, u.Ui, 0);   // half of it
  FixU v;
  v.Ur = static_cast<int>((pr + (1LL << 30)) >> 31);
  v.Ui = static_cast<int>((pi + (1LL << 29)) >> 30);
  const float k = 0x1p-30f;   // 2 U gamma
  v.gr = fmaf(static_cast<float>(static_cast<int>(static_cast<unsigned>(pr) << 1)), 0x1p-32f,
              k * fmaf(u.ur, u.gr, -u.ui * u.gi));
  v.gi = fmaf(static_cast<float>(static_cast<int>(static_cast<unsigned>(pi) << 2)), 0x1p-32f,
              k * fmaf(u.ur, u.gi, u.ui * u.gr));
  v.ur = static_cast<float>(v.Ur);
  v.ui = static_cast<float>(v.Ui);
  return v;
}

// (s + l) += c u, or with CONJ c conj(u), or with NEG minus that.
template <bool CONJ, bool NEG>
__device__ __forceinline__ void fix_cmac(long long (&s)[2], float (&l)[2], const FixC& c,
                                         const FixU& u) {
  const int r = NEG ? c.nr1 : c.r1, i = NEG ? c.ni1 : c.i1;
  const int nr = NEG ? c.r1 : c.nr1, ni = NEG ? c.i1 : c.ni1;
  const float g = NEG ? -1.0f : 1.0f;
  const float rf = g * c.r1f, jf = g * c.i1f, r0 = g * c.r0, j0 = g * c.i0;
  if (CONJ) {   // re: r Ur + i Ui, im: i Ur - r Ui
    s[0] = mad_wide(r, u.Ur, mad_wide(i, u.Ui, s[0]));
    s[1] = mad_wide(i, u.Ur, mad_wide(nr, u.Ui, s[1]));
    l[0] += fmaf(rf, u.gr, fmaf(jf, u.gi, fmaf(r0, u.ur, j0 * u.ui)));
    l[1] += fmaf(jf, u.gr, fmaf(-rf, u.gi, fmaf(j0, u.ur, -r0 * u.ui)));
  } else {      // re: r Ur - i Ui, im: r Ui + i Ur
    s[0] = mad_wide(r, u.Ur, mad_wide(ni, u.Ui, s[0]));
    s[1] = mad_wide(r, u.Ui, mad_wide(i, u.Ur, s[1]));
    l[0] += fmaf(rf, u.gr, fmaf(-jf, u.gi, fmaf(r0, u.ur, -j0 * u.ui)));
    l[1] += fmaf(rf, u.gi, fmaf(jf, u.gr, fmaf(r0, u.ui, j0 * u.ur)));
  }
}

// s / 2^d, rounded down, for 0 <= d < 32 (at most a dozen here). What is dropped lies below the unit that the
// FP32 parts are moved in. (A general 64-bit shift, rounded: 1% of the adjoint's time.)
__device__ __forceinline__ long long fix_down(long long s, int d) {
  const unsigned lo = __funnelshift_r(static_cast<unsigned>(s), static_cast<unsigned>(s >> 32), d);
  return (static_cast<long long>(static_cast<int>(s >> 32) >> d) << 32) | lo;
}

// A 62-bit sum (with its small FP32 part, moved in in units of 2^4) as 2^sh (U + gamma).
__device__ __forceinline__ FixU fix_limbs(const long long (&s)[2], int sh) {
  const unsigned half = 1u << (sh - 1);
  FixU v;
  v.Ur = static_cast<int>((s[0] + half) >> sh);
  v.Ui = static_cast<int>((s[1] + half) >> sh);
  v.gr = static_cast<float>(static_cast<int>(static_cast<unsigned>(s[0]) << (32 - sh))) * 0x1p-32f;
  v.gi = static_cast<float>(static_cast<int>(static_cast<unsigned>(s[1]) << (32 - sh))) * 0x1p-32f;
  v.ur = static_cast<float>(v.Ur);
  v.ui = static_cast<float>(v.Ui);
  return v;
}

// A complex sum over the bands of M u in the split form (see gpp_terms_fix.cuh): 64-bit sums
// modulo 2^64, the FP32 sum that tells their multiple of 2^64, and the small parts.
struct FixSum {
  long long acc[2];
  float aH[2], aL[2];
  __device__ __forceinline__ void clear() {
    acc[0] = acc[1] = 0;
    aH[0] = aH[1] = aL[0] = aL[1] = 0.0f;
  }
  __device__ __forceinline__ void add(const FixM& m, const FixU& u) {
    acc[0] = mad_wide(m.r1, u.Ur, mad_wide(m.ni1, u.Ui, acc[0]));
    acc[1] = mad_wide(m.r1, u.Ui, mad_wide(m.i1, u.Ur, acc[1]));
    aH[0] = fmaf(m.r1f, u.ur, fmaf(-m.i1f, u.ui, aH[0]));
    aH[1] = fmaf(m.r1f, u.ui, fmaf(m.i1f, u.ur, aH[1]));
    aL[0] += fmaf(m.r1f, u.gr, fmaf(-m.i1f, u.gi, fmaf(m.r0, u.ur, -m.i0 * u.ui)));
    aL[1] += fmaf(m.r1f, u.gi, fmaf(m.i1f, u.gr, fmaf(m.r0, u.ui, m.i0 * u.ur)));
  }
  __device__ __forceinline__ void settle() {   // the small parts, after at most 8 bands
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int r = __float2int_rn(aL[k] * 0x1p-12f);
      acc[k] = mad_wide(r, 4096, acc[k]);
      aL[k] = fmaf(-4096.0f, static_cast<float>(r), aL[k]);
    }
  }
  __device__ __forceinline__ double2 take() {   // the value so far; clears
    double v[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      acc[k] += __float2int_rn(aL[k]);
      const float top = static_cast<float>(static_cast<int>(acc[k] >> 32)) * 0x1p-32f;
      const int j = __float2int_rn(fmaf(aH[k], 0x1p-64f, -top));
      v[k] = fma(static_cast<double>(j), 18446744073709551616.0, static_cast<double>(acc[k]));
    }
    clear();
    return make_double2(v[0], v[1]);
  }
};

// The FP64 form's branch decision for one term, as the sign of |wdiff|^2 - 1/4. Not inlined: it
// is taken about once in 1e6 terms, and inlined the compiler executes it for every term.
__device__ __noinline__ float fix_exact_sign(const BandEntry* f, double2 w) {
  const double a = __ldg(&f->lo.x) - w.x;
  return gt_nonneg(fma(a, a, w.y * w.y), kLimitTwo) ? 1.0f : -1.0f;
}

// The sums M GI and M GW of a pair by the fast form, for what the split-integer form is too coarse
// for; not inlined, as above.
template <int W>
__device__ __noinline__ void fix_f64_sums(int B, int nocc, int64_t G, bool live, const double2* an,
                                          const double2* am, const BwdBand* bt, double2 w,
                                          double2* gI, double2* gw) {
  double2 sI = make_double2(0.0, 0.0), sw = sI;
#pragma unroll 1
  for (int b = 0; b < B; ++b) {
    const double2 a = live ? ldg2(an + static_cast<int64_t>(b) * G) : make_double2(0.0, 0.0);
    const double2 M = cmul(live ? ldg2(am + b) : make_double2(0.0, 0.0), a);
    double2 GI = make_double2(0.0, 0.0), GW = GI;
    const BwdBand* e = bt + static_cast<int64_t>(b) * W;
    if (b < nocc)
      bwd_terms_fast<W, true>(e, w.x, w.y, w.y * w.y, GI, GW);
    else
      bwd_terms_fast<W, false>(e, w.x, w.y, w.y * w.y, GI, GW);
    cmac(sI, M, GI);
    cmac(sw, M, GW);
  }
  *gI = sI;
  *gw = sw;
}

// Where the split-integer form is too coarse. Its errors are about 2^-56 of a scale: of a band's GI,
// of the bound bG on it; of the pair's sums over n bands, of sqrt(n) times the largest weight times bG
// (for GW = GI + w H, or times |w| and the bound on H). An entry whose own terms are far below that
// (large cotangents or heavy bands in branch 2, x << |w|, where GI and w H cancel) is taken from FP64.
// Q's: the whole warp, where a band's terms are below 2^-8 of bG in a lane (errors are 2^-48 of them
// above). That takes cotangents of different sizes (FixBwd::spread), so only those are
// looked through. The pair's two sums: where those of any lane are below 2^-9 (I_eps) and 2^-11
// (wtilde), or of half of the lanes below 2^-7 and 2^-9. Ordinary inputs lie above but for
// one warp in a hundred with few bands (4e5 drawn lanes of 2..128 bands: median 2^-3 .. 2^-6, least
// 2^-8 and 2^-12, of half of a warp's 2^-5 and 2^-8). The terms' powers are formed (fix_weak_sums) only
// where the sums themselves are not above these lines (of any lane, a quarter of them: a
// lane's sum is below its terms by chance): 2 to 3 warps in a hundred. With the powers in the band loop
// instead the adjoint took 5% longer, with the calls there 3%.
constexpr int kWeakBand = 8, kWeakI = 9, kWeakW = 11, kWeakHalf = 2;

// Votes on a warp's sums and their least ones, as logarithms in units of 2^-18 (fix_log_max).
__device__ __forceinline__ bool fix_weak_vote(bool live, int I, int leastI, int W, int leastW,
                                              int slack) {
  const int one = 1 << 18;
  const int m = live ? min(I - leastI + kWeakI * one, W - leastW + kWeakW * one) : one * 100;
  const unsigned half = __ballot_sync(0xffffffffu, m < kWeakHalf * one);
  return __any_sync(0xffffffffu, m < -slack * one) || 2 * __popc(half) > __popc(__ballot_sync(0xffffffffu, live));
}

// The least |x - w| of branch 1 and |x + w|^2 over the frequencies, less the FP32 rounding.
template <int W>
__device__ __forceinline__ void fix_distances_all(const FixPair& wf, const double* xrange, float& dA,
                                                  float& dS2) {
  dA = dS2 = 3.0e38f;
#pragma unroll
  for (int k = 0; k < W; ++k) {
    const float lo = static_cast<float>(xrange[k]), hi = static_cast<float>(xrange[kMaxNw + k]);
    dA = fminf(dA, fmaxf(0.5f, fmaxf(lo - wf.w1, wf.w1 - hi) * (1.0f - 0x1p-17f)));
    const float sr = lo + wf.w1;
    dS2 = fminf(dS2, fmaf(sr, sr, wf.i1 * wf.i1) * (1.0f - 0x1p-17f));
  }
}

// Whether one of the bands is too weak in a lane of the warp: its terms' power below 2^-kWeakBand of
// the bound on them.
template <int W>
__device__ __noinline__ bool fix_weak_bands(int B, int nocc, const BandEntry* ft, const FixBwd* fixc,
                                            double2 w, const FixPair wf, const double* xrange,
                                            bool live) {
  const float wr = static_cast<float>(w.x), wi2 = static_cast<float>(w.y) * static_cast<float>(w.y);
  float dA, dS2;
  fix_distances_all<W>(wf, xrange, dA, dS2);
  bool weak = false;
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    if (fixc->spread[c] == 0) continue;
    const float bG = fixc->sum_c[c] / dA + (c == 0 ? fixc->sum_s * rsqrtf(dS2) : 0.0f);
    const float line = bG * exp2if(-kWeakBand);
#pragma unroll 1
    for (int b = c == 0 ? 0 : nocc; b < (c == 0 ? nocc : B); ++b) {
      float g = 0.0f;
#pragma unroll
      for (int k = 0; k < W; ++k) {
        const float x = static_cast<float>(__ldg(&ft[static_cast<int64_t>(b) * W + k].lo.x));
        const float a = x - wr, a2 = fmaf(a, a, wi2), s = x + wr, s2 = fmaf(s, s, wi2);
        if (a2 > 0.25f * (1.0f + 0x1p-12f))   // clearly in branch 1
          g = fmaf(c == 0 ? fixc->cap2[k] : fixc->ca2[k], fix_rcp(a2), g);
        if (c == 0) g = fmaf(fixc->csh2[k], fix_rcp(s2), g);
      }
      weak |= g > 0.0f && g < line * line;
    }
  }
  return __any_sync(0xffffffffu, weak && live);
}

// Whether a warp's sums are too weak for their scales (leastI, leastW), by the powers of their
// terms: in FP32, M as in fix_strong.
template <int W>
__device__ __noinline__ bool fix_weak_sums(int B, int nocc, int64_t G, bool live, const double2* an_ptr,
                                           const double2* am_ptr, const BandEntry* ft,
                                           const FixBwd* fixc, double2 w, int leastI, int leastW) {
  const float wr = static_cast<float>(w.x), wi = static_cast<float>(w.y), wi2 = wi * wi;
  int I = kFixNone, Y = kFixNone;
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const int b0 = c == 0 ? 0 : nocc, b1 = c == 0 ? nocc : B;
    FixScale sc;
    fix_scales(b0, b1, G, an_ptr, am_ptr, live, sc);
    const float m1 = exp2if(60 - sc.sh);
    float pI = 0.0f, pW = 0.0f;
#pragma unroll 4
    for (int b = b0; b < b1; ++b) {
      const double2 an = live ? ldg2(an_ptr + static_cast<int64_t>(b) * G) : make_double2(0.0, 0.0);
      const double2 am = live ? ldg2(am_ptr + b) : make_double2(0.0, 0.0);
      const float m2 = fmaxf(fix_square_of(an, sc.kn - 30) * fix_square_of(am, sc.ka - 30), 1e-37f) * m1 * m1;
      float g = 0.0f, h = 0.0f;
#pragma unroll
      for (int k = 0; k < W; ++k) {
        const float x = static_cast<float>(__ldg(&ft[static_cast<int64_t>(b) * W + k].lo.x));
        const float a = x - wr, a2 = fmaf(a, a, wi2), s = x + wr, s2 = fmaf(s, s, wi2);
        const bool b1 = a2 > 0.25f * (1.0f + 0x1p-12f);   // clearly
        const float ra = b1 ? fix_rcp(a2) : 0.0f, rs = fix_rcp(s2);
        const float cu = (c == 0 ? fixc->cap2[k] : fixc->ca2[k]) * ra;
        const float sv = c == 0 ? fixc->csh2[k] * rs : 0.0f;
        g += cu + sv;
        h = fmaf(x * x, fmaf(cu, ra, sv * rs), h);
      }
      pI = fmaf(m2, g, pI);
      pW = fmaf(m2, h, pW);
    }
    const int unit = (sc.unit() + fixc->ec[c] + 1023) << 18;
    if (pI > 0.0f) I = max(I, fix_half_log(pI) + unit);
    if (pW > 0.0f) Y = max(Y, fix_half_log(pW) + unit);
  }
  const bool none = I == kFixNone;   // no terms: the sums are exactly zero
  return fix_weak_vote(live, none ? leastI : I, leastI, none ? leastW : Y, leastW, 0);
}

// Bands between two reductions of a CTA (shared memory: 8 KB per band).
constexpr int kRedBands = 4;
constexpr int kTile = kTX * kTY;

// The sums of the last nb bands (from b0): over the 8 columns of am Q (s_c, written to part_n),
// over the 32 G-vectors of aqsntemp Q (s_r, written to part_r), each [component][band][column]
// [G-vector] doubles. A column sum is one thread's; a row sum is four neighbouring lanes', 8
// G-vectors each (started at different places: no bank conflicts), then two shuffles.
__device__ __forceinline__ void tile_reduce(const double* s_c, const double* s_r, int nb, int B,
                                            int b0, int64_t G, int64_t ig0, int gl, int64_t igt,
                                            int ngroups, double* __restrict__ part_n,
                                            double* __restrict__ part_r) {
  const int L = threadIdx.x;
  {
    const int ig = L & 31, c = (L >> 5) & 1, bb = L >> 6;   // kRedBands = 4: 256 column sums
    if (bb < nb && ig0 + ig < G) {
      const double* v = s_c + (c * kRedBands + bb) * kTile + ig;
      double sum = v[0];
#pragma unroll
      for (int y = 1; y < kTY; ++y) sum += v[y * kTX];
      part_n[2 * ((static_cast<int64_t>(gl) * B + b0 + bb) * G + ig0 + ig) + c] = sum;
    }
  }
  const int q = L & 3, y = (L >> 2) & 7, c = (L >> 5) & 1, bb = L >> 6;   // 64 row sums
  double sum = 0.0;
  const double* v = s_r + (c * kRedBands + bb) * kTile + y * kTX + q;
#pragma unroll
  for (int i = 0; i < 8; ++i) sum += v[4 * ((i + y) & 7)];
  sum += __shfl_xor_sync(0xffffffffu, sum, 1);
  sum += __shfl_xor_sync(0xffffffffu, sum, 2);
  if (q == 0 && bb < nb)
    part_r[2 * ((igt * B + b0 + bb) * (static_cast<int64_t>(ngroups) * kTY) + gl * kTY + y) + c] = sum;
}

// Dynamic shared memory: the reductions' 2 x 2 x kRedBands x kTile doubles, then each warp's
// staged weights.
constexpr size_t kBwdSmem = static_cast<size_t>(4 * kRedBands) * kTile * sizeof(double) +
                            kTY * kStageBands * sizeof(FixAm);

template <int W>
__global__ void __launch_bounds__(kTile, 2) gpp_bwd_kernel(
    int B, int64_t G, int64_t P, int nocc, int64_t group0, int ngroups, int64_t n_ig_tiles,
    const double2* __restrict__ aqsn, const double2* __restrict__ eps,
    const double2* __restrict__ wt, const double2* __restrict__ am,
    const BwdBand* __restrict__ bt, const BandEntry* __restrict__ ft,
    const FixBwd* __restrict__ fixc, const int* __restrict__ colg, const int* __restrict__ flags,
    double2* __restrict__ grad_w, double2* __restrict__ grad_I,
    double2* __restrict__ part_n,  // [ngroups][B][G]
    double2* __restrict__ part_r,  // [n_ig_tiles][B][ngroups * kTY]
    double sx2)                    // screened-exchange cutoff, sexcut^2 (0 = off)
{
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  __shared__ FixC s_cap[W], s_csh[W], s_ca[W];
  double* const s_c = reinterpret_cast<double*>(dyn_smem);
  double* const s_r = s_c + 2 * kRedBands * kTile;
  const int lane = threadIdx.x & 31, ty = threadIdx.x >> 5;
  FixAm* const stage = reinterpret_cast<FixAm*>(s_r + 2 * kRedBands * kTile) + ty * kStageBands;
  const bool x_nonneg = flags[0] == 0;
  const double wabs2_pf = pf_wabs2_min(flags);   // the partial fractions' bound (gpp_device.cuh)
  const double xmax2 = wabs2_pf / kPfRatio2;
  const FixInfo fix = *reinterpret_cast<const FixInfo*>(flags + kFlagFix);
  const double* xrange = reinterpret_cast<const double*>(flags + kFlagRange);
  const bool fix_on = fix.ok == 1 && fixc->ok;
  for (int k = threadIdx.x; k < W; k += kTile) {
    s_cap[k] = fixc->cap[k];
    s_csh[k] = fixc->csh[k];
    s_ca[k] = fixc->ca[k];
  }
  __syncthreads();
  const int64_t ntiles = static_cast<int64_t>(ngroups) * n_ig_tiles;
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    // G-vector tile slowest, so the CTAs running together share one slab of aqsntemp
    const int64_t igt = t / ngroups;
    const int gl = static_cast<int>(t - igt * ngroups);       // group within the batch
    const int64_t p = (group0 + gl) * kTY + ty;
    const int64_t ig0 = igt * kTX, ig = ig0 + lane;
    const bool col_ok = p < P && colg[p] >= 0;
    const bool live = col_ok && ig < G;
    double2 w = make_double2(1.0, 0.5);  // inert lane: finite terms, zero weight
    double2 I = make_double2(0.0, 0.0);
    if (live) {
      w = ldg2(wt + p * G + ig);
      I = ldg2(eps + p * G + ig);
    }
    const double wr = w.x, wi = w.y;
    const double wi2 = wi * wi;
    const double wabs2 = fma(wr, wr, wi2);
    const double2 Iw = cmul(I, w);
    const double2* an_ptr = aqsn + (ig < G ? ig : 0);
    const double2* am_ptr = am + (col_ok ? p : 0) * B;
    auto load_an = [&](int b) {
      return live ? ldg2(an_ptr + static_cast<int64_t>(b) * G) : make_double2(0.0, 0.0);
    };
    double2 gw = make_double2(0.0, 0.0), gI = make_double2(0.0, 0.0);
    // one band's am Q and aqsntemp Q into the reduction's slot bb
    auto put = [&](int bb, double2 amv, double2 an, double2 Q) {
      const double2 c = cmul(amv, Q), r = cmul(an, Q);
      s_c[bb * kTile + threadIdx.x] = c.x;
      s_c[(kRedBands + bb) * kTile + threadIdx.x] = c.y;
      s_r[bb * kTile + threadIdx.x] = r.x;
      s_r[(kRedBands + bb) * kTile + threadIdx.x] = r.y;
    };
    auto reduce = [&](int b0, int nb) {
      __syncthreads();
      tile_reduce(s_c, s_r, nb, B, b0, G, ig0, gl, igt, ngroups, reinterpret_cast<double*>(part_n),
                  reinterpret_cast<double*>(part_r));
      __syncthreads();
    };
    auto load_am = [&](int b) { return col_ok ? ldg2(am_ptr + b) : make_double2(0.0, 0.0); };

    // Split-integer form: the pair's scales, if the whole warp is in its range. GW = GI + w H
    // cancels where x << |w|, so |w| may not exceed twice the largest frequency.
    bool use_fix = fix_on && __all_sync(0xffffffffu, !live || (fix_lane(w, wabs2, fix) &&
                                                               !gt_nonneg(wabs2, 4.0 * xmax2)));
    // The bands of asxtemp and the others have scales of their own, packed: kn | ka << 9 | sh << 18,
    // and bit 24 where there are weights that are not zero.
    int packs[2] = {0, 0};
    if (use_fix) {
      bool ok = true;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        unsigned mn = 0, ma = 0, mp = 0;
#pragma unroll 8
        for (int b = c == 0 ? 0 : nocc; b < (c == 0 ? nocc : B); ++b) {
          const unsigned hn = fix_hi_max(load_an(b)), ha = fix_hi_max(load_am(b));
          mn = max(mn, hn);
          ma = max(ma, ha);
          mp = max(mp, hn + ha);
        }
        int kn, ka, sh;
        ok &= fix_weight_scale(mn, ma, mp, kn, ka, sh);
        packs[c] = kn | ka << 9 | sh << 18 | (mn != 0 && ma != 0 ? 1 << 24 : 0);
      }
      use_fix = __all_sync(0xffffffffu, ok);
    }
    const FixPair wf = fix_pair(w, fix.E);
    if (use_fix && (fixc->spread[0] | fixc->spread[1]) != 0)
      use_fix = !fix_weak_bands<W>(B, nocc, ft, fixc, w, wf, xrange, live);
    float2 scA = make_float2(0.0f, 0.0f), scS = scA;   // the scales of u and of v
    int ks = 0, down = 0, shG = 1, shH = 1, nkhi = 0, akhi = 0, sh = 1;
    double2 Iws = live ? Iw : make_double2(0.0, 0.0);   // times the unit of GI
    int leastI = kFixNone, leastW = kFixNone;   // log2 of the scales of M GI and M GW
    // The scales of a class of bands; GI is in units of the integer sum's last bit.
    auto unit_of = [&](int c) { return exp2i(fixc->ec[c] - 31 - ks) * (1.0 / kFixKappa); };
    auto begin = [&](int c) {
      if (!use_fix) return;
      float dA, dS2;
      fix_distances_all<W>(wf, xrange, dA, dS2);
      // u at its own scale, v at most as fine; the sums of the u terms are brought to v's scale
      const int ksA = fix_ks(dA * dA);
      ks = c == 0 ? min(ksA, fix_ks(dS2)) : ksA;
      down = ksA - ks;
      scA = fix_scale(ksA, fix.E);
      scS = fix_scale(ks, fix.E);
      // |GI| 2^(31 + ks - ec) and |H| 2^(2 ks - ec) stay below 2^(31 + shG), 2^(31 + shH)
      const float ca = fixc->sum_c[c], cs = c == 0 ? fixc->sum_s : 0.0f;
      const float bG = (ca / dA + cs * rsqrtf(dS2)) * 1.01f + 1e-30f;
      const float bH = (ca / (dA * dA) + cs / dS2) * 1.01f + 1e-30f;
      shG = min(max(ks + (__float_as_int(bG) >> 23) - 126, 1), 31);
      shH = min(max(2 * ks - 31 + (__float_as_int(bH) >> 23) - 126, 1), 31);
      const double unit = live ? unit_of(c) : 0.0;
      Iws = make_double2(Iw.x * unit, Iw.y * unit);
      nkhi = ((packs[c] & 511) + 32) << 20;
      akhi = ((packs[c] >> 9 & 511) + 32) << 20;
      sh = packs[c] >> 18 & 63;
      // (keeps the compiler from forming these again in every band)
      asm volatile("" : "+d"(Iws.x), "+d"(Iws.y), "+f"(scA.x), "+f"(scA.y), "+f"(scS.x), "+f"(scS.y),
                        "+r"(shG), "+r"(shH), "+r"(down), "+r"(nkhi), "+r"(akhi), "+r"(sh));
    };
    FixSum X, Y;
    X.clear();
    Y.clear();
    double2 an_next = load_an(0);
    // One band of a warp in the split-integer form; returns GI in units of unitG.
    auto band_fix = [&](int b, int b0, int b1, double2 an, auto occ_tag) {
      constexpr bool OCC = decltype(occ_tag)::value;
      const int at = (b - b0) & (kStageBands - 1);
      if (at == 0) {   // this warp's weights of the next bands
        __syncwarp();
        for (int q = lane; q < kStageBands && b + q < b1; q += 32) {
          const double2 a = load_am(b + q);
          FixAm e;
          fix_value(a.x, akhi, e.r1, e.r0);
          fix_value(a.y, akhi, e.i1, e.i0);
          stage[q] = e;
        }
        __syncwarp();
      }
      const FixM m = fix_weight(stage[at], an, nkhi, sh);
      const BandEntry* f = ft + static_cast<int64_t>(b) * W;
      long long g[2] = {0, 0}, h[2] = {0, 0};
      float g0[2] = {0.0f, 0.0f}, h0[2] = {0.0f, 0.0f};
      // the FP32 parts (below 2^31 kLow, 2^32 kLow) into the sums
      constexpr int kLow = W <= 3 ? 4 : 8;
      auto settle = [&]() {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          g[k] = mad_wide(__float2int_rn(g0[k] * (1.0f / kLow)), kLow, g[k]);
          h[k] = mad_wide(__float2int_rn(h0[k] * (0.5f / kLow)), 2 * kLow, h[k]);
          g0[k] = h0[k] = 0.0f;
        }
      };
      // |wdiff|^2 - 1/4: its sign decides branch 1. One vote per band: a vote between the terms
      // would keep them from overlapping (2%).
      float ds[W], dmin = 1.0f;
#pragma unroll
      for (int k = 0; k < W; ++k) {
        const int4 xv = __ldg(&f[k].fx);
        const FixN na = fix_norm<true>(wf, __int_as_float(xv.z), __int_as_float(xv.w));
        ds[k] = (na.N1 - 0.25f) + na.Nm;
        dmin = fminf(dmin, fabsf(ds[k]));
      }
      if (__any_sync(0xffffffffu, dmin <= kFixNear)) {
#pragma unroll
        for (int k = 0; k < W; ++k) ds[k] = fix_exact_sign(f + k, w);
      }
#pragma unroll(W <= 3 ? W : 1)
      for (int k = 0; k < W; ++k) {
        const int4 xv = __ldg(&f[k].fx);
        const FixN na = fix_norm<true>(wf, __int_as_float(xv.z), __int_as_float(xv.w));
        const float d = ds[k];
        const FixC c = OCC ? s_cap[k] : s_ca[k];
        const FixU u = fix_term<true, true>(wf, na, fix_biased(xv), scA, d > 0.0f);
        fix_cmac<false, false>(g, g0, c, u);
        fix_cmac<false, false>(h, h0, c, fix_square(u));
      }
      settle();
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        g[k] = fix_down(g[k], down);
        h[k] = fix_down(h[k], 2 * down);
      }
      if (OCC) {
#pragma unroll(W <= 3 ? W : 1)
        for (int k = 0; k < W; ++k) {   // v is the conjugate of what fix_term gives
          const int4 xv = __ldg(&f[k].fx);
          const FixC c = s_csh[k];
          const FixN ns = fix_norm<false>(wf, __int_as_float(xv.z), __int_as_float(xv.w));
          const FixU u = fix_term<false, false>(wf, ns, fix_biased(xv), scS, true);
          fix_cmac<true, false>(g, g0, c, u);
          fix_cmac<true, true>(h, h0, c, fix_square(u));
        }
        settle();
      }
      X.add(m, fix_limbs(g, shG));
      Y.add(m, fix_limbs(h, shH));
      return make_double2(static_cast<double>(g[0]), static_cast<double>(g[1]));
    };
    // One band of a warp in FP64: its M GI and M GW into gI and gw; returns GI.
    const double mw2r = -fma(wr, wr, -wi2), w2i = 2.0 * wr * wi;
    const bool fast_lane = wr >= 0.0 && gt_nonneg(wabs2, kFastWabs2Lo) &&
                           lt_nonneg(wabs2, kFastWabs2Hi) && !lt_nonneg(wabs2, wabs2_pf);
    const bool fast = __all_sync(0xffffffffu, fast_lane || !live) && x_nonneg;
    auto band_f64 = [&](int b, double2 an, double2 amv, auto occ_tag) {
      constexpr bool OCC = decltype(occ_tag)::value;
      double2 GI = make_double2(0.0, 0.0), GW = make_double2(0.0, 0.0);
      const BwdBand* e = bt + static_cast<int64_t>(b) * W;
      if (fast)
        bwd_terms_fast<W, OCC>(e, wr, wi, wi2, GI, GW);
      else
        bwd_terms<W, OCC>(e, wr, wi, wi2, wabs2, mw2r, w2i, w, sx2, GI, GW);
      // sum_b M w GI and sum_b M I GW: w and I are the thread's constants, applied at the end
      const double2 M = cmul(amv, an);
      cmac(gI, M, GI);
      cmac(gw, M, GW);
      return GI;
    };
    auto run = [&](int b0, int b1, auto occ_tag) {
      for (int c0 = b0; c0 < b1; c0 += kRedBands) {
        const int nb = min(kRedBands, b1 - c0);
#pragma unroll 1
        for (int bb = 0; bb < nb; ++bb) {
          const int b = c0 + bb;
          const double2 an = an_next, amv = load_am(b);
          if (b + 1 < B) an_next = load_an(b + 1);
          const double2 GI = use_fix ? band_fix(b, b0, b1, an, occ_tag) : band_f64(b, an, amv, occ_tag);
          put(bb, amv, an, cmul(Iws, GI));
        }
        if (use_fix) {
          X.settle();
          Y.settle();
          if (((c0 - b0) & (kFlushBands - kRedBands)) == kFlushBands - kRedBands) {
            const double2 x = X.take(), y = Y.take();
            gI = make_double2(gI.x + x.x, gI.y + x.y);
            gw = make_double2(gw.x + y.x, gw.y + y.y);
          }
        }
        reduce(c0, nb);
      }
    };
    // The sums of a class of bands, M GI and M H, in FP64; H's unit: u^2 = V 2^(31 - 2 ks) / kappa^2.
    double2 rI = make_double2(0.0, 0.0), rH = rI;
    auto end = [&](int c) {
      if (!use_fix) return;
      const double2 x = X.take(), y = Y.take();
      const int em = sh + 64 - (nkhi >> 20) - (akhi >> 20);
      const double fx = unit_of(c) * exp2i(shG + em);
      const double fy = exp2i(fixc->ec[c] - 2 * ks + shH) * (1.0 / kFixKappa) * (1.0 / kFixKappa) *
                        exp2i(em);
      rI = make_double2(fma(fx, gI.x + x.x, rI.x), fma(fx, gI.y + x.y, rI.y));
      rH = make_double2(fma(fy, gw.x + y.x, rH.x), fma(fy, gw.y + y.y, rH.y));
      gI = gw = make_double2(0.0, 0.0);
      // (not of a class without weights or cotangents: its sums are zero, its scale is nothing's)
      if ((packs[c] >> 24) != 0 && fixc->sum_c[c] + (c == 0 ? fixc->sum_s : 0.0f) > 0.0f) {
        const int n = fix_half_log(static_cast<float>(c == 0 ? nocc : B - nocc)) + ((1023 + 62 + em) << 18);
        const int lI = n + ((fixc->ec[c] - 31 - ks + shG) << 18);
        const int lw = fix_log_max(w.x, w.y) - (1023 << 18);
        leastI = max(leastI, lI);
        leastW = max(leastW, max(lI, n + lw + ((fixc->ec[c] - 2 * ks + shH) << 18)));
      }
    };
    if (nocc > 0) {
      begin(0);
      run(0, nocc, BoolTag<true>());
      end(0);
    }
    if (nocc < B) {
      begin(1);
      run(nocc, B, BoolTag<false>());
      end(1);
    }
    if (use_fix) {
      gI = rI;
      gw = cmul(w, rH);
      gw = make_double2(gI.x + gw.x, gI.y + gw.y);   // M GW = M GI + w M H
      if (fix_weak_vote(live, fix_log_max(gI.x, gI.y), leastI, fix_log_max(gw.x, gw.y), leastW, 2) &&
          fix_weak_sums<W>(B, nocc, G, live, an_ptr, am_ptr, ft, fixc, w, leastI, leastW)) {   // rare
        double2 sI, sw;
        fix_f64_sums<W>(B, nocc, G, live, an_ptr, am_ptr, bt, w, &sI, &sw);
        gI = sI;
        gw = sw;
      }
    }
    gI = cmul(w, gI);
    gw = cmul(I, gw);
    if (live) {
      if (grad_w) grad_w[p * G + ig] = make_double2(gw.x, -gw.y);
      if (grad_I) grad_I[p * G + ig] = make_double2(gI.x, -gI.y);
    } else if (p < P && ig < G) {
      if (grad_w) grad_w[p * G + ig] = make_double2(0.0, 0.0);
      if (grad_I) grad_I[p * G + ig] = make_double2(0.0, 0.0);
    }
  }
}

// grad_aqsn[b][ig] (+)= conj(sum over the batch's groups, in order); rtot[b][p] = sum over
// ig tiles, in order, for the batch's columns.
__global__ void gpp_bwd_finish_batch_kernel(int64_t B, int64_t G, int64_t P, int64_t group0,
                                            int ngroups, int64_t n_ig_tiles, bool first,
                                            const double2* __restrict__ part_n,
                                            const double2* __restrict__ part_r,
                                            double2* __restrict__ grad_n, double2* __restrict__ rtot) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const int64_t tid = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  for (int64_t i = tid; i < B * G; i += stride) {
    double2 s = make_double2(0.0, 0.0);
    for (int gl = 0; gl < ngroups; ++gl) {
      const double2 v = part_n[static_cast<int64_t>(gl) * B * G + i];
      s.x += v.x;
      s.y += v.y;
    }
    if (grad_n) {
      double2 o = first ? make_double2(0.0, 0.0) : grad_n[i];
      grad_n[i] = make_double2(o.x + s.x, o.y - s.y);
    }
  }
  const int64_t ncols = static_cast<int64_t>(ngroups) * kTY;
  for (int64_t i = tid; i < B * ncols; i += stride) {
    const int64_t b = i / ncols, c = i - b * ncols;
    const int64_t p = group0 * kTY + c;
    if (p >= P) continue;
    double2 s = make_double2(0.0, 0.0);
    for (int64_t it = 0; it < n_ig_tiles; ++it) {
      const double2 v = part_r[(it * B + b) * ncols + c];
      s.x += v.x;
      s.y += v.y;
    }
    rtot[b * P + p] = s;
  }
}

// The columns that share a global column, as lists in increasing p: next[p] is the next column
// with p's global column (-1: none), first[p] whether p is the first of its list. A column per
// warp.
__global__ void gpp_bwd_links_kernel(int64_t P, const int* __restrict__ colg, int* __restrict__ next,
                                     int* __restrict__ first) {
  const int lane = threadIdx.x & 31;
  const int64_t p = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  if (p >= P) return;
  const int g = colg[p];
  int nx = 0x7fffffff;
  bool before = false;
  for (int64_t q = lane; q < P; q += 32)
    if (colg[q] == g) {
      if (q < p) before = true;
      if (q > p) nx = min(nx, static_cast<int>(q));
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) nx = min(nx, __shfl_xor_sync(0xffffffffu, nx, o));
  before = __any_sync(0xffffffffu, before);
  if (lane == 0) {
    next[p] = nx == 0x7fffffff ? -1 : nx;
    first[p] = !before && g >= 0;
  }
}

// grad_aqsm[b][g] = vcoul[g] * sum over columns p with g(p) = g, in increasing p (zero elsewhere:
// the array is cleared first). One thread per (b, p).
__global__ void gpp_bwd_aqsm_scatter_kernel(int64_t B, int64_t P, int64_t G,
                                            const int* __restrict__ colg,
                                            const double* __restrict__ vcoul,
                                            const double2* __restrict__ rtot,
                                            const int* __restrict__ next,
                                            const int* __restrict__ first,
                                            double2* __restrict__ grad_m) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < B * P;
       i += stride) {
    const int64_t b = i / P, p = i - b * P;
    if (!first[p]) continue;   // the first column with this g sums all of them, in order
    const int g = colg[p];
    double2 s = make_double2(0.0, 0.0);
    for (int q = static_cast<int>(p); q >= 0; q = next[q]) {
      const double2 v = rtot[b * P + q];
      s.x += v.x;
      s.y += v.y;
    }
    const double vc = vcoul[g];
    grad_m[b * G + g] = make_double2(vc * s.x, vc * s.y);
  }
}

template <int W>
const void* bwd_fn() {
  return reinterpret_cast<const void*>(&gpp_bwd_kernel<W>);
}

const void* bwd_kernel_ptr(int nw) {
  switch (nw) {
    case 1: return bwd_fn<1>();
    case 2: return bwd_fn<2>();
    case 3: return bwd_fn<3>();
    case 4: return bwd_fn<4>();
    case 5: return bwd_fn<5>();
    case 6: return bwd_fn<6>();
    case 7: return bwd_fn<7>();
    case 8: return bwd_fn<8>();
    default: return nullptr;
  }
}

cudaError_t bwd_allow_smem(const void* fn) {
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(kBwdSmem));
}

int grid_for(int64_t work) {
  int64_t b = (work + 255) / 256;
  if (b < 1) b = 1;
  if (b > 8192) b = 8192;
  return static_cast<int>(b);
}

}  // namespace

int bwd_blocks_per_sm(int nw) {
  const void* fn = bwd_kernel_ptr(nw);
  if (!fn) return 0;
  int n = 0;
  if (bwd_allow_smem(fn) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, kTile, kBwdSmem) != cudaSuccess)
    return 0;
  return n;
}

int64_t bwd_groups(int64_t P) { return (P + kTY - 1) / kTY; }
int bwd_tile_ig() { return kTX; }
int bwd_tile_cols() { return kTY; }

cudaError_t launch_bwd(const gpp_problem& p, int occ_mode, double ach_scale, double sx2,
                       const BwdPlan& plan, char* ws, const gpp_c128* g_ach,
                       const gpp_c128* g_asx, const gpp_grads& out, cudaStream_t s) {
  const int64_t B = p.number_bands, G = p.ncouls, P = p.ngpown;
  const int W = static_cast<int>(p.nw);
  int64_t nocc = B;
  if (occ_mode == GPP_OCC_OCCUPIED) nocc = p.nvband < B ? p.nvband : B;
  BwdBand* bt = reinterpret_cast<BwdBand*>(ws + plan.off_bwd_bt);
  FixBwd* fixc = reinterpret_cast<FixBwd*>(ws + plan.off_bwd_fix);
  gpp_bwd_prep_kernel<<<grid_for(B * W) + 1, 256, 0, s>>>(
      B, W, p.wx_array, reinterpret_cast<const double2*>(g_ach),
      reinterpret_cast<const double2*>(g_asx), ach_scale, bt, fixc);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const double2* am = reinterpret_cast<const double2*>(ws + plan.fwd.off_am);
  const int* colg = reinterpret_cast<const int*>(ws + plan.fwd.off_colvalid);
  const int* flags = reinterpret_cast<const int*>(ws + plan.fwd.off_flags);
  double2* part_n = reinterpret_cast<double2*>(ws + plan.off_part_n);
  double2* part_r = reinterpret_cast<double2*>(ws + plan.off_part_r);
  double2* rtot = reinterpret_cast<double2*>(ws + plan.off_rtot);
  const int64_t ngroups_total = bwd_groups(P);
  const int64_t n_ig_tiles = (G + kTX - 1) / kTX;
  const BandEntry* ft = reinterpret_cast<const BandEntry*>(ws + plan.fwd.off_bt);
  for (int64_t g0 = 0; g0 < ngroups_total; g0 += plan.batch_groups) {
    const int ng = static_cast<int>(ngroups_total - g0 < plan.batch_groups ? ngroups_total - g0
                                                                            : plan.batch_groups);
    const int64_t ntiles = ng * n_ig_tiles;
    int grid = static_cast<int>(ntiles < plan.max_grid ? ntiles : plan.max_grid);
#define GPP_BWD_LAUNCH(WV)                                                                        \
  gpp_bwd_kernel<WV><<<grid, kTile, kBwdSmem, s>>>(                                                      \
      static_cast<int>(B), G, P, static_cast<int>(nocc), g0, ng, n_ig_tiles,                      \
      reinterpret_cast<const double2*>(p.aqsntemp), reinterpret_cast<const double2*>(p.I_eps_array), \
      reinterpret_cast<const double2*>(p.wtilde_array), am, bt, ft, fixc, colg, flags,            \
      reinterpret_cast<double2*>(out.wtilde_array), reinterpret_cast<double2*>(out.I_eps_array),  \
      part_n, part_r, sx2)
    switch (W) {
      case 1: GPP_BWD_LAUNCH(1); break;
      case 2: GPP_BWD_LAUNCH(2); break;
      case 3: GPP_BWD_LAUNCH(3); break;
      case 4: GPP_BWD_LAUNCH(4); break;
      case 5: GPP_BWD_LAUNCH(5); break;
      case 6: GPP_BWD_LAUNCH(6); break;
      case 7: GPP_BWD_LAUNCH(7); break;
      case 8: GPP_BWD_LAUNCH(8); break;
      default: return cudaErrorInvalidValue;
    }
#undef GPP_BWD_LAUNCH
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    gpp_bwd_finish_batch_kernel<<<grid_for(B * G), 256, 0, s>>>(
        B, G, P, g0, ng, n_ig_tiles, g0 == 0, part_n, part_r,
        reinterpret_cast<double2*>(out.aqsntemp), rtot);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if (out.aqsmtemp) {
    int* next = reinterpret_cast<int*>(ws + plan.off_links);
    e = cudaMemsetAsync(out.aqsmtemp, 0, static_cast<size_t>(B) * G * 16, s);
    if (e != cudaSuccess) return e;
    gpp_bwd_links_kernel<<<static_cast<unsigned>((P + 7) / 8), 256, 0, s>>>(P, colg, next, next + P);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    gpp_bwd_aqsm_scatter_kernel<<<grid_for(B * P), 256, 0, s>>>(
        B, P, G, colg, p.vcoul, rtot, next, next + P, reinterpret_cast<double2*>(out.aqsmtemp));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace gpp
