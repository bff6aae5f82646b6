// The split-integer evaluation of the FP64 fast path's terms (gpp_terms_f64.cuh, "fast
// path"), for warps whose inputs lie in its range.
//
// Why. GB300's FP64 pipe issues one warp instruction per SM sub-partition every 64 cycles,
// the integer and FP32 pipes one every 1 (FFMA), 2 (IMAD, shift, convert) or 4 (32 x 32 -> 64
// bit multiply-add) cycles (measured: 1.9 DFMA, 113 FFMA, 60 IMAD, 30 IMAD.WIDE per clock per
// SM). A term of the sum costs 18 FP64 instructions per frequency (1152 cycles); the same
// term on 32-bit integers and floats, to at least the same accuracy, takes about 95
// instructions and 140 cycles (a band with three frequencies, u and v: 612 and 956). What bounds
// it is the dispatch of those instructions: 64% of the issue slots are used, since a 64-bit
// multiply-add, a shift or a conversion holds the port for two to four cycles.
//
// What. Per (band, frequency) the sums need u = 1/(x - w) (branch 1 only) and v = 1/(x + w),
// times the weight M = am an, accumulated over the bands. Every quantity is held as a leading
// 31-bit integer plus a small remainder:
//   A = x - w    = Ah 2^-h + Al 2^-(h+32)   (62 bits, exact differences of the split x and w)
//   u kappa 2^ks = U + gamma                (U 31-bit integer, |gamma| about one unit, FP32)
//   M 2^..       = M1 + M0                  (M1 31-bit integer, |M0| about half a unit, FP32)
// so that the product M u is M1 U (exact, 62 bits, accumulated in 64-bit integers) plus
// M1 gamma + M0 u (2^-30 of it: FP32 suffices, 2^-54 overall).
//
// U: an FP32 reciprocal of |A|^2 corrected once in FP32 (the residual 1 - rho |A|^2 from an
// error-free square), rounded to an integer: accurate to about one unit, 2^-31 of the
// largest u. gamma: the remaining error e = 1 - A U / (kappa 2^ks) of the integer U,
// *exactly*, from integer products modulo 2^32 (e is below 2^-24, so the high product words
// vanish and only bits 2^-24 .. 2^-(h+ks) are formed): gamma = U e in FP32.
// kappa = 1 - 2^-12 keeps U below 2^31 where u reaches its bound.
//
// Accumulation. The 64-bit sums of M1 U are taken modulo 2^64 (a product alone reaches 2^62)
// beside an FP32 sum of the same products, which tells the multiple of 2^64 at the end
// (kFlushBands bounds its error). The small parts are summed in FP32 over kLowBands bands and
// then moved to the integer sums. Integer sums do not round, so the error does not grow with
// the number of bands as a running FP64 sum's does. Against 128-bit arithmetic on the drawn
// workloads, over the root of the sum of the terms' squares (achtemp, asxtemp): 1.7e-16,
// 1.9e-16 / 2.0, 2.1 / 2.1, 2.2 / 2.4, 2.5 for 1 / 5 / 64 / 200 bands; the FP64 form: 1.8,
// 2.8 / 2.1, 2.4 / 3.1, 3.6 / 4.4, 5.0.
//
// Range (fix_lane, FixInfo): |x| <= 48, x >= 0 unless the screened-exchange cutoff bounds the
// terms near x = -w, Re w >= 0, 2^(E-7) <= |w| <= 1.375 2^E - max x with
// the binary scale E of the instance's frequencies; weights whose row and column maxima over
// the bands are finite and of ordinary exponent, and whose largest product over the bands is
// within 2^-7 of the product of those maxima (the product of the split weights is exact to
// 2^-60 of that), in the bands of asxtemp and in the others each by itself; and every output's
// terms not far below the scale of its sums (kFixWeak). A warp with a lane outside, or an output
// that is too weak, takes the FP64 form.
#pragma once

#include "gpp_device.cuh"

namespace gpp {

constexpr int kStageBands = 64;    // bands of one warp's staged weights in shared memory
constexpr int kLowBands = 8;       // bands between moves of the FP32 low sums to the integers
constexpr int kFlushBands = 1024;  // bands of the modular sums between flushes
constexpr int kFixMaxGroup = 3;    // frequencies per group: more accumulators would not fit
constexpr float kFixKappa = 1.0f - 0x1p-12f;
constexpr float kFixNear = 0x1p-20f;  // |(|wdiff|^2 - 1/4)| below which FP64 decides
constexpr int kFixMinTop = 55;        // fewest bits of the largest weight (of at most 62)

// The gathered weight of one band, split: a comp 2^ka = a1 + a0 2^-32.
struct alignas(16) FixAm {
  int r1, i1, r0, i0;
};

// Per-thread constants of a (p, ig) pair.
struct FixPair {
  long long w64;       // Re w 2^(h+32)
  int ih, il;          // Im w = ih 2^-h + il 2^-(h+32)
  float w1, w2;        // Re w = w1 (multiple of 2^(E-23)) + w2
  float i1, i2;        // Im w = i1 + i2
  float n1, n2;        // (Im w)^2 = n1 (multiple of 2^(2E-21)) + n2
};

__device__ __forceinline__ double exp2i(int k) {  // 2^k, -1022 <= k <= 1023
  return __hiloint2double((k + 1023) << 20, 0);
}
__device__ __forceinline__ float exp2if(int k) { return __int_as_float((k + 127) << 23); }

__device__ __forceinline__ float fix_rcp(float d) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(d));
  return y;
}
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}
__device__ __forceinline__ int mad_hi(int a, int b, int c) {
  int d;
  asm("mad.hi.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

// a b + c modulo 2^32.
__device__ __forceinline__ int mad_lo(int a, int b, int c) {
  int d;
  asm("mad.lo.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

// What the split-integer form needs to know of an instance's frequencies, whose least is xmin
// and whose largest magnitude is xmax: whether they are in its range (1: all >= 0, 2: some
// negative), the binary scale E, and the bounds on |w|^2.
__device__ __forceinline__ FixInfo fix_info(double xmin, double xmax) {
  FixInfo f;
  f.ok = !(xmax <= 48.0) ? 0 : xmin >= 0.0 ? 1 : 2;
  int E = 2;
  while (E < 6 && xmax > 0.75 * static_cast<double>(1 << E)) ++E;
  const double lim = 1.375 * static_cast<double>(1 << E) - xmax;
  f.E = E;
  f.wlo2 = exp2i(2 * E - 14);
  f.whi2 = lim * lim;
  return f;
}

// Whether a lane's w lies in the split-integer range.
__device__ __forceinline__ bool fix_lane(double2 w, double wabs2, const FixInfo& f) {
  return w.x >= 0.0 && !lt_nonneg(wabs2, f.wlo2) && !gt_nonneg(wabs2, f.whi2);
}

// v 2^k = n1 + n0 2^-32 (|n0| <= 2^31), for |v| 2^k < 2^31 - 1; khi = (k + 32) 2^20. The
// scaling is an addition to the exponent field (k >= 0; a zero or subnormal v gives a value
// far below the last unit), the rest one FP64 -> 64-bit integer conversion (as slow as an FP64
// multiply-add, but the only FP64 instruction here).
__device__ __forceinline__ void fix_value(double v, int khi, int& n1, int& n0) {
  const double s = __hiloint2double(__double2hiint(v) + khi, __double2loint(v));
  const long long i = __double2ll_rn(s);   // v 2^(k + 32)
  n1 = static_cast<int>((i + 0x80000000LL) >> 32);
  n0 = static_cast<int>(i);
}

// The FP32 form of hi 2^-h + lo 2^-(h+32), h = 30 - E: a, a multiple of 2^(E-23), plus b.
__device__ __forceinline__ void fix_floats(int hi, int lo, int E, float& a, float& b) {
  const int q = (hi + 64) >> 7;
  a = static_cast<float>(q) * exp2if(E - 23);
  b = fmaf(static_cast<float>(lo), exp2if(E - 62), static_cast<float>(hi - (q << 7)) * exp2if(E - 30));
}

// One band-table entry's split frequency: x 2^(h+32) + 2^31 as a 64-bit integer (of its sums and
// differences with Re w the high word is then the rounded one, without a carry from the signed
// low word), and the two floats.
__device__ __forceinline__ int4 fix_x(double x, int E) {
  int hi, lo;
  float a, b;
  fix_value(x, (62 - E) << 20, hi, lo);
  if (x < 0.0 && hi == 0 && lo == 0) lo = -1;   // the sign tells the cutoff's terms
  fix_floats(hi, lo, E, a, b);
  const long long i = (static_cast<long long>(hi) << 32) + lo + 0x80000000LL;
  return make_int4(static_cast<int>(i >> 32), static_cast<int>(i), __float_as_int(a), __float_as_int(b));
}
__device__ __forceinline__ long long fix_biased(const int4& xv) {
  return (static_cast<long long>(xv.x) << 32) | static_cast<unsigned>(xv.y);
}

__device__ __forceinline__ FixPair fix_pair(double2 w, int E) {
  FixPair q;
  int wh, wl;
  fix_value(w.x, (62 - E) << 20, wh, wl);
  q.w64 = (static_cast<long long>(wh) << 32) + wl;
  fix_value(w.y, (62 - E) << 20, q.ih, q.il);
  q.il = max(q.il, -0x7fffffff);   // its negative is taken (2^-32 of the unit is below rounding)
  fix_floats(wh, wl, E, q.w1, q.w2);
  // Im w = i1 + i2: the leading 24 bits of the high part, and the rest
  const float r = static_cast<float>(q.ih);
  q.i1 = r * exp2if(E - 30);
  q.i2 = fmaf(static_cast<float>(q.il), exp2if(E - 62),
              static_cast<float>(q.ih - __float2int_rn(r)) * exp2if(E - 30));
  // (Im w)^2 = n1 + n2, n1 a multiple of 2^(2E-21)
  const float p = q.i1 * q.i1, g = exp2if(2 * E - 21);
  q.n1 = rintf(p * exp2if(21 - 2 * E)) * g;
  q.n2 = (p - q.n1) + fmaf(q.i1 + q.i1, q.i2, fmaf(q.i1, q.i1, -p));
  return q;
}

// The scales of u (or v) of one frequency: with |u| <= 1/d, ks = 31 + floor(log2 d) (U stays
// below 2^31; from d^2, whose exponent halves), s = 2^ks and c = -1/(kappa 2^(h+ks)), minus
// the unit of the residual e.
__device__ __forceinline__ int fix_ks(float d2) {
  return 31 + (((__float_as_int(d2) >> 23) - 127) >> 1);
}
__device__ __forceinline__ float2 fix_scale(int ks, int E) {
  return make_float2(exp2if(ks), (-1.0f / kFixKappa) * exp2if(-(30 - E + ks)));
}

struct FixU {
  int Ur, Ui;            // the integer part of 1/(Ar - i wi), in units of 2^-ks / kappa
  float gr, gi, ur, ui;  // gamma and the FP32 value of the whole, in the same units
};

// The FP32 part of a difference (SIDE_A: x - Re w) or sum (x + Re w): its value A1 + A2 (A1
// exact) and |A|^2 = N1 + Nm, N1 the rounded square plus n1, Nm its exact error and the rest.
struct FixN {
  float A1, A2, N1, Nm;
};
template <bool SIDE_A>
__device__ __forceinline__ FixN fix_norm(const FixPair& w, float xa, float xb) {
  FixN o;
  o.A1 = SIDE_A ? xa - w.w1 : xa + w.w1;
  o.A2 = SIDE_A ? xb - w.w2 : xb + w.w2;
  o.N1 = fmaf(o.A1, o.A1, w.n1);
  o.Nm = fmaf(o.A1, o.A1, w.n1 - o.N1) + w.n2;
  o.Nm = fmaf(o.A1 + o.A1, o.A2, o.Nm);
  return o;
}

// 1/(Ar - i wi) with Ar = x - Re w (SIDE_A) or x + Re w (then that is conj(v)), from its norm;
// with MASK zero where `on` is false.
template <bool SIDE_A, bool MASK>
__device__ __forceinline__ FixU fix_term(const FixPair& w, const FixN& n, long long xb, float2 sc,
                                         bool on) {
  FixU o;
  const long long a64 = SIDE_A ? xb - w.w64 : xb + w.w64;    // A 2^(h+32) + 2^31
  const int Ah = static_cast<int>(a64 >> 32);
  const int Al = static_cast<int>(static_cast<unsigned>(a64) - 0x80000000u);
  float rho = fix_rcp(fmaf(n.N1, 1.0f + 0x1p-12f, n.Nm));    // kappa / |A|^2
  if (MASK) rho = on ? rho : 0.0f;
  float eps = fmaf(-rho, n.N1, kFixKappa);                   // kappa - rho |A|^2
  eps = fmaf(-rho, n.Nm, eps);
  const float rs = rho * sc.x, re = rs * eps;
  const float p = n.A1 * rs;
  float cr = fmaf(n.A1, rs, -p);
  cr = fmaf(n.A1, re, cr);
  cr = fmaf(n.A2, rs, cr);
  const float q = w.i1 * rs;
  float ci = fmaf(w.i1, rs, -q);
  ci = fmaf(w.i1, re, ci);
  ci = fmaf(w.i2, rs, ci);
  o.Ur = __float2int_rn(p) + __float2int_rn(cr);
  o.Ui = __float2int_rn(q) + __float2int_rn(ci);
  o.ur = p + cr;
  o.ui = q + ci;
  // A U modulo 2^32 units of 2^-(h+ks): minus the residual (the high words of the low-limb
  // products are floors; the initial 1 takes the mean of the two out)
  int Er = mad_hi(Al, o.Ur, 1);
  Er = mad_hi(w.il, o.Ui, Er);
  Er = mad_lo(Ah, o.Ur, Er);
  Er = mad_lo(w.ih, o.Ui, Er);
  int Ei = mad_hi(Al, o.Ui, 1);
  Ei = mad_hi(-w.il, o.Ur, Ei);
  Ei = mad_lo(Ah, o.Ui, Ei);
  Ei = mad_lo(-w.ih, o.Ur, Ei);
  const float fr = static_cast<float>(Er) * sc.y, fi = static_cast<float>(Ei) * sc.y;
  o.gr = fmaf(o.ur, fr, -o.ui * fi);
  o.gi = fmaf(o.ur, fi, o.ui * fr);
  return o;
}

// Shared memory of the split-integer path, per CTA: the threads' FP64 sums (4 WG doubles,
// strided by blockDim.x), their scales (2 WG float2, likewise), then each warp's staged
// weights (kStageBands FixAm).
__host__ __device__ constexpr size_t fix_smem_bytes(int threads, int wg) {
  return static_cast<size_t>(threads) * (4 * wg * 8 + 2 * wg * 8) +
         static_cast<size_t>(threads / 32) * kStageBands * sizeof(FixAm);
}

// The weight M = am an of a band, times 2^(ka + kn - sh): M1 + M0.
struct FixM {
  int r1, i1, nr1, ni1;   // M1 and -M1
  float r0, i0, r1f, i1f;
};
__device__ __forceinline__ FixM fix_weight(const FixAm& a, double2 an, int nkhi, int sh) {
  int nr1, ni1, nr0, ni0;
  fix_value(an.x, nkhi, nr1, nr0);
  fix_value(an.y, nkhi, ni1, ni0);
  // the 60-bit products of the leading parts plus the cross products rounded to their last
  // unit (a truncation would add its mean to every weight, which random phases do not average
  // out); the products of the remainders are below that unit. |P| < 2^61
  const long long h = 0x80000000LL;
  const int qr = static_cast<int>(mad_wide(a.r1, nr0, mad_wide(-a.i1, ni0, mad_wide(a.r0, nr1, mad_wide(a.i0, -ni1, h)))) >> 32);
  const int qi = static_cast<int>(mad_wide(a.r1, ni0, mad_wide(a.i1, nr0, mad_wide(a.r0, ni1, mad_wide(a.i0, nr1, h)))) >> 32);
  const long long Pr = mad_wide(a.r1, nr1, mad_wide(-a.i1, ni1, qr));
  const long long Pi = mad_wide(a.r1, ni1, mad_wide(a.i1, nr1, qi));
  const unsigned half = 1u << (sh - 1);   // (sh <= 30: one word)
  FixM m;
  m.r1 = static_cast<int>((Pr + half) >> sh);
  m.i1 = static_cast<int>((Pi + half) >> sh);
  // what the shift drops, signed: the low sh bits as the top of a word
  m.r0 = static_cast<float>(static_cast<int>(static_cast<unsigned>(Pr) << (32 - sh))) * 0x1p-32f;
  m.i0 = static_cast<float>(static_cast<int>(static_cast<unsigned>(Pi) << (32 - sh))) * 0x1p-32f;
  m.r1f = static_cast<float>(m.r1);
  m.i1f = static_cast<float>(m.i1);
  m.nr1 = -m.r1;
  m.ni1 = -m.i1;
  return m;
}

// What a pair's band loops share, and the scales of the weights of one class of bands (the bands
// of asxtemp, or the others; see FixScale), nkhi = (kn + 32) 2^20 and so on.
struct FixCtx {
  int64_t G;
  const double2* an;   // the pair's column of aqsntemp (stride G)
  const double2* am;   // the row of weights
  const double2* w64;  // the FP64 w, for exact branch decisions
  const BandEntry* bt;
  int W, nkhi, akhi, sh;
  FixAm* stage;
};

// The screened-exchange cutoff (negative frequencies only): a term whose |ssx| / |I|, which is
// |w|^2 / (|A| |S|) on branch 1 and |w| / (2 |S|) on branch 2, exceeds sexcut leaves asxtemp.
// So |w|^4 > sx2 |S|^2 (branch 1: |A|^2, branch 2: 4 |w|^2) is tested, in FP32 and, within
// kFixNearCut of equality, in FP64 as the general form does. A kept term has
//   |S| >= |w| min(sqrt(1 + 1 / sexcut) - 1, 1 / (2 sexcut)),
// which bounds v near x = -w; v there, above the bound the sums are scaled for, is taken at a
// scale 2^-delta and its product shifted back (the sums are modular).
constexpr float kFixNearCut = 0x1p-18f;
struct FixCut {
  float w4, w24, sx2f;   // |w|^4, 4 |w|^2
  double sx2;
  int delta[kFixMaxGroup];
};

// v 2^k for a zero v or one that stays normal.
__device__ __forceinline__ double fix_shift(double v, int k) {
  const int hi = __double2hiint(v);
  return __hiloint2double((hi & 0x7fffffff) == 0 ? hi : hi + (k << 20), __double2loint(v));
}
// D 2^e, rounded by one conversion: an FP64 instruction takes as long as 30 of these. (By FP64
// arithmetic on halves of the sums a pair's FP64 instructions were 107, now 44: B = 37, P = 95,
// G = 1901, nw = 2: 181 -> 168 us; B = 32, P = 64, G = 512, nw = 3: 69.8 -> 65.9 us.)
static __device__ __noinline__ double fix_round(__int128 D, int e) {
  const long long hi = static_cast<long long>(D >> 64), lo = static_cast<long long>(D);
  // the bits beyond the conversion's 64 are dropped (|D| >= 2^63 then)
  const int k = hi == (lo >> 63) ? 0 : 65 - __clzll(hi ^ (hi >> 63));
  return fix_shift(static_cast<double>(static_cast<long long>(D >> k)), k + e);
}

// Bands [b0, b1) of the thread's pair, WG frequencies from iw0, into the thread's FP64 sums
// st[k blockDim.x] (units of kappa 2^ks M with the ks of u; values 4 iw + {0, 1}: sum M u, and
// with OCC + {2, 3}: sum M u - sum M v), added to them, or with `fresh` replacing them.
template <int WG, bool OCC, bool CUT>
__device__ __forceinline__ void fix_range(int b0, int b1, bool fresh, const FixCtx& ctx, int iw0,
                                          const FixPair& w, const FixCut& cut, double* st,
                                          const float2* sc) {
  const int nt = blockDim.x, lane = threadIdx.x & 31;
  const int64_t G = ctx.G;
  int nkhi = ctx.nkhi, sh = ctx.sh;
  // (keeps the compiler from forming these again in every band: 1%)
  asm volatile("" : "+r"(nkhi), "+r"(sh));
  FixAm* const stage = ctx.stage;
  // bands of the modular sums: the FP32 sum beside them has to be good to 2^62 (terms below
  // 2^62, with the cutoff's scale 2^69)
  constexpr int kFlush = CUT ? 128 : kFlushBands;
#pragma unroll 1
  for (int f0 = b0; f0 < b1; f0 += kFlush) {
    const int f1 = min(f0 + kFlush, b1);
    long long acc[4 * WG];
    float aH[4 * WG], aL[4 * WG];
#pragma unroll
    for (int k = 0; k < 4 * WG; ++k) {
      acc[k] = 0;
      aH[k] = 0.0f;
      aL[k] = 0.0f;
    }
    double2 an_next = ldg2(ctx.an + static_cast<int64_t>(f0) * G);
#pragma unroll 1
    for (int s0 = f0; s0 < f1; s0 += kStageBands) {
      const int s1 = min(s0 + kStageBands, f1);
      __syncwarp();
      for (int b = s0 + lane; b < s1; b += 32) {   // this warp's weights of the next bands
        const double2 a = ldg2(ctx.am + b);
        FixAm e;
        fix_value(a.x, ctx.akhi, e.r1, e.r0);
        fix_value(a.y, ctx.akhi, e.i1, e.i0);
        stage[b - s0] = e;
      }
      __syncwarp();
#pragma unroll 1
      for (int l0 = s0; l0 < s1; l0 += kLowBands) {
        const int l1 = min(l0 + kLowBands, s1);
#pragma unroll 1
        for (int b = l0; b < l1; ++b) {
          const double2 an = an_next;
          if (b + 1 < b1) an_next = ldg2(ctx.an + static_cast<int64_t>(b + 1) * G);
          const FixM m = fix_weight(stage[b - s0], an, nkhi, sh);
          const BandEntry* btb = ctx.bt + static_cast<int64_t>(b) * ctx.W + iw0;
          int4 xv[WG];
          FixN na[WG];
          float d[WG];   // |wdiff|^2 - 1/4: its sign decides branch 1
          float dmin = 1.0f;
#pragma unroll
          for (int k = 0; k < WG; ++k) {
            xv[k] = __ldg(&btb[k].fx);
            na[k] = fix_norm<true>(w, __int_as_float(xv[k].z), __int_as_float(xv[k].w));
            d[k] = (na[k].N1 - 0.25f) + na[k].Nm;
            dmin = fminf(dmin, fabsf(d[k]));
          }
          if (__any_sync(0xffffffffu, dmin <= kFixNear)) {   // rare: the FP64 form's decisions
            const double2 wv = ldg2(ctx.w64);
#pragma unroll
            for (int k = 0; k < WG; ++k) {
              const double a = __ldg(&btb[k].lo.x) - wv.x;
              d[k] = gt_nonneg(fma(a, a, wv.y * wv.y), kLimitTwo) ? 1.0f : -1.0f;
            }
          }
#pragma unroll
          for (int k = 0; k < WG; ++k) {
            {
              const FixU u = fix_term<true, true>(w, na[k], fix_biased(xv[k]), sc[2 * k * nt], d[k] > 0.0f);
              acc[4 * k] = mad_wide(m.r1, u.Ur, mad_wide(m.ni1, u.Ui, acc[4 * k]));
              acc[4 * k + 1] = mad_wide(m.r1, u.Ui, mad_wide(m.i1, u.Ur, acc[4 * k + 1]));
              aH[4 * k] = fmaf(m.r1f, u.ur, fmaf(-m.i1f, u.ui, aH[4 * k]));
              aH[4 * k + 1] = fmaf(m.r1f, u.ui, fmaf(m.i1f, u.ur, aH[4 * k + 1]));
              aL[4 * k] += fmaf(m.r1f, u.gr, fmaf(-m.i1f, u.gi, fmaf(m.r0, u.ur, -m.i0 * u.ui)));
              aL[4 * k + 1] += fmaf(m.r1f, u.gi, fmaf(m.i1f, u.gr, fmaf(m.r0, u.ui, m.i0 * u.ur)));
            }
            if (OCC) {   // v = conj of the computed value
              const FixN ns = fix_norm<false>(w, __int_as_float(xv[k].z), __int_as_float(xv[k].w));
              const float2 ss = sc[(2 * k + 1) * nt];
              bool on = true;
              if (CUT && fix_biased(xv[k]) < 0x80000000LL) {   // x < 0: warp-uniform
                const float NS = ns.N1 + ns.Nm;
                const bool b1 = d[k] > 0.0f;
                const float lim = cut.sx2f * NS * (b1 ? na[k].N1 + na[k].Nm : cut.w24);
                bool drop = cut.w4 > lim;
                const bool edge = fabsf(cut.w4 - lim) <= kFixNearCut * cut.w4;
                if (__any_sync(0xffffffffu, edge)) {
                  const double2 wv = ldg2(ctx.w64);
                  const double x = __ldg(&btb[k].lo.x), a = x - wv.x, s = x + wv.x, i2 = wv.y * wv.y;
                  const double A2 = fma(a, a, i2), S2 = fma(s, s, i2), w2 = fma(wv.x, wv.x, i2);
                  const bool e = b1 ? gt_nonneg(w2 * w2 * rcp_refined(A2 * S2), cut.sx2)
                                    : gt_nonneg(w2, 4.0 * cut.sx2 * S2);
                  drop = edge ? e : drop;
                }
                // |S| below 2^(31 - ks): beyond this scale
                const int e = __float_as_int(ss.x) >> 23;   // ks + 127
                const bool small = !drop && NS < __int_as_float((443 - 2 * e) << 23);
                on = !drop && !small;
                if (__any_sync(0xffffffffu, drop && b1)) {   // take sum M u back out of asxtemp
                  const FixU u = fix_term<true, true>(w, na[k], fix_biased(xv[k]), ss, drop && b1);
                  acc[4 * k + 2] = mad_wide(m.r1, u.Ur, mad_wide(m.ni1, u.Ui, acc[4 * k + 2]));
                  acc[4 * k + 3] = mad_wide(m.r1, u.Ui, mad_wide(m.i1, u.Ur, acc[4 * k + 3]));
                  aH[4 * k + 2] = fmaf(m.r1f, u.ur, fmaf(-m.i1f, u.ui, aH[4 * k + 2]));
                  aH[4 * k + 3] = fmaf(m.r1f, u.ui, fmaf(m.i1f, u.ur, aH[4 * k + 3]));
                  aL[4 * k + 2] += fmaf(m.r1f, u.gr, fmaf(-m.i1f, u.gi, fmaf(m.r0, u.ur, -m.i0 * u.ui)));
                  aL[4 * k + 3] += fmaf(m.r1f, u.gi, fmaf(m.i1f, u.gr, fmaf(m.r0, u.ui, m.i0 * u.ur)));
                }
                if (__any_sync(0xffffffffu, small)) {
                  const int dl = cut.delta[k];
                  const float up = exp2if(dl);
                  const FixU u = fix_term<false, true>(w, ns, fix_biased(xv[k]),
                                                       make_float2(ss.x * exp2if(-dl), ss.y * up), small);
                  const long long pr = mad_wide(m.r1, u.Ur, mad_wide(m.i1, u.Ui, 0));
                  const long long pi = mad_wide(m.i1, u.Ur, mad_wide(m.nr1, u.Ui, 0));
                  acc[4 * k + 2] += static_cast<long long>(static_cast<unsigned long long>(pr) << dl);
                  acc[4 * k + 3] += static_cast<long long>(static_cast<unsigned long long>(pi) << dl);
                  aH[4 * k + 2] = fmaf(up, fmaf(m.r1f, u.ur, m.i1f * u.ui), aH[4 * k + 2]);
                  aH[4 * k + 3] = fmaf(up, fmaf(m.i1f, u.ur, -m.r1f * u.ui), aH[4 * k + 3]);
                  aL[4 * k + 2] = fmaf(up, fmaf(m.r1f, u.gr, fmaf(m.i1f, u.gi, fmaf(m.r0, u.ur, m.i0 * u.ui))), aL[4 * k + 2]);
                  aL[4 * k + 3] = fmaf(up, fmaf(m.i1f, u.gr, fmaf(-m.r1f, u.gi, fmaf(m.i0, u.ur, -m.r0 * u.ui))), aL[4 * k + 3]);
                }
              }
              const FixU u = fix_term<false, CUT>(w, ns, fix_biased(xv[k]), ss, on);
              acc[4 * k + 2] = mad_wide(m.r1, u.Ur, mad_wide(m.i1, u.Ui, acc[4 * k + 2]));
              acc[4 * k + 3] = mad_wide(m.i1, u.Ur, mad_wide(m.nr1, u.Ui, acc[4 * k + 3]));
              aH[4 * k + 2] = fmaf(m.r1f, u.ur, fmaf(m.i1f, u.ui, aH[4 * k + 2]));
              aH[4 * k + 3] = fmaf(m.i1f, u.ur, fmaf(-m.r1f, u.ui, aH[4 * k + 3]));
              aL[4 * k + 2] += fmaf(m.r1f, u.gr, fmaf(m.i1f, u.gi, fmaf(m.r0, u.ur, m.i0 * u.ui)));
              aL[4 * k + 3] += fmaf(m.i1f, u.gr, fmaf(-m.r1f, u.gi, fmaf(m.i0, u.ur, -m.r0 * u.ui)));
            }
          }
        }
        // the low sums (below 2^43) into the integer sums in units of 2^12; the rest stays
#pragma unroll
        for (int k = 0; k < 4 * WG; ++k)
          if (OCC || (k & 2) == 0) {
            const int r = __float2int_rn(aL[k] * 0x1p-12f);
            acc[k] = mad_wide(r, 4096, acc[k]);
            aL[k] = fmaf(-4096.0f, static_cast<float>(r), aL[k]);
          }
      }
    }
#pragma unroll
    for (int k = 0; k < 4 * WG; ++k) acc[k] += __float2int_rn(aL[k]);
    // the sums are acc + j 2^64, with j from the FP32 sums (mostly zero)
    int j[4 * WG], any = 0;
#pragma unroll
    for (int k = 0; k < 4 * WG; ++k) {
      const float top = static_cast<float>(static_cast<int>(acc[k] >> 32)) * 0x1p-32f;
      j[k] = __float2int_rn(fmaf(aH[k], 0x1p-64f, -top));
      any |= j[k];
    }
    const bool carry = __any_sync(0xffffffffu, any != 0);
    auto total = [&](int k) { return static_cast<__int128>(j[k]) * (static_cast<__int128>(1) << 64) + acc[k]; };
    auto sum = [&](int k) { return carry ? fix_round(total(k), 0) : static_cast<double>(acc[k]); };
    auto put = [&](int k, double v) { st[k * nt] = (!fresh || f0 > b0) ? st[k * nt] + v : v; };
#pragma unroll
    for (int k = 0; k < WG; ++k) {
      if (!OCC) {
        put(4 * k, sum(4 * k));
        put(4 * k + 1, sum(4 * k + 1));
        continue;
      }
      const int dl = (__float_as_int(sc[2 * k * nt].x) - __float_as_int(sc[(2 * k + 1) * nt].x)) >> 23;
#pragma unroll
      for (int c = 4 * k; c < 4 * k + 2; ++c) {
        put(c, sum(c));
        // the difference (which may cancel) is exact and rounded once
        const int q = max(-dl, 0);
        put(c + 2, fix_round((total(c) << q) - (total(c + 2) << max(dl, 0)), -q));
      }
    }
  }
}

// The high words of doubles without the sign order like their magnitudes and, read as
// exponent.mantissa fixed-point numbers, are their binary logarithms (plus 1023) to within
// 0.087 from above.
__device__ __forceinline__ unsigned fix_hi_max(double2 v) {
  return static_cast<unsigned>(
      max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff));
}
// k with 2^k v < 2^30 for every value whose high word is at most m, also after rounding to an
// integer; false if m's exponent is out of the ordinary (m = 0: k = 0).
__device__ __forceinline__ bool fix_exponent(unsigned m, int& k) {
  const int e = static_cast<int>((m + 1) >> 20);          // a mantissa of all ones counts as the next binade
  k = m == 0 ? 0 : 30 - (e - 1022);     // e <= 2047 (infinity, NaN) gives k < 0
  return m == 0 || (k >= 0 && k <= 400);
}

// The weights' scales from the largest high words over the bands of the column of aqsntemp
// (mn), of the row of weights (ma) and of their products' sums (mp): kn, ka, and the shift sh
// that takes the largest |M| comp to 31 bits. False outside the range.
__device__ __forceinline__ bool fix_weight_scale(unsigned mn, unsigned ma, unsigned mp, int& kn,
                                                 int& ka, int& sh) {
  const bool n_ok = fix_exponent(mn, kn), a_ok = fix_exponent(ma, ka);
  // every |M| comp 2^(ka + kn) < 2^top: twice (complex) the largest product, 0.18 for its
  // logarithm
  const int top = static_cast<int>((mp + (1u << 20) + 188744u) >> 20) + 1 - 2046 + ka + kn;
  sh = max(min(top - 31, 30), 1);
  return n_ok && a_ok && (mn == 0 || ma == 0 || top >= kFixMinTop);
}

constexpr int kFixNoWeight = 401;   // beyond fix_exponent's

// The scales of one class of bands [b0, b1) for a pair, from the magnitudes of the column of
// aqsntemp, of the row of weights and of their products: am 2^ka and an 2^kn as integers, their
// product shifted by sh. `any`: it has weights that are not zero (an inert lane has none).
struct FixScale {
  int kn, ka, sh;
  bool any;
  __device__ __forceinline__ int unit() const { return sh - ka - kn; }   // log2 of M1's unit
};
__device__ __forceinline__ bool fix_scales(int b0, int b1, int64_t G, const double2* an_ptr,
                                           const double2* am_ptr, bool live, FixScale& s) {
  unsigned mn = 0, ma = 0, mp = 0;
#pragma unroll 8
  for (int b = b0; b < b1; ++b) {
    const unsigned hn = fix_hi_max(ldg2(an_ptr + static_cast<int64_t>(b) * G));
    const unsigned ha = fix_hi_max(ldg2(am_ptr + b));
    mn = max(mn, hn);
    ma = max(ma, ha);
    mp = max(mp, hn + ha);
  }
  if (!live) mn = mp = 0;   // whatever its column holds: the values stay finite and I is zero
  s.any = mn != 0 && ma != 0;
  const bool ok = fix_weight_scale(mn, ma, mp, s.kn, s.ka, s.sh);
  // without weights a unit far below any other, which tells them apart (ka stays the warp's: its
  // lanes share the staged weights)
  if (mn == 0) s.kn = kFixNoWeight;
  if (ma == 0) s.ka = kFixNoWeight;
  return ok;
}

// Whether an output is too weak for the scale that its sums were rounded at. A sum of n terms M u
// carries an error of about sqrt(n) 2^-56 of its scale, which is 2^62 in the units of M1 U; so
// relative to its own terms it is as good as the FP64 form's only while these are not far below
// that. They are where other bands hold the large weights and add nothing to this output
// (branch 2, the cutoff), or where one light band sets the scale of u. The line, 2^-kFixWeak of sqrt(n)
// times the scale, bounds the error by about 2^-50 of the root of the sum of the terms' squares. It is
// drawn for the largest lane of a warp, since the results are sums over all pairs: of 60000
// pairs of 1..512 bands drawn as in the package's inputs, that lane's terms (root mean square) lie
// at 2^-3.5 in the median and at 2^-5.3 at the least. (On the host, 64 bands, nw = 3: error 1.4e-16
// of the terms there, FP64 form 2.4e-16.)
// Two stages: the sums themselves, whose squares are the terms' powers but for what cancels, cost
// a few instructions per pair (fix_band_loop's result); only a warp that this doubts has the
// terms' powers formed (fix_strong).
constexpr int kFixWeak = 6;
constexpr int kFixNone = -0x20000000;   // the logarithm of zero: below all others, and so is a sum with it

// log2 (sqrt(n)) in units of 2^-18.
__device__ __forceinline__ int fix_half_log(float n) { return (__float_as_int(n) - (127 << 23)) >> 6; }
// The least root that n terms M1 U may add up to in one class of bands, for U in units of 1 (plus
// 1023); `any`: the pair has weights there that are not zero.
__device__ __forceinline__ int fix_least(bool any, int n) {
  return any && n > 0 ? fix_half_log(static_cast<float>(n)) + ((1023 + 62 - kFixWeak) << 18) : kFixNone;
}
// log2 of the larger component (plus 1023), in units of 2^-18.
__device__ __forceinline__ int fix_log_max(double re, double im) {
  const unsigned m = fix_hi_max(make_double2(re, im));
  return m == 0 ? kFixNone : static_cast<int>(m >> 2);
}

// |v|^2 2^(2 k) in FP32 from the leading 20 bits of each component (conversions of FP64 are as slow
// as its arithmetic); below FP32's range 0.
__device__ __forceinline__ float fix_square_of(double2 v, int k) {
  auto part = [&](double c) {
    const int h = (__double2hiint(c) & 0x7fffffff) - ((896 - k) << 20);
    return __int_as_float(max(h, 0) << 3);
  };
  const float r = part(v.x), i = part(v.y);
  return fmaf(r, r, i * i);
}

// The scales of one frequency's u and v, from the distance of its frequencies [lo, hi] from w and
// -w, less the FP32 rounding. CUT: dcut is the least |S| of a kept term with x < 0; `delta` is
// how far below the scale of most terms the kept ones near x = -w may lie.
template <bool CUT>
__device__ __forceinline__ void fix_distances(const FixPair& w, float w2f, float lo, float hi,
                                              float dcut, int& ksu, int& ksv, int& delta) {
  const float da = fmaxf(0.0f, fmaxf(lo - w.w1, w.w1 - hi));
  const float dA2 = fmaxf(0.25f, fmaf(da, da, w.i1 * w.i1) * (1.0f - 0x1p-16f));
  const float sr = fmaxf(lo + w.w1, -(hi + w.w1));
  const float dr = CUT ? fmaxf(sr, 0.0f) : sr;
  float dS2 = fmaf(dr, dr, w.i1 * w.i1) * (1.0f - 0x1p-17f);
  if (CUT) {
    const float least = fmaxf(dS2, dcut * dcut), most = fminf(w2f * (1.0f - 0x1p-17f), 0.0625f);
    dS2 = fmaxf(least, most);
    delta = fix_ks(dS2) - fix_ks(least);
  }
  ksu = fix_ks(dA2);
  ksv = fix_ks(dS2);
}
// The least |S| of a kept term with x < 0 (see FixCut).
__device__ __forceinline__ float fix_dcut(float w2f, float sx2f) {
  const float sc = sqrtf(sx2f);
  return sqrtf(w2f) * fminf(1.0f, fminf(sqrtf(1.0f + 1.0f / sc) - 1.0f, 0.5f / sc)) * (1.0f - 0x1p-17f);
}

// Whether every output of the warp is strong enough, by the powers of its terms: the sums over
// the bands of |M u|^2 on branch 1 and of |M v|^2 (with the cutoff: of the kept terms' 4 |M w u v|^2
// or |M v|^2), in FP32, counting only terms that are clearly on their side of a threshold; a weight
// below FP32's range still counts a little, so that only an output without terms is zero.
template <int W, bool CUT>
__device__ __noinline__ bool fix_strong(int B, int64_t G, int nocc, const double2* __restrict__ an_ptr,
                                        const double2* __restrict__ am_ptr,
                                        const BandEntry* __restrict__ bt, bool live, double2 wv,
                                        double2 I, int E, double sx2,
                                        const double* __restrict__ xrange) {
  const FixPair w = fix_pair(wv, E);
  const float wr = static_cast<float>(wv.x), wi = static_cast<float>(wv.y), wi2 = wi * wi;
  const float w2 = fmaf(wr, wr, wi2), sx2f = static_cast<float>(sx2);
  const int lgI = live ? fix_log_max(fma(I.x, wv.x, -I.y * wv.y), fma(I.x, wv.y, I.y * wv.x)) : kFixNone;
  float pu[2][W], pv[W];
  int unit[2], least[2];
#pragma unroll
  for (int k = 0; k < W; ++k) pu[0][k] = pu[1][k] = pv[k] = 0.0f;
#pragma unroll
  for (int c = 0; c < 2; ++c) {   // the bands of asxtemp, the others
    const int b0 = c == 0 ? 0 : nocc, b1 = c == 0 ? nocc : B;
    FixScale s;
    fix_scales(b0, b1, G, an_ptr, am_ptr, live, s);
    unit[c] = s.unit();
    least[c] = fix_least(s.any, b1 - b0);
    const float m1 = exp2if(60 - s.sh);   // of (am 2^(ka - 30)) (an 2^(kn - 30)) in M1's units
#pragma unroll 2
    for (int b = b0; b < b1; ++b) {
      const double2 an = ldg2(an_ptr + static_cast<int64_t>(b) * G), am = ldg2(am_ptr + b);
      const float m2 = fmaxf(fix_square_of(an, s.kn - 30) * fix_square_of(am, s.ka - 30), 1e-37f) * m1 * m1;
#pragma unroll
      for (int k = 0; k < W; ++k) {
        const float x = static_cast<float>(__ldg(&bt[static_cast<int64_t>(b) * W + k].lo.x));
        const float a = x - wr, a2 = fmaf(a, a, wi2), t = x + wr, s2 = fmaf(t, t, wi2);
        const bool b1 = a2 > 0.25f * (1.0f + 0x1p-12f), b2 = a2 < 0.25f * (1.0f - 0x1p-12f);
        const float ra = fix_rcp(a2), rs = fix_rcp(s2);
        if (b1) pu[c][k] = fmaf(m2, ra, pu[c][k]);
        if (c == 0) {
          const float h = CUT && b1 ? w2 * ra * rs : 0.25f * rs;   // with the cutoff |ssx / (I w)|^2
          if (!CUT || ((b1 || b2) && (x >= 0.0f || h * w2 < sx2f * (1.0f - 0x1p-10f))))
            pv[k] += m2 * (4.0f * h);
        }
      }
    }
  }
  const float dcut = CUT ? fix_dcut(w2, sx2f) : 0.0f;
  bool strong = true;
#pragma unroll
  for (int k = 0; k < W; ++k) {
    int ku, kv, delta;
    fix_distances<CUT>(w, w2, static_cast<float>(xrange[k]), static_cast<float>(xrange[kMaxNw + k]),
                       dcut, ku, kv, delta);
    // of class c, times |I w|: a power as the logarithm of its root, and a scale's least root
    auto root = [&](float e, int c) {
      return e > 0.0f && least[c] != kFixNone ? lgI + (1023 << 18) + fix_half_log(e) + (unit[c] << 18)
                                              : kFixNone;
    };
    auto floor_of = [&](float e, int c, int ks) {
      return e > 0.0f && least[c] != kFixNone ? lgI + least[c] + ((unit[c] - ks) << 18) : kFixNone;
    };
    const int lu = floor_of(pu[0][k], 0, ku);
    const int sa = max(root(pu[0][k], 0), root(pu[1][k], 1)), la = max(lu, floor_of(pu[1][k], 1, ku));
    const int ss = root((CUT ? 0.0f : pu[0][k]) + pv[k], 0), ls = max(lu, floor_of(pv[k], 0, kv));
    strong = strong && __reduce_max_sync(0xffffffffu, sa) >= __reduce_max_sync(0xffffffffu, la) &&
             __reduce_max_sync(0xffffffffu, ss) >= __reduce_max_sync(0xffffffffu, ls);
  }
  return strong;
}

// Whether an output of N frequencies may be too weak for its scale, by the sums alone: those of a
// pair, as fix_range left them in st, against half the least root of each class of its terms (a warp
// with a single pair, past the last whole 32 G-vectors, would be doubted half of the time at all of
// it). Passed by a lane whose scale, times |I w|, is within 2^1.5 of the largest in the warp: no single
// lane decides, whose sum may be small by chance.
template <int N>
__device__ __noinline__ bool fix_doubt(const double* st, const float2* sc, int nt, int nocc, int B,
                                       const FixCtx o, const FixCtx r, double Iwr, double Iwi) {
  const int lgI = static_cast<int>(fix_hi_max(make_double2(Iwr, Iwi)) >> 2), one = 1 << 18;
  auto unit_of = [](const FixCtx& c) { return c.sh + 64 - (c.nkhi >> 20) - (c.akhi >> 20); };
  auto least_of = [&](const FixCtx& c, int n) {
    const int none = (kFixNoWeight + 32) << 20;
    const int l = fix_least(c.nkhi != none && c.akhi != none, n);
    return l == kFixNone ? l : l + unit_of(c) * one;
  };
  const int exo = unit_of(o), exr = unit_of(r);
  const int no = least_of(o, nocc), nr = least_of(r, B - nocc);
  bool doubt = false;
  auto test = [&](double re, double im, int unit, int least) {
    const int m = fix_log_max(re, im);
    const bool ok = least == kFixNone || (m != kFixNone && m + unit * one >= least - one);
    const int strong = ok ? lgI + least : 2 * kFixNone;
    doubt |= __reduce_max_sync(0xffffffffu, strong) <
             __reduce_max_sync(0xffffffffu, lgI + least) - 3 * one / 2;
  };
#pragma unroll
  for (int k = 0; k < N; ++k) {
    auto ks = [&](int q) { return (__float_as_int(sc[q * nt].x) >> 23) - 127; };
    const int ku = ks(2 * k), kv = ks(2 * k + 1);
    auto least = [&](int l, int ks) { return l == kFixNone ? l : l - ks * one; };
    test(st[4 * k * nt], st[(4 * k + 1) * nt], (nocc < B ? exr : exo) - ku, least(max(no, nr), ku));
    if (nocc > 0)
      test(st[(4 * k + 2) * nt], st[(4 * k + 3) * nt], exo - ku, least(no, min(ku, kv)));
  }
  return doubt;
}

// All bands of the thread's pair by the split-integer form, multiplied by Iw = I w and added
// to tacc[4 W]. kFixOut (nothing added): a lane of the warp is out of range. kFixDoubt: an output
// of the warp may be too weak for its scale; the sums are then in `apart` (W <= kFixMaxGroup) or
// added to tacc all the same. B >= 1.
//
// Bands [0, nocc), which enter both sums, and the rest have weight scales of their own, so that
// asxtemp is as accurate where its bands' weights are far below the others' (or above).
enum FixResult { kFixOut, kFixDoubt, kFixDone };
template <int W, bool CUT>
__device__ __noinline__ FixResult fix_band_loop(int B, int64_t G, int nocc,
                                                const double2* __restrict__ an_ptr,
                                                const double2* __restrict__ am_ptr,
                                                const BandEntry* __restrict__ bt, bool live,
                                                double2 wv, const double2* __restrict__ w_ptr,
                                                double2 I, int E, double sx2,
                                                const double* __restrict__ xrange,
                                                unsigned char* smem, double* tacc, double* apart) {
  constexpr int WG = W < kFixMaxGroup ? W : kFixMaxGroup;
  const int nt = blockDim.x, warp = threadIdx.x >> 5;
  double* st = reinterpret_cast<double*>(smem) + threadIdx.x;
  float2* sc = reinterpret_cast<float2*>(smem + static_cast<size_t>(nt) * 4 * WG * 8) + threadIdx.x;
  FixScale o, r;
  const bool o_ok = fix_scales(0, nocc, G, an_ptr, am_ptr, live, o);
  const bool r_ok = fix_scales(nocc, B, G, an_ptr, am_ptr, live, r);
  if (!__all_sync(0xffffffffu, o_ok && r_ok)) return kFixOut;
  FixAm* const stage = reinterpret_cast<FixAm*>(smem + static_cast<size_t>(nt) * 6 * WG * 8) +
                       warp * kStageBands;
  const FixCtx ctx{G, an_ptr, am_ptr, w_ptr, bt, W, (o.kn + 32) << 20, (o.ka + 32) << 20, o.sh, stage};
  const FixCtx ctx_r{G, an_ptr, am_ptr, w_ptr, bt, W, (r.kn + 32) << 20, (r.ka + 32) << 20, r.sh, stage};
  const int exo = o.unit(), exr = r.unit(), ex = nocc < B ? exr : exo;
  const FixPair w = fix_pair(wv, E);
  // I w / (2 kappa); the 2 is in the shifts below (so that nothing overflows that I w does not)
  const double Ir = I.x * (0.5 / kFixKappa), Ii = I.y * (0.5 / kFixKappa);
  const double Iwr = fma(Ir, wv.x, -Ii * wv.y), Iwi = fma(Ir, wv.y, Ii * wv.x);
  const float wrf = w.w1 + w.w2, w2f = fmaf(wrf, wrf, w.i1 * w.i1);
  float dcut = 0.0f;
  FixCut cut{w2f * w2f, 4.0f * w2f, static_cast<float>(sx2), sx2, {}};
  if (CUT) {
    dcut = fix_dcut(w2f, cut.sx2f);
    // a cutoff so high that its least |S| needs a scale far from the others', or so low that
    // its tests leave FP32's range
    const bool good = dcut >= 0x1p-6f * fminf(sqrtf(w2f), 0.25f) && sqrtf(cut.sx2f) > 0x1p-20f;
    if (!__all_sync(0xffffffffu, good)) return kFixOut;
  }
  bool doubt = false;
  auto group = [&](auto tag, int iw0) {
    constexpr int N = decltype(tag)::value;
    int ks[2 * N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
      fix_distances<CUT>(w, w2f, static_cast<float>(xrange[iw0 + k]),
                         static_cast<float>(xrange[kMaxNw + iw0 + k]), dcut, ks[2 * k], ks[2 * k + 1],
                         cut.delta[k]);
      sc[2 * k * nt] = fix_scale(ks[2 * k], E);
      sc[(2 * k + 1) * nt] = fix_scale(ks[2 * k + 1], E);
    }
    // units: M1 = M 2^(ka + kn - sh), U = u kappa 2^ks
    if (nocc > 0) {
      fix_range<N, true, CUT>(0, nocc, true, ctx, iw0, w, cut, st, sc);
      if (nocc < B) {
#pragma unroll
        for (int k = 0; k < N; ++k) {   // the others' units
          st[4 * k * nt] = fix_shift(st[4 * k * nt], exo - exr);
          st[(4 * k + 1) * nt] = fix_shift(st[(4 * k + 1) * nt], exo - exr);
        }
      }
    }
    if (nocc < B) fix_range<N, false, false>(nocc, B, nocc == 0, ctx_r, iw0, w, cut, st, sc);
    doubt |= fix_doubt<N>(st, sc, nt, nocc, B, ctx, ctx_r, Iwr, Iwi);
    const bool aside = W <= kFixMaxGroup && doubt;
#pragma unroll
    for (int k = 0; k < N; ++k) {   // tacc += I w times the pair's sums (units: I w / (2 kappa))
      const double ar = fix_shift(st[4 * k * nt], ex - ks[2 * k] + 1);
      const double ai = fix_shift(st[(4 * k + 1) * nt], ex - ks[2 * k] + 1);
      double sr = 0.0, si = 0.0;   // asxtemp: (its bands' achtemp - sum M v) / 2
      if (nocc > 0) {
        sr = fix_shift(st[(4 * k + 2) * nt], exo - ks[2 * k]);
        si = fix_shift(st[(4 * k + 3) * nt], exo - ks[2 * k]);
      }
      double* p = tacc + 4 * (iw0 + k);
      double v[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = aside ? 0.0 : p[i];
      if (aside) p = apart + 4 * (iw0 + k);
      p[0] = fma(Iwr, ar, fma(-Iwi, ai, v[0]));
      p[1] = fma(Iwr, ai, fma(Iwi, ar, v[1]));
      p[2] = fma(Iwr, sr, fma(-Iwi, si, v[2]));
      p[3] = fma(Iwr, si, fma(Iwi, sr, v[3]));
    }
  };
  // frequency groups of at most three; the weights are formed again for each
  constexpr int NG = (W + kFixMaxGroup - 1) / kFixMaxGroup;
  constexpr int LO = W / NG, NHI = W - LO * NG;   // NHI groups of LO + 1, then groups of LO
#pragma unroll
  for (int g = 0; g < NG; ++g) {
    const int iw0 = g * LO + (g < NHI ? g : NHI);
    if (g < NHI)
      group(IntTag<LO + 1>(), iw0);
    else
      group(IntTag<LO>(), iw0);
  }
  return doubt ? kFixDoubt : kFixDone;
}

}  // namespace gpp
