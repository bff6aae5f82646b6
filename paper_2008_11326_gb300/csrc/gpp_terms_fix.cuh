// The split-integer evaluation of the FP64 fast path's terms (gpp_terms_f64.cuh, "fast
// path"), for warps whose inputs lie in its range.
//
// Why. GB300's FP64 pipe issues one warp instruction per SM sub-partition every 64 cycles,
// the integer and FP32 pipes one every 1 (FFMA), 2 (IMAD, shift, convert) or 4 (32 x 32 -> 64
// bit multiply-add) cycles (measured: 1.9 DFMA, 113 FFMA, 60 IMAD, 30 IMAD.WIDE per clock per
// SM). A term of the sum costs 18 FP64 instructions per frequency (1152 cycles); the same
// term on 32-bit integers and floats, to at least the same accuracy, costs about 300.
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
// (kFlushBands bounds its error). The small parts are summed in FP32 over kLowBands bands,
// then in FP64. Integer sums do not round, so the error does not grow with the number of
// bands as a running FP64 sum's does. Against 128-bit arithmetic, per (p, ig) sum relative to
// its root mean square: 2^-53.1 / -52.7 / -52.0 / -51.6 for 1 / 5 / 64 / 512 bands, the FP64
// form's 2^-52.9 / -52.7 / -51.7 / -50.3.
//
// Range (fix_lane, FixInfo): 0 <= x <= 48, Re w >= 0, 2^(E-7) <= |w| <= 1.375 2^E - max x with
// the binary scale E of the instance's frequencies; weights whose row and column maxima over
// the bands are finite and of ordinary exponent, and whose largest product over the bands is
// within 2^-7 of the product of those maxima (the product of the split weights is exact to
// 2^-60 of that). A warp with a lane outside takes the FP64 form.
#pragma once

#include "gpp_device.cuh"

namespace gpp {

constexpr int kStageBands = 64;    // bands of one warp's staged weights in shared memory
constexpr int kLowBands = 16;      // bands of the FP32 low sums between FP64 flushes
constexpr int kFlushBands = 1024;  // bands of the modular sums between flushes
constexpr float kFixKappa = 1.0f - 0x1p-12f;
constexpr float kFixNear = 0x1p-20f;  // |(|wdiff|^2 - 1/4)| below which FP64 decides
constexpr int kFixMinTop = 55;        // fewest bits of the largest weight (of at most 62)

// The gathered weight of one band, split: a comp 2^ka = a1 + a0 2^-32.
struct alignas(16) FixAm {
  int r1, i1, r0, i0;
};

// Per-thread constants of a (p, ig) pair.
struct FixPair {
  int wh, wl, ih, il;  // Re w, Im w = hi 2^-h + lo 2^-(h+32)
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

// The instance's frequencies fit the split-integer range with binary scale E.
__device__ __forceinline__ FixInfo fix_info(double xmin, double xmax) {
  FixInfo f;
  f.ok = xmin >= 0.0 && xmax <= 48.0;
  int E = 2;
  while (E < 6 && xmax > 0.75 * static_cast<double>(1 << E)) ++E;
  f.E = E;
  return f;
}

// v = hi 2^-h + lo 2^-(h+32) for |v| < 2^(31-h), to 2^-(h+33).
__device__ __forceinline__ void fix_split(double v, int h, int& hi, int& lo) {
  const double s = v * exp2i(h);
  double r = rint(s), l = rint((s - r) * 4294967296.0);
  if (l >= 2147483648.0) {
    r += 1.0;
    l -= 4294967296.0;
  }
  hi = static_cast<int>(r);
  lo = static_cast<int>(l);
}
// v = a + b with a a multiple of 2^ge (v / 2^ge below 2^24) and b its FP32-rounded remainder.
__device__ __forceinline__ void fix_fsplit(double v, int ge, float& a, float& b) {
  const double r = rint(v * exp2i(-ge)) * exp2i(ge);
  a = static_cast<float>(r);
  b = static_cast<float>(v - r);
}

// One band-table entry's split frequency.
__device__ __forceinline__ int4 fix_x(double x, int E) {
  int hi, lo;
  float a, b;
  fix_split(x, 30 - E, hi, lo);
  fix_fsplit(x, E - 23, a, b);
  return make_int4(hi, lo, __float_as_int(a), __float_as_int(b));
}

__device__ __forceinline__ FixPair fix_pair(double2 w, int E) {
  FixPair q;
  fix_split(w.x, 30 - E, q.wh, q.wl);
  fix_split(w.y, 30 - E, q.ih, q.il);
  fix_fsplit(w.x, E - 23, q.w1, q.w2);
  q.i1 = static_cast<float>(w.y);
  q.i2 = static_cast<float>(w.y - static_cast<double>(q.i1));
  fix_fsplit(w.y * w.y, 2 * E - 21, q.n1, q.n2);
  return q;
}

// Whether a lane's w lies in the split-integer range (see the top of this file).
__device__ __forceinline__ bool fix_lane(double2 w, double wabs2, int E, double xmax) {
  const double lim = 1.375 * exp2i(E) - xmax;
  return w.x >= 0.0 && wabs2 >= exp2i(2 * E - 14) && wabs2 <= lim * lim;
}

// The scales of u (or v) of one frequency: with |u| <= 1/d, ks = 31 + floor(log2 d) (U stays
// below 2^31; from d^2, whose exponent halves), s = 2^ks and c = -1/(kappa 2^(h+ks)), minus
// the unit of the residual e.
__device__ __forceinline__ int fix_ks(double d2) {
  return 31 + ((((__double2hiint(d2) >> 20) & 0x7ff) - 1023) >> 1);
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
// zero where `on` is false.
template <bool SIDE_A>
__device__ __forceinline__ FixU fix_term(const FixPair& w, const FixN& n, int xh, int xl, float2 sc,
                                         bool on) {
  FixU o;
  const long long x64 = (static_cast<long long>(xh) << 32) + xl;
  const long long w64 = (static_cast<long long>(w.wh) << 32) + w.wl;
  const long long a64 = SIDE_A ? x64 - w64 : x64 + w64;
  const int Al = static_cast<int>(a64);
  const int Ah = static_cast<int>(a64 >> 32) - (Al >> 31);   // signed low word
  float rho = fix_rcp(fmaf(n.N1, 1.0f + 0x1p-12f, n.Nm));    // kappa / |A|^2
  if (SIDE_A) rho = on ? rho : 0.0f;
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

// Largest frequency group: more accumulators than 16 x 3 would not fit the register budget.
constexpr int kFixMaxGroup = 3;

// v 2^k = n1 + n0 2^-32 (|n0| <= 2^31), for |v| 2^k < 2^30. The scaling is an addition to the
// exponent field (k >= 0; a zero or subnormal v gives a value far below the last unit), the
// rest one FP64 -> 64-bit integer conversion (as slow as an FP64 multiply-add, but the only
// FP64 instruction here).
__device__ __forceinline__ void fix_value(double v, int khi, int& n1, int& n0) {
  const double s = __hiloint2double(__double2hiint(v) + khi, __double2loint(v));
  const long long i = __double2ll_rn(s);   // v 2^(k + 32)
  n1 = static_cast<int>((i + 0x80000000LL) >> 32);
  n0 = static_cast<int>(i);
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
  const long long half = 1LL << (sh - 1);
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

// Bands [b0, b1) of the thread's pair, WG frequencies from iw0 of W, added to the thread's
// FP64 sums st[k blockDim.x] (units of kappa 2^ks M; values 4 iw + {0, 1}: sum M u, + {2, 3},
// with OCC: sum M v).
template <int WG, bool OCC>
__device__ __forceinline__ void fix_range(int b0, int b1, int64_t G, int W, int iw0,
                                           const double2* __restrict__ an_ptr, int nkhi,
                                           const double2* __restrict__ am_ptr, int akhi,
                                           const BandEntry* __restrict__ bt, const FixPair& w,
                                           const double2* __restrict__ w_ptr, int sh, double* st,
                                          const float2* sc, FixAm* stage) {
  const int nt = blockDim.x, lane = threadIdx.x & 31;
#pragma unroll 1
  for (int f0 = b0; f0 < b1; f0 += kFlushBands) {
    const int f1 = min(f0 + kFlushBands, b1);
    long long acc[4 * WG];
    float aH[4 * WG], aL[4 * WG];
#pragma unroll
    for (int k = 0; k < 4 * WG; ++k) {
      acc[k] = 0;
      aH[k] = 0.0f;
      aL[k] = 0.0f;
    }
    double2 an_next = ldg2(an_ptr + static_cast<int64_t>(f0) * G);
#pragma unroll 1
    for (int s0 = f0; s0 < f1; s0 += kStageBands) {
      const int s1 = min(s0 + kStageBands, f1);
      __syncwarp();
      for (int b = s0 + lane; b < s1; b += 32) {   // this warp's weights of the next bands
        const double2 a = ldg2(am_ptr + b);
        FixAm e;
        fix_value(a.x, akhi, e.r1, e.r0);
        fix_value(a.y, akhi, e.i1, e.i0);
        stage[b - s0] = e;
      }
      __syncwarp();
#pragma unroll 1
      for (int l0 = s0; l0 < s1; l0 += kLowBands) {
        const int l1 = min(l0 + kLowBands, s1);
#pragma unroll 1
        for (int b = l0; b < l1; ++b) {
          const double2 an = an_next;
          if (b + 1 < b1) an_next = ldg2(an_ptr + static_cast<int64_t>(b + 1) * G);
          const FixM m = fix_weight(stage[b - s0], an, nkhi, sh);
          const BandEntry* btb = bt + static_cast<int64_t>(b) * W + iw0;
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
            const double2 wv = ldg2(w_ptr);
#pragma unroll
            for (int k = 0; k < WG; ++k) {
              const double a = __ldg(&btb[k].lo.x) - wv.x;
              d[k] = gt_nonneg(fma(a, a, wv.y * wv.y), kLimitTwo) ? 1.0f : -1.0f;
            }
          }
#pragma unroll
          for (int k = 0; k < WG; ++k) {
            {
              const FixU u = fix_term<true>(w, na[k], xv[k].x, xv[k].y, sc[2 * k * nt], d[k] > 0.0f);
              acc[4 * k] = mad_wide(m.r1, u.Ur, mad_wide(m.ni1, u.Ui, acc[4 * k]));
              acc[4 * k + 1] = mad_wide(m.r1, u.Ui, mad_wide(m.i1, u.Ur, acc[4 * k + 1]));
              aH[4 * k] = fmaf(m.r1f, u.ur, fmaf(-m.i1f, u.ui, aH[4 * k]));
              aH[4 * k + 1] = fmaf(m.r1f, u.ui, fmaf(m.i1f, u.ur, aH[4 * k + 1]));
              aL[4 * k] += fmaf(m.r1f, u.gr, fmaf(-m.i1f, u.gi, fmaf(m.r0, u.ur, -m.i0 * u.ui)));
              aL[4 * k + 1] += fmaf(m.r1f, u.gi, fmaf(m.i1f, u.gr, fmaf(m.r0, u.ui, m.i0 * u.ur)));
            }
            if (OCC) {   // v = conj of the computed value
              const FixN ns = fix_norm<false>(w, __int_as_float(xv[k].z), __int_as_float(xv[k].w));
              const FixU u = fix_term<false>(w, ns, xv[k].x, xv[k].y, sc[(2 * k + 1) * nt], true);
              acc[4 * k + 2] = mad_wide(m.r1, u.Ur, mad_wide(m.i1, u.Ui, acc[4 * k + 2]));
              acc[4 * k + 3] = mad_wide(m.i1, u.Ur, mad_wide(m.nr1, u.Ui, acc[4 * k + 3]));
              aH[4 * k + 2] = fmaf(m.r1f, u.ur, fmaf(m.i1f, u.ui, aH[4 * k + 2]));
              aH[4 * k + 3] = fmaf(m.i1f, u.ur, fmaf(-m.r1f, u.ui, aH[4 * k + 3]));
              aL[4 * k + 2] += fmaf(m.r1f, u.gr, fmaf(m.i1f, u.gi, fmaf(m.r0, u.ur, m.i0 * u.ui)));
              aL[4 * k + 3] += fmaf(m.i1f, u.gr, fmaf(-m.r1f, u.gi, fmaf(m.i0, u.ur, -m.r0 * u.ui)));
            }
          }
        }
#pragma unroll
        for (int k = 0; k < 4 * WG; ++k)
          if (OCC || (k & 2) == 0) {
            st[k * nt] += static_cast<double>(aL[k]);
            aL[k] = 0.0f;
          }
      }
    }
#pragma unroll
    for (int k = 0; k < 4 * WG; ++k)
      if (OCC || (k & 2) == 0) {
        // the sum is acc + j 2^64 with j from the FP32 sum
        const float top = static_cast<float>(static_cast<int>(acc[k] >> 32)) * 0x1p-32f;
        const int j = __float2int_rn(fmaf(aH[k], 0x1p-64f, -top));
        st[k * nt] += fma(static_cast<double>(j), 18446744073709551616.0, static_cast<double>(acc[k]));
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

// All bands of the thread's pair by the split-integer form, multiplied by Iw = I w and added
// to tacc[4 W]. Returns false (nothing added) if any lane of the warp is out of range.
template <int W>
__device__ __noinline__ bool fix_band_loop(int B, int64_t G, int nocc,
                                           const double2* __restrict__ an_ptr,
                                           const double2* __restrict__ am_ptr,
                                           const BandEntry* __restrict__ bt, bool live, double2 wv,
                                           const double2* __restrict__ w_ptr, double2 I, int E,
                                           const double* __restrict__ xrange, unsigned char* smem,
                                           double* tacc) {
  constexpr int WG = W < kFixMaxGroup ? W : kFixMaxGroup;
  const int nt = blockDim.x, warp = threadIdx.x >> 5;
  double* st = reinterpret_cast<double*>(smem) + threadIdx.x;
  float2* sc = reinterpret_cast<float2*>(smem + static_cast<size_t>(nt) * 4 * WG * 8) + threadIdx.x;
  FixAm* stage = reinterpret_cast<FixAm*>(smem + static_cast<size_t>(nt) * 6 * WG * 8) +
                 warp * kStageBands;
  // the magnitudes of the column of aqsntemp, of the row of weights and of their products
  unsigned mn = 0, ma = 0, mp = 0;
  int kn, ka;
#pragma unroll 8
  for (int b = 0; b < B; ++b) {
    const unsigned hn = fix_hi_max(ldg2(an_ptr + static_cast<int64_t>(b) * G));
    const unsigned ha = fix_hi_max(ldg2(am_ptr + b));
    mn = max(mn, hn);
    ma = max(ma, ha);
    mp = max(mp, hn + ha);
  }
  const bool exp_ok = fix_exponent(mn, kn) && fix_exponent(ma, ka);
  // every |M| comp 2^(ka + kn) < 2^top: twice (complex) the largest product, 0.18 for its
  // logarithm; sh takes the largest to 31 bits
  const int top = static_cast<int>((mp + (1u << 20) + 188744u) >> 20) + 1 - 2046 + ka + kn;
  const bool m_ok = exp_ok && (mn == 0 || ma == 0 || top >= kFixMinTop);
  if (!__all_sync(0xffffffffu, m_ok || !live)) return false;
  const int sh = max(min(top - 31, 30), 1);
  const int nkhi = (kn + 32) << 20, akhi = (ka + 32) << 20;   // for fix_value
  const FixPair w = fix_pair(wv, E);
  const double Iwr = fma(I.x, wv.x, -I.y * wv.y), Iwi = fma(I.x, wv.y, I.y * wv.x);
  double add[4 * W];
  auto group = [&](auto tag, int iw0, double* out) {
    constexpr int N = decltype(tag)::value;
    int ks[2 * N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const double lo = xrange[iw0 + k], hi = xrange[kMaxNw + iw0 + k];
      const double dA = fmax(0.5, fmax(lo - wv.x, wv.x - hi));
      const double sr = lo + wv.x;
      ks[2 * k] = fix_ks(dA * dA);
      ks[2 * k + 1] = fix_ks(fma(sr, sr, wv.y * wv.y));
      sc[2 * k * nt] = fix_scale(ks[2 * k], E);
      sc[(2 * k + 1) * nt] = fix_scale(ks[2 * k + 1], E);
#pragma unroll
      for (int i = 0; i < 4; ++i) st[(4 * k + i) * nt] = 0.0;
    }
    fix_range<N, true>(0, nocc, G, W, iw0, an_ptr, nkhi, am_ptr, akhi, bt, w, w_ptr, sh,
                       st, sc, stage);
#pragma unroll
    for (int k = 0; k < N; ++k) {
      // units: M1 = M 2^(ka + kn - sh), U = u kappa 2^ks
      const double fa = exp2i(sh - ka - kn - ks[2 * k]) * (1.0 / kFixKappa);
      const double fs = exp2i(sh - ka - kn - ks[2 * k + 1]) * (1.0 / kFixKappa);
      out[4 * k + 2] = 0.5 * fma(fa, st[4 * k * nt], -fs * st[(4 * k + 2) * nt]);
      out[4 * k + 3] = 0.5 * fma(fa, st[(4 * k + 1) * nt], -fs * st[(4 * k + 3) * nt]);
    }
    if (nocc < B)
      fix_range<N, false>(nocc, B, G, W, iw0, an_ptr, nkhi, am_ptr, akhi, bt, w, w_ptr, sh,
                         st, sc, stage);
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const double fa = exp2i(sh - ka - kn - ks[2 * k]) * (1.0 / kFixKappa);
      out[4 * k] = fa * st[4 * k * nt];
      out[4 * k + 1] = fa * st[(4 * k + 1) * nt];
    }
  };
  // frequency groups of at most three; the weights are formed again for each
  constexpr int NG = (W + kFixMaxGroup - 1) / kFixMaxGroup;
  constexpr int LO = W / NG, NHI = W - LO * NG;   // NHI groups of LO + 1, then groups of LO
#pragma unroll
  for (int g = 0; g < NG; ++g) {
    const int iw0 = g * LO + (g < NHI ? g : NHI);
    if (g < NHI)
      group(IntTag<LO + 1>(), iw0, add + 4 * iw0);
    else
      group(IntTag<LO>(), iw0, add + 4 * iw0);
  }
#pragma unroll
  for (int k = 0; k < 2 * W; ++k) {   // tacc += Iw add, per complex value
    const double tr = add[2 * k], ti = add[2 * k + 1];
    tacc[2 * k] = fma(Iwr, tr, fma(-Iwi, ti, tacc[2 * k]));
    tacc[2 * k + 1] = fma(Iwr, ti, fma(Iwi, tr, tacc[2 * k + 1]));
  }
  return true;
}

}  // namespace gpp
