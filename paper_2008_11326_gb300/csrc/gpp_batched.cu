// The main GPP sum: one persistent launch over the tiles of one or many instances (a
// single gpp_sigma call is a batch of one).
//
// Work unit: a tile = one local column p of one instance x (threads * ig_per_thread)
// G-vectors, all bands. Tiles of all instances form one list, ordered by instance band count
// (largest first, so the longest tiles start first and the tail is short); within an
// instance the G-vector tile varies slowest, so the tiles running at the same time share
// the same slab of aqsntemp (all bands x the tile's G-vectors) through L2. CTAs of a
// persistent grid take tiles from an atomic counter; the counter only schedules, and every
// tile writes its own partial slot, so the result does not depend on which CTA ran which
// tile. A per-instance kernel then sums the instance's tile partials in tile order. The
// per-pair arithmetic is in gpp_terms_fix.cuh, gpp_terms_f64.cuh and gpp_terms_f32.cuh.

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "gpp_device.cuh"
#include "gpp_internal.h"
#include "gpp_terms_f32.cuh"
#include "gpp_terms_f64.cuh"
#include "gpp_terms_fix.cuh"

namespace gpp {

namespace {

// Band count from which the FP32-bulk kernel sorts a tile's G-vectors by Re w.
constexpr int kSortBands = 128;

// Smallest power of two >= n (n >= 1).
__host__ __device__ inline int pow2_ceil(int n) {
  int k = 1;
  while (k < n) k <<= 1;
  return k;
}

// Sorts every aligned segment key[s seg, (s + 1) seg) of key[0, n) and permutes idx with
// it (n and seg powers of two, seg <= n; every thread of the block takes part): even
// segments ascending, odd ones descending (seg = n: all of it ascending). The first stages
// of a bitonic network: deterministic for fixed keys, and a permutation of idx within each
// segment whatever the keys (NaN compares false and never swaps).
__device__ inline void bitonic_sort(float* key, int* idx, int n, int seg) {
  for (int k = 2; k <= seg; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int l = i ^ j;
        if (l > i) {
          const float a = key[i], b = key[l];
          if ((i & k) == 0 ? a > b : a < b) {
            key[i] = b;
            key[l] = a;
            const int t = idx[i];
            idx[i] = idx[l];
            idx[l] = t;
          }
        }
      }
      __syncthreads();
    }
  }
}

// The FP32-bulk kernel's general path for one (igp, ig) pair: the FP64 band loop, folded
// into the thread's tile pairs. Not inlined: its FP64 accumulators would otherwise count
// against the register budget of the FP32 band loop, which it shares a kernel with (and
// the warps that take it are rare).
template <int W>
__device__ __noinline__ void f32_general_pair(int B, int64_t G, int nocc,
                                              const double2* __restrict__ aqsn,
                                              const double2* __restrict__ am,
                                              const BandEntry* __restrict__ bt, bool live,
                                              double wr, double wi, double Iwr, double Iwi,
                                              double sx2, float4* tp) {
  double a[4 * W];
#pragma unroll
  for (int k = 0; k < 4 * W; ++k) a[k] = 0.0;
  band_loop<W, false>(B, G, nocc, aqsn, am, bt, live, wr, wi, Iwr, Iwi, sx2, a);
#pragma unroll
  for (int qd = 0; qd < W; ++qd) {
    float4 th = tp[qd], tl = tp[W + qd];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const double v = a[4 * qd + i];
      const float h = static_cast<float>(v);
      pair_add(quad_elem(th, i), quad_elem(tl, i), h, static_cast<float>(v - static_cast<double>(h)));
    }
    tp[qd] = th;
    tp[W + qd] = tl;
  }
}

// One (igp, ig) pair of the FP64 sum in FP64 arithmetic, by the fast or the general form, for
// the warps outside the split-integer form's range. Not inlined, so that its registers do
// not count against the split-integer band loop.
template <int W, bool FAST>
__device__ __noinline__ void f64_pair(int B, int64_t G, int nocc, const double2* __restrict__ aqsn,
                                      const double2* __restrict__ am,
                                      const BandEntry* __restrict__ bt, bool live, double2 w,
                                      double2 I, double sx2, double* tacc) {
  double a[4 * W];
#pragma unroll
  for (int k = 0; k < 4 * W; ++k) a[k] = tacc[k];
  band_loop<W, FAST>(B, G, nocc, aqsn, am, bt, live, w.x, w.y, fma(I.x, w.x, -I.y * w.y),
                     fma(I.x, w.y, I.y * w.x), sx2, a);
#pragma unroll
  for (int k = 0; k < 4 * W; ++k) tacc[k] = a[k];
}

// The FP64 sum's tiles: every warp of a pass takes the split-integer form where its inputs
// allow (gpp_terms_fix.cuh), else the FP64 fast or general form. smem: fix_smem_bytes.
template <int W>
__device__ __forceinline__ void f64_body(const BatchInst* __restrict__ inst, int ninst,
                                         int64_t t_begin, int64_t ntiles, int igpt,
                                         unsigned long long* counter,
                                         double* __restrict__ partials) {
  __shared__ double red[(256 / 32) * 4 * kMaxNw];
  __shared__ long long s_t;
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  double acc[4 * W];   // the thread's tile sums, in local memory (touched once per pair)
  for (;;) {
    if (threadIdx.x == 0) s_t = t_begin + static_cast<long long>(atomicAdd(counter, 1ULL));
    __syncthreads();
    const int64_t t = s_t;
    __syncthreads();
    if (t >= ntiles) break;
    int ilo = 0, ihi = ninst - 1;  // instance holding tile t (tile ranges are sorted)
    while (ilo < ihi) {
      const int mid = (ilo + ihi) >> 1;
      if (__ldg(&inst[mid].tile_end) > t)
        ihi = mid;
      else
        ilo = mid + 1;
    }
    const BatchInst& d = inst[ilo];
    const int B = d.B, nocc = d.nocc;
    const int64_t G = d.G;
    const int64_t local = t - d.tile0;
    const int64_t igt = local / d.P;
    const int64_t p = local - igt * d.P;
    const bool col_ok = d.colg[p] >= 0;
    const bool x_fast = d.flags[0] == 0;
    const FixInfo fix = *reinterpret_cast<const FixInfo*>(d.flags + kFlagFix);
    const bool fix_on = fix.ok == 1 || (fix.ok == 2 && d.sx2 > 0.0);
    const double* xrange = reinterpret_cast<const double*>(d.flags + kFlagRange);
    const double2* am = d.am + p * B;
#pragma unroll
    for (int k = 0; k < 4 * W; ++k) acc[k] = 0.0;
    for (int j = 0; j < igpt; ++j) {
      const int64_t ig = (igt * igpt + j) * blockDim.x + threadIdx.x;
      const bool live = ig < G && col_ok;
      if (!__any_sync(0xffffffffu, live)) continue;   // a dead column, or past G
      double2 w = make_double2(1.0, 0.5);  // inert lane: in every range, finite terms, zero weight
      double2 I = make_double2(0.0, 0.0);
      if (live) {
        w = ldg2(d.wt + p * G + ig);
        I = ldg2(d.eps + p * G + ig);
      }
      const double2* an = d.aqsn + (live ? ig : 0);
      const double wabs2 = fma(w.x, w.x, w.y * w.y);
      if (fix_on && __all_sync(0xffffffffu, fix_lane(w, wabs2, fix) || !live)) {
        const double2* w64 = live ? d.wt + p * G + ig : d.wt;
        // with several groups of frequencies the sums before them, to be put back; else a doubted
        // pair's own (local memory, as acc)
        double other[4 * W];
        if (W > kFixMaxGroup) {
#pragma unroll
          for (int k = 0; k < 4 * W; ++k) other[k] = acc[k];
        }
        const bool cut = fix.ok == 2;
        const FixResult r =
            cut ? fix_band_loop<W, true>(B, G, nocc, an, am, d.bt, live, w, w64, I, fix.E, d.sx2,
                                         xrange, dyn_smem, acc, other)
                : fix_band_loop<W, false>(B, G, nocc, an, am, d.bt, live, w, w64, I, fix.E, 0.0,
                                          xrange, dyn_smem, acc, other);
        if (r == kFixDone) continue;
        if (r == kFixDoubt) {   // rare
          const bool ok =
              cut ? fix_strong<W, true>(B, G, nocc, an, am, d.bt, live, w, I, fix.E, d.sx2, xrange)
                  : fix_strong<W, false>(B, G, nocc, an, am, d.bt, live, w, I, fix.E, 0.0, xrange);
          const bool add = ok && W <= kFixMaxGroup, back = !ok && W > kFixMaxGroup;
#pragma unroll
          for (int k = 0; k < 4 * W; ++k) acc[k] = add ? acc[k] + other[k] : back ? other[k] : acc[k];
          if (ok) continue;
        }
      }
      // the FP64 fast form's conditions, with the partial fractions' bound on x / |w|
      const bool fast_lane = w.x >= 0.0 && gt_nonneg(wabs2, kFastWabs2Lo) &&
                             lt_nonneg(wabs2, kFastWabs2Hi) &&
                             !lt_nonneg(wabs2, pf_wabs2_min(d.flags));
      if (__all_sync(0xffffffffu, fast_lane || !live) && x_fast)
        f64_pair<W, true>(B, G, nocc, an, am, d.bt, live, w, I, 0.0, acc);
      else
        f64_pair<W, false>(B, G, nocc, an, am, d.bt, live, w, I, d.sx2, acc);
    }
    block_partials<4 * W>(acc, red, partials + t * 4 * W);
  }
}

// Tile partials: FP64 sums (double) for GPP_FP64; compensated FP32 pairs (float2, hi + lo)
// for GPP_FP32_BULK, so that its main kernel needs no FP64 arithmetic outside the rare
// exact-decision and near-pole branches and the once-per-pair I w. Both are 8 bytes per
// value. The FP32-bulk instantiation is held to 72 registers per thread: with its shared
// memory (the compensated pairs) that is 7 CTAs of 128 threads per SM either way, and on
// GB300 (nw = 3, benchmark instance) its main kernel ran 111.2 ms at 64 registers (spilled
// values reloaded in the band loop), 104.5 ms at 72 and 105.9 ms at 80.
#ifndef GPP_F32_MAXNREG
#define GPP_F32_MAXNREG 72
#endif

template <int W>
__device__ __forceinline__ void f32_body(const BatchInst* __restrict__ inst, int ninst,
                                             int64_t t_begin, int64_t ntiles, int igpt,
                                             unsigned long long* counter,
                                             double* __restrict__ partials) {
  __shared__ double red[(256 / 32) * 4 * kMaxNw];
  __shared__ long long s_t;
  __shared__ const BandEntry* s_bt64;  // FP32-bulk: the FP64 band table, for the exact path
  // FP32-bulk: the threads' slots (F32Slots: band compensated pairs, FP64 wtilde; (8 W + 4)
  // floats per thread), then the tile's G-vector positions in sorted order
  // (int[pow2_ceil(blockDim.x * igpt)]); the sort keys (float, as many) alias the start of
  // the slots, which are written only after the sort, and the slot area is at least as long
  // as the keys (dynamic shared memory of batched_smem_bytes)
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  float* const s_slots = reinterpret_cast<float*>(dyn_smem);
  const int tile_n = blockDim.x * igpt;
  const int sort_n = pow2_ceil(tile_n);
  float* const s_key = s_slots;
  int* const s_pos = reinterpret_cast<int*>(
      s_slots + max(F32Slots<W>::kFloats * static_cast<int>(blockDim.x), sort_n));
  // FP32-bulk: the thread's tile sums as compensated pairs (hi quads [0, W), lo quads
  // [W, 2W)), in local memory (the address goes to the non-inlined fold and general-path
  // functions); touched once per (igp, ig) pair
  float4 tpair[2 * W];
  for (;;) {
    if (threadIdx.x == 0) s_t = t_begin + static_cast<long long>(atomicAdd(counter, 1ULL));
    __syncthreads();
    const int64_t t = s_t;
    __syncthreads();
    if (t >= ntiles) break;
    int ilo = 0, ihi = ninst - 1;  // instance holding tile t (tile ranges are sorted)
    while (ilo < ihi) {
      const int mid = (ilo + ihi) >> 1;
      if (__ldg(&inst[mid].tile_end) > t)
        ihi = mid;
      else
        ilo = mid + 1;
    }
    const BatchInst& d = inst[ilo];
    const int B = d.B, nocc = d.nocc;
    const int64_t G = d.G;
    const int64_t local = t - d.tile0;
    const int64_t igt = local / d.P;
    const int64_t p = local - igt * d.P;
    const bool col_ok = d.colg[p] >= 0;
    const bool x_fast = d.flags[0] == 0 && d.flags[2] == 0;
    {
      if (threadIdx.x == 0) s_bt64 = d.bt;
      // With at least kSortBands bands, the G-vectors of each pass over the tile (blockDim.x
      // of them, when that is a power of two; else the whole tile) are taken in order of
      // Re w, so that the 32 of a warp (consecutive in that order) span a narrow range of
      // Re w and most frequencies fall outside it (the far-from-threshold path). Sorting
      // within a pass keeps a warp's aqsntemp loads inside the pass's contiguous slice
      // (blockDim.x x 8 bytes per band). With fewer bands the sort and the scattered loads
      // cost more than they save. The sum does not depend on which thread takes which
      // G-vector; inert positions (past G, dead column) carry +inf keys.
      const bool sort = B >= kSortBands;
      for (int q = threadIdx.x; q < sort_n; q += blockDim.x) {
        const int64_t ig = igt * tile_n + q;
        float key = __int_as_float(0x7f800000);
        if (sort && q < tile_n && ig < G && col_ok) {
          key = static_cast<float>(__ldg(&d.wt[p * G + ig].x));
          key = key == key ? key : 0.0f;  // a NaN must still sort among the live positions
        }
        s_key[q] = key;
        s_pos[q] = q;
      }
      __syncthreads();
      if (sort) {
        const int nt = blockDim.x;
        bitonic_sort(s_key, s_pos, sort_n, (nt & (nt - 1)) == 0 ? nt : sort_n);
      }
      __syncthreads();  // the keys' space becomes the threads' slots
#pragma unroll
      for (int k = 0; k < 2 * W; ++k) tpair[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    for (int j = 0; j < igpt; ++j) {
      // a padding position (>= tile_n, key +inf like an inert one) can sort into the
      // first tile_n slots when the whole tile is sorted; it is inert
      const int q = s_pos[j * blockDim.x + threadIdx.x];
      const int64_t ig = igt * tile_n + q;
      const bool live = q < tile_n && ig < G && col_ok;
      double2 w = make_double2(0.5, 1.0);  // inert lane: finite terms, zero weight
      if (live) w = ldg2(d.wt + p * G + ig);
      const double wabs2 = fma(w.x, w.x, w.y * w.y);
      const bool fast_lane = w.x >= 0.0 && gt_nonneg(wabs2, kFastWabs2Lo) &&
                             lt_nonneg(wabs2, kFastWabs2Hi);
      const bool fast = __all_sync(0xffffffffu, fast_lane) && x_fast;
      if (fast) {
        band_loop_f32<W>(B, G, nocc, d.aqsn32 + (live ? ig : 0), d.am32 + p * B, d.bt32,
                         &s_bt64, w, live, s_slots);
        // I w in FP64 once per pair (w re-read from the thread's slot, I from memory, so
        // that neither stays in registers through the band loop)
        const volatile double* ws = reinterpret_cast<volatile double*>(F32Slots<W>::w64(s_slots));
        const double2 wv = make_double2(ws[0], ws[1]);
        double2 I = make_double2(0.0, 0.0);
        if (live) I = ldg2(d.eps + p * G + ig);
        fold_band_sums<W>(s_slots, tpair, make_double2(fma(I.x, wv.x, -I.y * wv.y),
                                                       fma(I.x, wv.y, I.y * wv.x)));
        continue;
      }
      double2 I = make_double2(0.0, 0.0);
      if (live) I = ldg2(d.eps + p * G + ig);
      const double Iwr = fma(I.x, w.x, -I.y * w.y);
      const double Iwi = fma(I.x, w.y, I.y * w.x);
      // the general path in FP64, folded into the tile pairs
      f32_general_pair<W>(B, G, nocc, d.aqsn + (live ? ig : 0), d.am + p * B, d.bt, live, w.x, w.y,
                          Iwr, Iwi, d.sx2, tpair);
    }
    float hi[4 * W], lo[4 * W];
#pragma unroll
    for (int qd = 0; qd < W; ++qd) {
      float4 th = tpair[qd], tl = tpair[W + qd];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        hi[4 * qd + i] = quad_elem(th, i);
        lo[4 * qd + i] = quad_elem(tl, i);
      }
    }
    block_pairs<4 * W>(hi, lo, reinterpret_cast<float2*>(red),
                       reinterpret_cast<float2*>(partials) + t * 4 * W);
  }
}

// The two instantiations of the main kernel. FP64: two 256-thread CTAs' worth of registers per
// SM (128 per thread), which the split-integer band loop all but fits (a few values that it
// reads once per band are spilled); the FP64 band loop runs as fast at 128 registers as at its
// unconstrained 166. FP32-bulk: held to
// GPP_F32_MAXNREG registers (80 for nw > 5, whose band loop would spill at fewer).
//
// Measured (GB300, main sum with the split-integer form against the FP64 form alone):
// B = 512, P = 819, G = 16384, nw = 3: 166.0 against 692.6 ms; B = 128, P = 410, G = 8192:
// 10.7 against 44.4 ms; B = 32, P = 64, G = 512: 0.055 against 0.30 ms (with shallower tiles
// and the cheaper reduction). Of these, what keeps every output at its own scale (gpp_terms_fix.cuh:
// the scales of two classes of bands, the test of the sums) is 162.3 -> 166.0, 10.52 -> 10.69 ms. Bound
// now: the instruction issue of the integer and FP32 pipes.
template <int W>
__global__ void __launch_bounds__(256, 2)
    gpp_batched_kernel_f64(const BatchInst* __restrict__ inst, int ninst, int64_t t_begin,
                           int64_t ntiles, int igpt, unsigned long long* counter,
                           double* __restrict__ partials) {
  f64_body<W>(inst, ninst, t_begin, ntiles, igpt, counter, partials);
}

template <int W>
__global__ void __launch_bounds__(256) __maxnreg__(W <= 5 ? GPP_F32_MAXNREG : 80)
    gpp_batched_kernel_f32(const BatchInst* __restrict__ inst, int ninst, int64_t t_begin,
                           int64_t ntiles, int igpt, unsigned long long* counter,
                           double* __restrict__ partials) {
  f32_body<W>(inst, ninst, t_begin, ntiles, igpt, counter, partials);
}

// A cluster of kReduceCtas CTAs per instance sums the instance's tile partials in a fixed
// order: CTA r takes the r-th share of the tiles; its thread t takes value t % nv of every
// (T / nv)-th tile of the share from tile t / nv on (so that the CTA reads the partials in
// order); warp k then sums value k's threads and hands the sum to the first CTA's shared
// memory, which adds the CTAs' in order. Bound by the latency of the loads (12 values, ncu):
// 64 tiles 4.9 us, 13120 tiles 18 us; one CTA of 256 threads taking a value at a time was 20 and
// 57 us (6560 tiles) between events.
constexpr int kReduceThreads = 512, kReduceCtas = 8;
template <bool F32>
__global__ void __launch_bounds__(kReduceThreads) __cluster_dims__(kReduceCtas, 1, 1)
    gpp_batched_reduce_kernel(const BatchInst* __restrict__ inst, int nv,
                              const double* __restrict__ part) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  __shared__ double s[kReduceThreads];
  __shared__ double total[kReduceCtas][4 * kMaxNw];
  const int rank = static_cast<int>(cluster.block_rank());
  const BatchInst& d = inst[blockIdx.x / kReduceCtas];
  const int per = kReduceThreads / nv, j0 = threadIdx.x / nv, k = threadIdx.x - j0 * nv;
  if (j0 < per) {
    const int64_t n = d.tile_end - d.tile0;
    const int64_t share = (n + kReduceCtas - 1) / kReduceCtas;
    const int64_t first = rank * share, last = min(first + share, n);
    double v = 0.0;
#pragma unroll 8
    for (int64_t j = first + j0; j < last; j += per) {
      const int64_t at = (d.tile0 + j) * nv + k;
      if (F32) {
        const float2 q = reinterpret_cast<const float2*>(part)[at];
        v += static_cast<double>(q.x) + static_cast<double>(q.y);
      } else {
        v += part[at];
      }
    }
    s[threadIdx.x] = v;
  }
  cluster.sync();   // s is complete; every CTA of the cluster runs (its shared memory exists)
  const int lane = threadIdx.x & 31;
  double* const dst = cluster.map_shared_rank(&total[rank][0], 0);
  for (int q = threadIdx.x >> 5; q < nv; q += kReduceThreads / 32) {
    double v = 0.0;
    for (int j = lane; j < per; j += 32) v += s[j * nv + q];
    v = warp_sum(v);
    if (lane == 0) dst[q] = v;
  }
  cluster.sync();   // after it no CTA reads another's shared memory
  if (rank == 0 && threadIdx.x < nv) {
    double v = 0.0;
    for (int r = 0; r < kReduceCtas; ++r) v += total[r][threadIdx.x];
    const int iw = threadIdx.x / 4, c = threadIdx.x % 4;
    if (c < 2)
      reinterpret_cast<double*>(d.ach)[2 * iw + c] = v * d.ach_scale;
    else
      reinterpret_cast<double*>(d.asx)[2 * iw + c - 2] = v;
  }
}

template <int W, bool F32>
const void* batched_fn() {
  return F32 ? reinterpret_cast<const void*>(&gpp_batched_kernel_f32<W>)
             : reinterpret_cast<const void*>(&gpp_batched_kernel_f64<W>);
}

const void* batched_kernel_ptr(int nw, bool f32) {
  switch (nw) {
    case 1: return f32 ? batched_fn<1, true>() : batched_fn<1, false>();
    case 2: return f32 ? batched_fn<2, true>() : batched_fn<2, false>();
    case 3: return f32 ? batched_fn<3, true>() : batched_fn<3, false>();
    case 4: return f32 ? batched_fn<4, true>() : batched_fn<4, false>();
    case 5: return f32 ? batched_fn<5, true>() : batched_fn<5, false>();
    case 6: return f32 ? batched_fn<6, true>() : batched_fn<6, false>();
    case 7: return f32 ? batched_fn<7, true>() : batched_fn<7, false>();
    case 8: return f32 ? batched_fn<8, true>() : batched_fn<8, false>();
    default: return nullptr;
  }
}

}  // namespace

size_t batched_smem_bytes(int threads, int nw, bool f32, int igpt) {
  // F32Slots<nw>::kFloats floats per thread (at least as many as the sort keys, which alias
  // them), then the sorted positions
  if (!f32) return fix_smem_bytes(threads, nw < kFixMaxGroup ? nw : kFixMaxGroup);
  const size_t sort_n = static_cast<size_t>(pow2_ceil(threads * igpt));
  const size_t slots = static_cast<size_t>(threads) * (8 * nw + 4);
  return (slots > sort_n ? slots : sort_n) * sizeof(float) + sort_n * sizeof(int);
}

// A CTA whose static + dynamic shared memory exceeds 48 KB (nw >= 6 at 256 threads) must
// opt in; the kernel's static part (the reduction buffer) is below 4 KB. Called at plan
// time, outside any stream capture.
cudaError_t batched_prepare(int threads, int nw, bool f32, int igpt) {
  const void* fn = batched_kernel_ptr(nw, f32);
  if (!fn) return cudaErrorInvalidValue;
  const size_t smem = batched_smem_bytes(threads, nw, f32, igpt);
  if (smem + 4096 <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(smem));
}

int batched_blocks_per_sm(int threads, int nw, bool f32, int igpt) {
  const void* fn = batched_kernel_ptr(nw, f32);
  if (!fn) return 0;
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, threads,
                                                    batched_smem_bytes(threads, nw, f32, igpt)) !=
      cudaSuccess)
    return 0;
  return n;
}

cudaError_t launch_batched_main(const BatchInst* inst, int ninst, int64_t ntiles, int nw,
                                bool f32, int grid, int threads, int igpt,
                                unsigned long long* counter, bool cleared, double* partials,
                                cudaStream_t s, int64_t t_begin) {
  if (!cleared) {
    cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
  }
  const size_t smem = batched_smem_bytes(threads, nw, f32, igpt);
#define GPP_BATCHED_LAUNCH(WV)                                                                    \
  if (f32)                                                                                        \
    gpp_batched_kernel_f32<WV><<<grid, threads, smem, s>>>(inst, ninst, t_begin, ntiles, igpt,    \
                                                           counter, partials);                    \
  else                                                                                            \
    gpp_batched_kernel_f64<WV><<<grid, threads, smem, s>>>(inst, ninst, t_begin, ntiles, igpt,       \
                                                        counter, partials)
  switch (nw) {
    case 1: GPP_BATCHED_LAUNCH(1); break;
    case 2: GPP_BATCHED_LAUNCH(2); break;
    case 3: GPP_BATCHED_LAUNCH(3); break;
    case 4: GPP_BATCHED_LAUNCH(4); break;
    case 5: GPP_BATCHED_LAUNCH(5); break;
    case 6: GPP_BATCHED_LAUNCH(6); break;
    case 7: GPP_BATCHED_LAUNCH(7); break;
    case 8: GPP_BATCHED_LAUNCH(8); break;
    default: return cudaErrorInvalidValue;
  }
#undef GPP_BATCHED_LAUNCH
  return cudaGetLastError();
}

cudaError_t launch_batched_reduce(const BatchInst* inst, int ninst, int nw, bool f32,
                                  const double* partials, cudaStream_t s) {
  if (f32)
    gpp_batched_reduce_kernel<true><<<ninst * kReduceCtas, kReduceThreads, 0, s>>>(inst, 4 * nw, partials);
  else
    gpp_batched_reduce_kernel<false><<<ninst * kReduceCtas, kReduceThreads, 0, s>>>(inst, 4 * nw, partials);
  return cudaGetLastError();
}

}  // namespace gpp
