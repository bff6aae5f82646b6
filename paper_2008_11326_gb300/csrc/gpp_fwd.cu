// Forward GPP sum: the column gather. The main sum runs in gpp_batched.cu (a single
// instance is a batch of one) with the per-band arithmetic of gpp_terms_fix.cuh (FP64-accurate,
// on the integer and FP32 pipes), gpp_terms_f64.cuh and gpp_terms_f32.cuh.
//
// Work decomposition (paper §III v4: the band loop runs serially inside a thread while
// (igp, ig) are spread over threads, which keeps every ig-contiguous array coalesced).
// A tile is one local column p and `threads * ig_per_thread` consecutive G-vectors; each
// thread owns (p, ig) pairs of the tile, hoists everything that depends on (p, ig) only,
// and walks all bands, evaluating every frequency iw from registers (the paper's v5 split
// of iw into separate launches would recompute the shared weights). Every tile writes its own partial and the partials are
// summed in tile order, so every bit of the result is fixed.
//
// Arithmetic (paper §III v1: reciprocals instead of divides; §III v3: squared moduli).
// With A = x - w, S = x + w, C = x^2 - w^2 = A S, K = M I w, K2 = K w:
//   branch 1:  M sch = K / A        = K conj(A) / |A|^2
//              M ssx = M w^2 I / C  = K2 conj(C) / |C|^2 = (K/A - K/S) / 2
//   branch 2:  M ssx = -M I delw / (4 delw + 2) = -(K/2) / S = -(K/2) conj(S) / |S|^2
// (branch 2 uses delw = w / A, so 4 delw + 2 = 2 S / A; branch 1's partial fractions use
// S - A = 2 w). On the fast path, where branch 3 cannot occur, asxtemp is therefore
// (achtemp - sum K/S) / 2 over the occupied bands: two reciprocals per term, 1/|A|^2 and
// 1/|S|^2, and no branch on the asxtemp side. The general form (both thresholds and the
// screened-exchange cutoff) keeps one reciprocal r = 1/(|A|^2 |S|^2) for all three
// denominators, 1/|A|^2 = |S|^2 r, 1/|C|^2 = r, 1/|S|^2 = |A|^2 r, and branch selection picks
// operands (Z, Y, coefficient) for one shared complex multiply-accumulate, so a warp whose
// lanes take different branches pays once.

#include <cuda_runtime.h>

#include <algorithm>

#include "gpp_device.cuh"
#include "gpp_internal.h"
#include "gpp_terms_f64.cuh"
#include "gpp_terms_fix.cuh"

namespace gpp {

namespace {

// Band count up to which every table block of the gather reads all the frequencies.
constexpr int64_t kScanBands = 16384;

// Global column of local column p, or -1 if it contributes nothing. Counts indices that
// are outside their arrays (the sentinel indinv[k] == G is legitimate).
__device__ __forceinline__ int column_of(int64_t p, int64_t G, const int32_t* inv,
                                         const int32_t* indinv, int* bad) {
  int64_t k = inv[p];
  if (k < 0 || k > G) {
    if (bad) atomicAdd(bad, 1);
    return -1;
  }
  int64_t g = indinv[k];
  if (g < 0 || g > G) {
    if (bad) atomicAdd(bad, 1);
    return -1;
  }
  return g < G ? static_cast<int>(g) : -1;
}

// max / min over the block of one value per thread (256 threads); every thread gets the result.
// `buf`: 8 entries of shared memory per call.
template <class T, class Op>
__device__ __forceinline__ T block_fold(T v, T* buf, Op op) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) buf[threadIdx.x >> 5] = v;
  __syncthreads();
  v = buf[0];
#pragma unroll
  for (int k = 1; k < 8; ++k) v = op(v, buf[k]);
  return v;
}

// One block's share of the gather of an instance: its first `table_blocks` blocks write the
// band tables and the flags, the others gather columns (paper §III v7: aqsmtemp_local(igp,
// band) stored band-contiguous), one column per warp so that the column's index chain
// (inv_igp_index, indinv, vcoul) is read once and the bands' loads are independent. A
// single-instance call also writes the instance descriptor the main kernel reads and clears
// its tile counter (so the call needs no host-to-device copy and no memset, and can be
// captured in a graph).
__device__ __forceinline__ void prep_block(const PrepArgs& a, int block, int nblocks) {
  const int64_t B = a.B, G = a.G, P = a.P;
  const int W = a.W, lane = threadIdx.x & 31;
  if (block >= a.table_blocks) {
    const int64_t nwarps = static_cast<int64_t>(nblocks - a.table_blocks) * 8;
    for (int64_t p = static_cast<int64_t>(block - a.table_blocks) * 8 + (threadIdx.x >> 5); p < P;
         p += nwarps) {
      const int g = column_of(p, G, a.inv, a.indinv, lane == 0 && a.debug ? a.flags + 1 : nullptr);
      const double vc = g >= 0 ? a.vcoul[g] : 0.0;
      if (lane == 0) a.colg[p] = g;
#pragma unroll 4
      for (int64_t b = lane; b < B; b += 32) {
        double2 v = make_double2(0.0, 0.0);
        if (g >= 0) {
          const double2 m = a.aqsm[b * G + g];
          v = make_double2(m.x * vc, -m.y * vc);
        }
        a.am[p * B + b] = v;
        if (a.am32) a.am32[p * B + b] = make_float2(static_cast<float>(v.x), static_cast<float>(v.y));
      }
    }
    return;
  }
  // The flags, and for the FP64 sum's split-integer form the ranges of the frequencies: every
  // table block reads all of them (a few KB from L2) and the first writes the result, so that
  // neither a second launch nor atomics are needed; with more bands than kScanBands each block
  // raises the flags for its own entries instead, after a memset.
  __shared__ double s_lo[8];
  __shared__ unsigned long long s_max[8];
  if (a.desc_out && block == 0 && threadIdx.x == 0) {
    *a.desc_out = a.desc;
    *a.counter = 0;
  }
  const int64_t n = B * W;
  const int64_t i0 = static_cast<int64_t>(block) * blockDim.x + threadIdx.x;
  FixInfo fix{0, 0, 0.0, 0.0};
  auto bits = [](double x) { return static_cast<unsigned long long>(__double_as_longlong(fabs(x))); };
  if (a.scan) {
    double lo = INFINITY;         // the least frequency (NaN apart)
    unsigned long long top = 0;   // the bits of max |wx| (NaN above infinity)
#pragma unroll 4
    for (int64_t i = threadIdx.x; i < n; i += 256) {
      const double x = a.wx[i];
      lo = fmin(lo, x);
      top = max(top, bits(x));
    }
    top = block_fold(top, s_max, [](unsigned long long u, unsigned long long v) { return max(u, v); });
    lo = block_fold(lo, s_lo, [](double u, double v) { return fmin(u, v); });
    const double xmax = __longlong_as_double(static_cast<long long>(top));
    if (a.want_fix) fix = fix_info(lo, xmax);
    if (block == 0) {
      if (threadIdx.x == 0) {
        a.flags[0] = lo >= 0.0 && xmax == xmax ? 0 : 1;
        a.flags[2] = top < bits(kFp32MaxX) ? 0 : 1;
        if (!a.debug) a.flags[1] = 0;
        *reinterpret_cast<unsigned long long*>(a.flags + kFlagXmax) = top;
      }
      double* range = reinterpret_cast<double*>(a.flags + kFlagRange);
      for (int iw = threadIdx.x >> 5; fix.ok && iw < W; iw += 8) {   // a warp per frequency
        double l = INFINITY, h = -INFINITY;
#pragma unroll 4
        for (int64_t b = lane; b < B; b += 32) {
          const double x = a.wx[b * W + iw];
          l = fmin(l, x);
          h = fmax(h, x);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          l = fmin(l, __shfl_xor_sync(0xffffffffu, l, o));
          h = fmax(h, __shfl_xor_sync(0xffffffffu, h, o));
        }
        if (lane == 0) {
          range[iw] = l;
          range[kMaxNw + iw] = h;
        }
      }
    }
  }
  if (i0 == 0) *reinterpret_cast<FixInfo*>(a.flags + kFlagFix) = fix;
  for (int64_t i = i0; i < n; i += static_cast<int64_t>(a.table_blocks) * 256) {
    const double x = a.wx[i];
    a.bt[i] = BandEntry{make_double2(x, 0.0), fix.ok ? fix_x(x, fix.E) : make_int4(0, 0, 0, 0)};
    if (!a.scan) {
      if (!(x >= 0.0)) a.flags[0] = 1;
      if (!(fabs(x) < kFp32MaxX)) a.flags[2] = 1;
      // max |wx|: non-negative doubles order as their bit patterns
      atomicMax(reinterpret_cast<unsigned long long*>(a.flags + kFlagXmax), bits(x));
    }
    if (a.bt32) {  // layout of f32_band_quads (gpp_device.cuh)
      const float xf = static_cast<float>(x);
      const int64_t b0 = i / W, iw = i - b0 * W;
      const int nq = (W + 4) / 4;
      float* fb = reinterpret_cast<float*>(a.bt32 + b0 * (2 * nq));
      fb[iw] = xf;
      fb[4 * nq + iw] = static_cast<float>(x - static_cast<double>(xf));
      if (iw == 0) {  // the band's frequency range, rounded outwards, and the padding
        float lo = __int_as_float(0x7f800000), hi = -lo;
        for (int k = 0; k < W; ++k) {
          lo = fminf(lo, __double2float_rd(a.wx[b0 * W + k]));
          hi = fmaxf(hi, __double2float_ru(a.wx[b0 * W + k]));
        }
        fb[W] = lo;
        fb[4 * nq + W] = hi;
        for (int k = W + 1; k < 4 * nq; ++k) fb[k] = fb[4 * nq + k] = 0.0f;
      }
    }
  }
}

__global__ void __launch_bounds__(256) gpp_prep_kernel(const PrepArgs a) {
  prep_block(a, blockIdx.x, gridDim.x);
}
// Many instances in one launch: blockIdx.y is the instance.
__global__ void __launch_bounds__(256) gpp_prep_batch_kernel(const PrepArgs* __restrict__ list) {
  prep_block(list[blockIdx.y], blockIdx.x, gridDim.x);
}

// Complex128 -> complex64 (round to nearest) over a block of rows x columns: the FP32-bulk
// copy of aqsntemp when the caller passes none. A streaming copy (read 16 bytes, write 8 per
// element), bound by HBM.
__global__ void gpp_convert_c64_kernel(const double2* __restrict__ src, int64_t ld_src,
                                       float2* __restrict__ dst, int64_t ld_dst, int64_t rows,
                                       int64_t c0, int64_t ncols) {
  const int64_t n = rows * ncols;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += stride) {
    const int64_t r = i / ncols, c = c0 + (i - r * ncols);
    const double2 v = __ldcs(src + r * ld_src + c);
    __stcs(dst + r * ld_dst + c, make_float2(static_cast<float>(v.x), static_cast<float>(v.y)));
  }
}

}  // namespace

cudaError_t launch_convert_c64(const gpp_c128* src, int64_t ld_src, gpp_c64* dst, int64_t ld_dst,
                               int64_t rows, int64_t c0, int64_t c1, cudaStream_t s) {
  const int64_t n = rows * (c1 - c0);
  if (n <= 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  // a grid of whole waves (8 CTAs of 256 threads per SM), fewer for small copies
  int64_t blocks = std::min<int64_t>((n + 255) / 256, static_cast<int64_t>(sms) * 8);
  gpp_convert_c64_kernel<<<static_cast<int>(blocks), 256, 0, s>>>(
      reinterpret_cast<const double2*>(src), ld_src, reinterpret_cast<float2*>(dst), ld_dst,
      rows, c0, c1 - c0);
  return cudaGetLastError();
}

PrepArgs prep_args(const gpp_problem& p, const FwdPlan& plan, char* ws, bool fp32, bool debug) {
  PrepArgs a;
  a.B = p.number_bands;
  a.G = p.ncouls;
  a.P = p.ngpown;
  a.W = static_cast<int>(p.nw);
  a.aqsm = reinterpret_cast<const double2*>(p.aqsmtemp);
  a.vcoul = p.vcoul;
  a.inv = p.inv_igp_index;
  a.indinv = p.indinv;
  a.wx = p.wx_array;
  a.flags = reinterpret_cast<int*>(ws + plan.off_flags);
  a.colg = reinterpret_cast<int*>(ws + plan.off_colvalid);
  a.bt = reinterpret_cast<BandEntry*>(ws + plan.off_bt);
  a.am = reinterpret_cast<double2*>(ws + plan.off_am);
  a.bt32 = fp32 ? reinterpret_cast<float4*>(ws + plan.off_bt32) : nullptr;
  a.am32 = fp32 ? reinterpret_cast<float2*>(ws + plan.off_am32) : nullptr;
  a.scan = p.number_bands <= kScanBands;
  a.want_fix = !fp32;
  a.debug = debug;
  a.table_blocks = static_cast<int>(std::min<int64_t>((p.number_bands * p.nw + 255) / 256, 1024));
  return a;
}

namespace {
int prep_blocks(const PrepArgs& a) {
  return a.table_blocks + static_cast<int>(std::min<int64_t>((a.P + 7) / 8, 4096));
}
// The flags start at zero where the kernel only raises them.
cudaError_t prep_clear(const PrepArgs& a, cudaStream_t s) {
  return a.scan && !a.debug ? cudaSuccess : cudaMemsetAsync(a.flags, 0, kFlagBytes, s);
}
}  // namespace

cudaError_t launch_prep(const gpp_problem& p, const FwdPlan& plan, char* ws, bool fp32, bool debug,
                        const BatchInst* desc, cudaStream_t s) {
  PrepArgs a = prep_args(p, plan, ws, fp32, debug);
  cudaError_t e = prep_clear(a, s);
  if (e != cudaSuccess) return e;
  if (fp32 && plan.convert_c64) {
    e = launch_convert_c64(p.aqsntemp, p.ncouls, reinterpret_cast<gpp_c64*>(ws + plan.off_aqsn32),
                           p.ncouls, p.number_bands, 0, p.ncouls, s);
    if (e != cudaSuccess) return e;
  }
  if (desc) {
    a.desc = *desc;
    a.desc_out = reinterpret_cast<BatchInst*>(ws + plan.off_desc);
    a.counter = reinterpret_cast<unsigned long long*>(ws + plan.off_counter);
  }
  gpp_prep_kernel<<<prep_blocks(a), 256, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_prep_batch(const PrepArgs* host_list, const PrepArgs* dev_list, int n,
                              cudaStream_t s) {
  int blocks = 1;
  for (int i = 0; i < n; ++i) {
    cudaError_t e = prep_clear(host_list[i], s);
    if (e != cudaSuccess) return e;
    blocks = std::max(blocks, prep_blocks(host_list[i]));
  }
  for (int i = 0; i < n; i += 65535) {   // the grid's y limit
    const int m = std::min(n - i, 65535);
    gpp_prep_batch_kernel<<<dim3(blocks, m), 256, 0, s>>>(dev_list + i);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace gpp
