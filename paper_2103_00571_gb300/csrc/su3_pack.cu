// Layout and precision conversion between the benchmark's packed FP64 Site array and the reduced
// forms (outside the timed path). Both ways stage tiles of 128 links through shared memory, so that
// the form's side and the FP64 side are each read and written in their own memory order.
// Pack rounds each real once, to nearest even, straight from FP64 (cvt.rn.{f32,f16,bf16}.f64: no
// FP64 -> FP32 -> FP16 double rounding); unpack widens exactly and rebuilds row 2 of a two-row
// link as conj(row0 x row1) in FP64.
#include <cuda_runtime.h>

#include <algorithm>
#include <string>
#include <type_traits>

#include "su3_device.cuh"
#include "su3_internal.h"

namespace su3 {

__device__ __forceinline__ float f64_to_f32_rn(double x) {
  float r;
  asm("cvt.rn.f32.f64 %0, %1;" : "=f"(r) : "d"(x));
  return r;
}
__device__ __forceinline__ unsigned short f64_to_f16_rn(double x) {
  unsigned short r;
  asm("cvt.rn.f16.f64 %0, %1;" : "=h"(r) : "d"(x));
  return r;
}
__device__ __forceinline__ unsigned short f64_to_bf16_rn(double x) {
  unsigned short r;
  asm("cvt.rn.bf16.f64 %0, %1;" : "=h"(r) : "d"(x));
  return r;
}
// Links per tile: 18 KB of FP64 links in shared memory, so that eight CTAs of 256 threads share an SM.
constexpr int kPackTile = 128;
constexpr int kPackThreads = 256;

// The elements of a tile of links in a form's memory order, so that consecutive threads touch
// consecutive addresses: AOS link-major, SOA element-major, AOSOA32 by blocks of 32 links,
// element-major inside a block. Tiles start at multiples of 32 links.
template <int NE, int LAYOUT, int VB>  // VB: bytes of one complex element
struct Order {
  // Items of a full tile; of those, the ones whose link is >= tl (the tile's links) are skipped.
  static constexpr int kItems = kPackTile * NE;
  // Item i: the tile's link ql and element e.
  __device__ static __forceinline__ void item(int i, int& ql, int& e) {
    if (LAYOUT == SU3_LAYOUT_AOS) {
      ql = i / NE;
      e = i - ql * NE;
    } else if (LAYOUT == SU3_LAYOUT_SOA) {
      e = i / kPackTile;
      ql = i - e * kPackTile;
    } else {
      const int blk = i / (32 * NE), rem = i - blk * 32 * NE;
      e = rem >> 5;
      ql = blk * 32 + (rem & 31);
    }
  }
  // Byte offset of element e of link q0 + ql (q0 the tile's first link).
  __device__ static __forceinline__ long long off(long long q0, int ql, int e, long long stride, long long n_links) {
    if (LAYOUT == SU3_LAYOUT_AOS) return ((q0 + ql) >> 2) * stride + ((ql & 3) * NE + e) * VB;
    if (LAYOUT == SU3_LAYOUT_SOA) return ((long long)e * n_links + q0 + ql) * VB;
    return ((((q0 + ql) >> 5) * NE + e) * 32 + (ql & 31)) * (long long)VB;
  }
};

// FP64 -> a binary32 that holds x with its last bit set when any lower bit was (rounded to odd), by
// integer operations. With 24 bits it rounds on to binary16 or bfloat16 exactly as x itself would
// (24 >= 11 + 2). Valid when fits_f32(x).
__device__ __forceinline__ float to_odd_f32(double x) {
  const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
  const unsigned t = __funnelshift_l(l, (h & 0x7fffffffu) - (896u << 20), 3);
  return __uint_as_float(t | (h & 0x80000000u) | ((l & 0x1fffffffu) != 0u));
}
// FP64 -> binary32, rounded to nearest even. Valid when fits_f32(x).
__device__ __forceinline__ float to_f32(double x) {
  const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
  unsigned t = __funnelshift_l(l, (h & 0x7fffffffu) - (896u << 20), 3);
  t += ((l & 0x1fffffffu) + 0x0fffffffu + (t & 1u)) >> 29;
  return __uint_as_float(t | (h & 0x80000000u));
}
// Whether |x| is at least 2^-126 and below 2^127: a normal binary32 also after rounding.
__device__ __forceinline__ bool fits_f32(double x) {
  return (((unsigned)__double2hiint(x) >> 20) & 0x7ffu) - 897u < 253u;
}

// One complex element of the form, each real rounded once, to nearest even, straight from FP64.
// cvt from FP64 runs on the FP64 pipe at 2 per clock and SM: 36 clocks for a site's 72 reals, beside
// 32 for the 720 bytes of a 16-bit form. So values in binary32's normal range are rounded with integer
// operations, to the same bits, and store_fast returns whether both were; for others (zeros,
// subnormals, infinities, NaN) the caller has store_cvt write the element again, in a loop of its own: as a
// branch here the compiler issued the conversions under a predicate for every element.
template <int DT>
__device__ __forceinline__ bool store_fast(unsigned char* d, double2 v) {
  if constexpr (DT == kF64) {
    stg_stream(reinterpret_cast<double2*>(d), v);
    return true;
  } else {
    if constexpr (DT == kF32) stg_stream(reinterpret_cast<float2*>(d), make_float2(to_f32(v.x), to_f32(v.y)));
    else stg_stream(reinterpret_cast<uint32_t*>(d), Storage<DT>::pack(to_odd_f32(v.x), to_odd_f32(v.y)));
    return fits_f32(v.x) && fits_f32(v.y);
  }
}
template <int DT>
__device__ __forceinline__ void store_cvt(unsigned char* d, double2 v) {
  if constexpr (DT == kF32)
    stg_stream(reinterpret_cast<float2*>(d), make_float2(f64_to_f32_rn(v.x), f64_to_f32_rn(v.y)));
  else if constexpr (DT == kF16)
    stg_stream(reinterpret_cast<uint32_t*>(d),
               (uint32_t)f64_to_f16_rn(v.x) | ((uint32_t)f64_to_f16_rn(v.y) << 16));
  else if constexpr (DT == kBF16)
    stg_stream(reinterpret_cast<uint32_t*>(d),
               (uint32_t)f64_to_bf16_rn(v.x) | ((uint32_t)f64_to_bf16_rn(v.y) << 16));
}

// Exact FP32 -> FP64 widening of normal numbers and zeros by integer operations (same value, same
// bits as the hardware conversion, without the FP64 pipe); ok = false for subnormals, infinities and
// NaN (none in SU(3) data).
__device__ __forceinline__ double widen_f32(float f, bool& ok) {
  const unsigned b = __float_as_uint(f);
  const unsigned mag = b & 0x7fffffffu;
  const unsigned hi = (mag >> 3) + (896u << 20);
  ok = ok && (mag == 0u || (mag >> 23) - 1u < 254u);
  return __hiloint2double((int)((mag ? hi : 0u) | (b & 0x80000000u)), (int)(b << 29));
}

// A complex element of the form widened exactly: widen_fast by integer operations (false: the caller
// takes widen_cvt, in a loop of its own as for store_cvt).
template <int DT>
__device__ __forceinline__ bool widen_fast(typename Storage<DT>::vec v, double2& x) {
  if constexpr (DT == kF64) {
    x = v;
    return true;
  } else {
    float re, im;
    bool ok = true;
    Storage<DT>::unpack(v, re, im);  // binary16 / bfloat16 -> binary32 is exact
    x.x = widen_f32(re, ok);
    x.y = widen_f32(im, ok);
    return ok;
  }
}
template <int DT>
__device__ __forceinline__ double2 widen_cvt(typename Storage<DT>::vec v) {
  typename Storage<DT>::acc re, im;
  Storage<DT>::unpack(v, re, im);
  return make_double2((double)re, (double)im);
}

// FP64 packed AoS links -> the form. A tile of links comes in with consecutive 16-byte loads, all of a
// thread's in flight at once, into shared memory, and leaves in the form's memory order. Bound by the
// memory: type, elements per link and layout are template parameters, because the divisions by them
// and the FP64 pipe's conversions took longer than the bytes. At L=40, GB/s of bytes read and written,
// one kernel for all forms -> these: FP64 AOS 5,836 -> 7,100, FP32 AOS 4,954 -> 6,970, FP16 AOS 4,340 ->
// 6,500, FP16 SOA 2,830 -> 6,930, two-row FP16 SOA 3,944 -> 7,220.
template <int DT, int NE, int LAYOUT>
__global__ void __launch_bounds__(kPackThreads) su3_pack_kernel(const double2* __restrict__ src,
                                                                unsigned char* __restrict__ dst, long long stride,
                                                                long long n_links) {
  using O = Order<NE, LAYOUT, (int)sizeof(typename Storage<DT>::vec)>;
  __shared__ double2 tile[kPackTile * 9];
  constexpr int kLoads = (kPackTile * 9 + kPackThreads - 1) / kPackThreads;
  constexpr int kStores = (O::kItems + kPackThreads - 1) / kPackThreads;
  const int tid = threadIdx.x;
  const long long n_tiles = (n_links + kPackTile - 1) / kPackTile;
  for (long long t = blockIdx.x; t < n_tiles; t += gridDim.x) {
    const long long q0 = t * kPackTile;
    const int tl = (int)min((long long)kPackTile, n_links - q0);
    double2 in[kLoads];
#pragma unroll
    for (int k = 0; k < kLoads; ++k) {
      const int i = tid + k * kPackThreads;
      if (i < tl * 9) in[k] = ldg_stream(src + q0 * 9 + i);
    }
#pragma unroll
    for (int k = 0; k < kLoads; ++k) {
      const int i = tid + k * kPackThreads;
      if (i < tl * 9) tile[i] = in[k];
    }
    __syncthreads();
    unsigned again = 0;
#pragma unroll
    for (int k = 0; k < kStores; ++k) {
      const int i = tid + k * kPackThreads;
      int ql, e;
      O::item(i, ql, e);
      if (i < O::kItems && ql < tl &&
          !store_fast<DT>(dst + O::off(q0, ql, e, stride, n_links), tile[ql * 9 + e]))
        again |= 1u << k;
    }
#pragma unroll 1
    for (; again; again &= again - 1) {
      int ql, e;
      O::item(tid + (__ffs((int)again) - 1) * kPackThreads, ql, e);
      store_cvt<DT>(dst + O::off(q0, ql, e, stride, n_links), tile[ql * 9 + e]);
    }
    __syncthreads();
  }
}

// The form -> FP64 packed AoS links: elements come in in the form's memory order, all of a thread's in
// flight at once, and are widened exactly into shared memory; two-row links get row 2 =
// conj(row0 x row1) there, in FP64; then the FP64 links leave with consecutive 16-byte stores.
// Measured as above: FP64 AOS 5,786 -> 7,130, FP32 AOS 4,636 -> 7,080, FP16 AOS 3,759 -> 6,950, FP16 SOA
// 3,902 -> 6,890; the two-row forms are bound by the rebuild's 96 FP64 FMAs per site (FP16 2,680 -> 3,430).
template <int DT, int NE, int LAYOUT>
__global__ void __launch_bounds__(kPackThreads) su3_unpack_kernel(const unsigned char* __restrict__ src,
                                                                  double2* __restrict__ dst, long long stride,
                                                                  long long n_links) {
  using V = typename Storage<DT>::vec;
  using O = Order<NE, LAYOUT, (int)sizeof(V)>;
  __shared__ double2 tile[kPackTile * 9];
  constexpr int kLoads = (O::kItems + kPackThreads - 1) / kPackThreads;
  constexpr int kStores = (kPackTile * 9 + kPackThreads - 1) / kPackThreads;
  const int tid = threadIdx.x;
  const long long n_tiles = (n_links + kPackTile - 1) / kPackTile;
  for (long long t = blockIdx.x; t < n_tiles; t += gridDim.x) {
    const long long q0 = t * kPackTile;
    const int tl = (int)min((long long)kPackTile, n_links - q0);
    V in[kLoads];
    unsigned again = 0;
#pragma unroll
    for (int k = 0; k < kLoads; ++k) {
      const int i = tid + k * kPackThreads;
      int ql, e;
      O::item(i, ql, e);
      if (i < O::kItems && ql < tl) in[k] = ldg_stream(reinterpret_cast<const V*>(src + O::off(q0, ql, e, stride, n_links)));
    }
#pragma unroll
    for (int k = 0; k < kLoads; ++k) {
      const int i = tid + k * kPackThreads;
      int ql, e;
      O::item(i, ql, e);
      if (i < O::kItems && ql < tl && !widen_fast<DT>(in[k], tile[ql * 9 + e])) again |= 1u << k;
    }
#pragma unroll 1
    for (; again; again &= again - 1) {
      int ql, e;
      O::item(tid + (__ffs((int)again) - 1) * kPackThreads, ql, e);
      tile[ql * 9 + e] = widen_cvt<DT>(*reinterpret_cast<const V*>(src + O::off(q0, ql, e, stride, n_links)));
    }
    __syncthreads();
    if (NE == 6) {
      if (tid < tl) {
        double r0re[3], r0im[3], r1re[3], r1im[3], ore[3], oim[3];
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          r0re[m] = tile[tid * 9 + m].x;
          r0im[m] = tile[tid * 9 + m].y;
          r1re[m] = tile[tid * 9 + 3 + m].x;
          r1im[m] = tile[tid * 9 + 3 + m].y;
        }
        rebuild_row2_elems(r0re, r0im, r1re, r1im, ore, oim);
#pragma unroll
        for (int m = 0; m < 3; ++m) tile[tid * 9 + 6 + m] = make_double2(ore[m], oim[m]);
      }
      __syncthreads();
    }
#pragma unroll
    for (int k = 0; k < kStores; ++k) {
      const int i = tid + k * kPackThreads;
      if (i < tl * 9) stg_stream(dst + q0 * 9 + i, tile[i]);
    }
    __syncthreads();
  }
}

// Launches K<DT, NE, LAYOUT> for the form.
template <class Launch>
static su3_status for_form(const Form& f, const LaunchCtx& ctx, const char* what, Launch&& launch) {
  const long long n_links = 4 * f.n_sites;
  const int grid = (int)std::min<long long>((n_links + kPackTile - 1) / kPackTile, 0x7fffffffLL);
  auto by_layout = [&](auto dt, auto ne) {
    switch (f.layout) {
      case SU3_LAYOUT_AOS: launch(dt, ne, std::integral_constant<int, SU3_LAYOUT_AOS>(), grid, n_links); break;
      case SU3_LAYOUT_AOSOA32: launch(dt, ne, std::integral_constant<int, SU3_LAYOUT_AOSOA32>(), grid, n_links); break;
      default: launch(dt, ne, std::integral_constant<int, SU3_LAYOUT_SOA>(), grid, n_links); break;
    }
  };
  auto by_repr = [&](auto dt) {
    if (f.repr_in == SU3_REPR_FULL18) by_layout(dt, std::integral_constant<int, 9>());
    else by_layout(dt, std::integral_constant<int, 6>());
  };
  switch (f.dtype) {
    case SU3_F64: by_repr(std::integral_constant<int, kF64>()); break;
    case SU3_F32: by_repr(std::integral_constant<int, kF32>()); break;
    case SU3_F16: by_repr(std::integral_constant<int, kF16>()); break;
    default: by_repr(std::integral_constant<int, kBF16>()); break;
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    *ctx.err = std::string(what) + ": " + cudaGetErrorString(e);
    return SU3_ERR_CUDA;
  }
  ++*ctx.launches;
  return SU3_OK;
}

su3_status launch_pack(const Form& dst, const double* src, void* dst_dev, const LaunchCtx& ctx) {
  return for_form(dst, ctx, "su3_pack_kernel launch", [&](auto dt, auto ne, auto layout, int grid, long long n_links) {
    su3_pack_kernel<decltype(dt)::value, decltype(ne)::value, decltype(layout)::value>
        <<<grid, kPackThreads, 0, ctx.stream>>>(reinterpret_cast<const double2*>(src),
                                                static_cast<unsigned char*>(dst_dev), dst.a_stride, n_links);
  });
}

su3_status launch_unpack(const Form& src, const void* src_dev, double* dst, const LaunchCtx& ctx) {
  return for_form(src, ctx, "su3_unpack_kernel launch", [&](auto dt, auto ne, auto layout, int grid, long long n_links) {
    su3_unpack_kernel<decltype(dt)::value, decltype(ne)::value, decltype(layout)::value>
        <<<grid, kPackThreads, 0, ctx.stream>>>(static_cast<const unsigned char*>(src_dev),
                                                reinterpret_cast<double2*>(dst), src.a_stride, n_links);
  });
}

}  // namespace su3
