// The streaming kernels for packed site strides (every layout), the failure-path self test and
// the default launch configurations; the kernels themselves are in su3_stream.cuh.
#include "su3_stream.cuh"

namespace su3 {

// ---- failure-path self test ------------------------------------------------------------------

// One CTA waits on an mbarrier that expects two arrivals but gets one, with a short limit; the
// bounded wait gives up, the kernel records the timeout and returns.
__global__ void su3_selftest_wait_kernel(unsigned* status, unsigned long long limit_ns) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 2);
    fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&bar)) : "memory");
  const bool ok = mbar_wait_bounded(&bar, 0u, limit_ns);
  if (__syncthreads_or(!ok) && threadIdx.x == 0) atomicOr(status, kDevErrTimeout);
}

su3_status launch_selftest_wait(int limit_ms, const LaunchCtx& ctx) {
  su3_selftest_wait_kernel<<<1, 32, 0, ctx.stream>>>(ctx.status, (unsigned long long)limit_ms * 1000000ull);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    *ctx.err = std::string("su3_selftest_wait_kernel launch: ") + cudaGetErrorString(e);
    return SU3_ERR_CUDA;
  }
  ++*ctx.launches;
  return SU3_OK;
}

// ---- host launchers -----------------------------------------------------------------------------

// The shape that suits every form of a layout somewhat, whatever its size. AOS: ~18 KB per tile for FP64
// full sites, 9-18 KB for the narrower ones, in 8 warps per SM, which divides small and middling arrays
// more evenly than larger tiles do; AOSOA32 and SOA: direct loads, 1/2/4 links of 16/8/4-byte elements.
LaunchCfg general_cfg(const Form& f) {
  const bool aos = f.layout == SU3_LAYOUT_AOS;
  const int tile = (int)std::max<int64_t>(32, std::min<int64_t>(128, 18432 / std::max<int64_t>(f.a_stride, 1)));
  LaunchCfg c{128, tile, 4, 2, 0, 1};
  if (!aos) c = LaunchCfg{256, f.dtype == SU3_F64 ? 1 : f.dtype == SU3_F32 ? 2 : 4, 0, 4, 0, 1};
  if (f.arith == SU3_ARITH_HYBRID) {
    c.native_permille = 125;
    c.block = 256;  // 8 warps, one of them native
    if (aos) {
      c.tile_sites = 64;  // 256 links: one per thread and tile
      c.stages = 3;       // two such CTAs fit in one SM's shared memory
    }
  }
  return c;
}

// The shapes that measured best (block, sites per tile, stages, CTAs per SM, threads per link); GB/s at
// 48^4 sites, in brackets those of general_cfg.
static LaunchCfg measured_cfg(const Form& f) {
  const bool two_in = f.repr_in == SU3_REPR_TWOROW12, two_out = f.repr_out == SU3_REPR_TWOROW12;
  const bool narrow = f.dtype == SU3_F16 || f.dtype == SU3_BF16;
  const long long n = f.n_sites > 0 ? f.n_sites : 1ll << 36;  // a form without a size: the large shape
  auto cfg = [](int block, int tile, int stages, int ctas, int tpl) {
    return LaunchCfg{block, tile, stages, ctas, 0, tpl};
  };
  if (f.layout != SU3_LAYOUT_AOS) {
    // direct loads, AOSOA32 (256 threads, 4 CTAs, 1/2/4 links for 16/8/4-byte elements before): FP64
    // 5,050 (4,223), FP32 6,717 (6,333), two-row FP32 6,668 (6,222), FP16 6,426 (6,389), two-row
    // FP16 6,407 (5,468)
    if (f.dtype == SU3_F64) return f.arith == SU3_ARITH_NATIVE ? cfg(128, 1, 0, 16, 1) : cfg(256, 1, 0, 4, 1);
    if (narrow) return two_out ? cfg(128, 2, 0, 8, 1) : cfg(128, 4, 0, 4, 1);
    return two_out ? cfg(128, 2, 0, 4, 1) : cfg(256, 2, 0, 8, 1);
  }
  if (f.dtype == SU3_F64 && f.arith == SU3_ARITH_NATIVE) {
    if (two_out) return cfg(128, 48, 3, 4, 3);  // 4,977: 16 warps, rows as work items
    if (two_in) return cfg(64, 24, 2, 6, 1);    // 3,019: 12 warps of 154 registers; with three stages they do not fit
    return cfg(128, 32, 3, 4, 1);               // 5,094: 16 warps of 108 registers
  }
  if (f.dtype == SU3_F64) {  // FP32 pairs
    if (two_in) return cfg(128, 64, 3, 3, 1);                   // 5,683 (3,758); to full 4,430 (3,194)
    return n >= 1 << 18 ? cfg(128, 32, 3, 4, 1) : general_cfg(f);  // 5,906 (4,716); level at 10^5 sites
  }
  if (two_in != two_out) return general_cfg(f);
  if (f.dtype == SU3_F32) {
    if (two_out) return cfg(256, 96, 6, 1, 3);                     // 6,940 (6,010)
    return n >= 1 << 20 ? cfg(64, 128, 4, 1, 1) : general_cfg(f);  // 6,951 (6,339); 14.7 (10.6) us at 10^5 sites
  }
  return two_out ? general_cfg(f) : cfg(128, 64, 6, 3, 3);  // FP16 6,639 (5,790); two-row level
}

// The adjacent products: their FP64 forms take the product's shapes (a^dagger b 4,590, a v 6,139 GB/s);
// the narrower storage types, which have no row split here, the general one (FP16 a^dagger b 6,210 GB/s, 5,840
// in the product's shape).
LaunchCfg default_adjacent_cfg(const Form& f) { return f.dtype == SU3_F64 ? default_cfg(f) : general_cfg(f); }

LaunchCfg default_cfg(const Form& f) {
  if (f.arith == SU3_ARITH_HYBRID) return general_cfg(f);
  LaunchCfg c = measured_cfg(f);
  // a tile's sites may span 1 MiB of the array; wide strides keep tiles of 32 sites
  if (f.layout == SU3_LAYOUT_AOS)
    c.tile_sites = (int)std::min<int64_t>(c.tile_sites, std::max<int64_t>(32, (1 << 20) / std::max<int64_t>(f.a_stride, 1)));
  return c;
}

// cuTensorMapEncodeTiled, reached through the runtime's driver entry point (no link to libcuda).
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_tiled() {
  static const EncodeTiledFn fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return (EncodeTiledFn) nullptr;
    return reinterpret_cast<EncodeTiledFn>(f);
  }();
  return fn;
}

su3_status encode_2d(CUtensorMap* m, const void* base, long long inner, long long rows, long long pitch,
                     long long box_inner, long long box_rows, const LaunchCtx& ctx) {
  const EncodeTiledFn enc = encode_tiled();
  if (!enc) {
    *ctx.err = "cuTensorMapEncodeTiled is not available from the CUDA driver";
    return SU3_ERR_CUDA;
  }
  const cuuint64_t dim[2] = {(cuuint64_t)inner, (cuuint64_t)rows};
  const cuuint64_t stride[1] = {(cuuint64_t)pitch};
  const cuuint32_t box[2] = {(cuuint32_t)box_inner, (cuuint32_t)box_rows};
  const cuuint32_t estride[2] = {1, 1};
  const CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_UINT64, 2, const_cast<void*>(base), dim, stride, box, estride,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    *ctx.err = "cuTensorMapEncodeTiled failed (error " + std::to_string((int)r) + ")";
    return SU3_ERR_CUDA;
  }
  return SU3_OK;
}

// AOS arrays whose a or c sites are wider than their links go to the padded kernels.
static bool padded_sites(const Form& f, long long link_in, long long link_out) {
  return f.layout == SU3_LAYOUT_AOS && (f.a_stride != 4 * link_in || f.c_stride != 4 * link_out);
}

su3_status launch_mult(const Form& f, const LaunchCfg& cfg, const void* a, const double* b, void* c,
                       const LaunchCtx& ctx) {
  if (padded_sites(f, link_bytes(f.dtype, f.repr_in), link_bytes(f.dtype, f.repr_out)))
    return launch_mult_padded(f, cfg, a, b, c, ctx);
  return mult_dispatch<false>(f, cfg, a, b, c, ctx);
}

su3_status launch_adjacent(int which, const Form& f, const LaunchCfg& cfg, const void* a, const double* bv, void* c,
                           const LaunchCtx& ctx) {
  // output link: a 3x3 matrix (a^dagger b) or a colour vector of 3 complex numbers (a v, a^dagger v)
  const long long out = which == 0 ? link_bytes(f.dtype, SU3_REPR_FULL18) : 3 * 2 * real_bytes(f.dtype);
  if (padded_sites(f, link_bytes(f.dtype, f.repr_in), out)) return launch_adjacent_padded(which, f, cfg, a, bv, c, ctx);
  return adjacent_dispatch<false>(which, f, cfg, a, bv, c, ctx);
}

}  // namespace su3
