// Device-side building blocks of libsu3 (sm_103a): PTX wrappers for mbarriers, bulk async copies
// and cache-hinted vector memory operations, storage conversions, and the 3x3 complex link
// product of the SU3_Bench kernel (arXiv 2103.00571, §Background "SU3_Bench").
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>
#include <string.h>

#include "su3_internal.h"

namespace su3 {

// Upper bound on any spin-wait, in globaltimer nanoseconds.
constexpr unsigned long long kWaitLimitNs = 4000000000ull;

enum Dtype { kF64 = 0, kF32 = 1, kF16 = 2, kBF16 = 3 };

// ---- PTX wrappers -----------------------------------------------------------------------------

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, unsigned parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Waits for phase `parity` of an mbarrier; gives up after `limit_ns` and returns false.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, unsigned parity,
                                                  unsigned long long limit_ns = kWaitLimitNs) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = globaltimer_ns();
  for (;;) {
    if (mbar_try_wait(bar, parity)) return true;
    if (globaltimer_ns() - t0 > limit_ns) return false;
  }
}

// 1-D bulk async copy global -> this CTA's shared memory, completing `bytes` on `bar`.
// Both addresses 16-byte aligned, bytes a multiple of 16 (checked by the callers' invariants).
__device__ __forceinline__ void bulk_g2s(void* sdst, const void* gsrc, unsigned bytes, uint64_t* bar,
                                         uint64_t policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], "
      "%2, [%3], %4;" ::"r"(smem_u32(sdst)),
      "l"(gsrc), "r"(bytes), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}

// 1-D bulk async copy shared -> global, tracked by this thread's bulk groups.
__device__ __forceinline__ void bulk_s2g(void* gdst, const void* ssrc, unsigned bytes, uint64_t policy) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group.L2::cache_hint [%0], [%1], %2, %3;" ::"l"(gdst),
               "r"(smem_u32(ssrc)), "r"(bytes), "l"(policy)
               : "memory");
}

// 2-D tensor copies (the TMA engine reading a tensor map): the box at element coordinates (x, y)
// of the map. Load: global -> this CTA's shared memory, completing the box's bytes on `bar` (rows
// past the tensor's end arrive as zeros and count like the rest). Store: shared -> global, tracked
// by this thread's bulk groups; rows past the tensor's end are not written. The map is a
// __grid_constant__ kernel parameter (its generic address); shared memory 128-byte aligned.
__device__ __forceinline__ void tma_load_2d(void* sdst, const void* tmap, int x, int y, uint64_t* bar,
                                            uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], "
      "[%1, {%2, %3}], [%4], %5;" ::"r"(smem_u32(sdst)),
      "l"(tmap), "r"(x), "r"(y), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}

__device__ __forceinline__ void tma_store_2d(const void* tmap, int x, int y, const void* ssrc, uint64_t policy) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group.L2::cache_hint [%0, {%1, %2}], [%3], %4;" ::"l"(
                   tmap),
               "r"(x), "r"(y), "r"(smem_u32(ssrc)), "l"(policy)
               : "memory");
}

__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }

template <int N>
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}

template <int N>
__device__ __forceinline__ void bulk_wait_all() {
  asm volatile("cp.async.bulk.wait_group %0;" ::"n"(N) : "memory");
}

// Orders this thread's generic-proxy shared-memory writes before later async-proxy reads.
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}

// ---- streaming global loads/stores (read once: no L1 allocation; write once: evict-first) ----

__device__ __forceinline__ double2 ldg_stream(const double2* p) {
  double2 v;
  asm volatile("ld.global.nc.L1::no_allocate.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ float2 ldg_stream(const float2* p) {
  float2 v;
  asm volatile("ld.global.nc.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ uint32_t ldg_stream(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.global.nc.L1::no_allocate.b32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ void stg_stream(double2* p, double2 v) {
  asm volatile("st.global.cs.v2.f64 [%0], {%1, %2};" ::"l"(p), "d"(v.x), "d"(v.y) : "memory");
}
__device__ __forceinline__ void stg_stream(float2* p, float2 v) {
  asm volatile("st.global.cs.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void stg_stream(uint32_t* p, uint32_t v) {
  asm volatile("st.global.cs.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// ---- storage <-> arithmetic conversions --------------------------------------------------------
// A "complex element" of storage type T is stored as one vector: double2 (F64), float2 (F32),
// or a 32-bit word holding two 16-bit reals (F16/BF16), re in the low half.

template <int DT>
struct Storage;

template <>
struct Storage<kF64> {
  using real = double;   // storage real
  using vec = double2;   // one complex element in memory
  using acc = double;    // arithmetic type
  static constexpr int real_bytes = 8;
  __device__ static __forceinline__ void unpack(vec v, acc& re, acc& im) { re = v.x; im = v.y; }
  __device__ static __forceinline__ vec pack(acc re, acc im) { return make_double2(re, im); }
};

template <>
struct Storage<kF32> {
  using real = float;
  using vec = float2;
  using acc = float;
  static constexpr int real_bytes = 4;
  __device__ static __forceinline__ void unpack(vec v, acc& re, acc& im) { re = v.x; im = v.y; }
  __device__ static __forceinline__ vec pack(acc re, acc im) { return make_float2(re, im); }
};

template <>
struct Storage<kF16> {
  using real = __half;
  using vec = uint32_t;
  using acc = float;
  static constexpr int real_bytes = 2;
  __device__ static __forceinline__ void unpack(vec v, acc& re, acc& im) {
    __half2 h = *reinterpret_cast<__half2*>(&v);
    float2 f = __half22float2(h);
    re = f.x;
    im = f.y;
  }
  __device__ static __forceinline__ vec pack(acc re, acc im) {
    __half2 h = __floats2half2_rn(re, im);  // both halves rounded to nearest even
    return *reinterpret_cast<uint32_t*>(&h);
  }
};

template <>
struct Storage<kBF16> {
  using real = __nv_bfloat16;
  using vec = uint32_t;
  using acc = float;
  static constexpr int real_bytes = 2;
  __device__ static __forceinline__ void unpack(vec v, acc& re, acc& im) {
    re = __uint_as_float(v << 16);          // a bfloat16 is the top half of a binary32
    im = __uint_as_float(v & 0xffff0000u);
  }
  __device__ static __forceinline__ vec pack(acc re, acc im) {
    __nv_bfloat162 h = __floats2bfloat162_rn(re, im);
    return *reinterpret_cast<uint32_t*>(&h);
  }
};

// ---- b in the kernel parameters ---------------------------------------------------------------

// The four b matrices by value in a kernel's parameter block: b[j][row][col][re/im], plus the
// constant 1.0 that FP32-pair arithmetic multiplies by (see dot_pair2: as a kernel parameter its
// value is unknown to the compiler, so no multiply can be folded into the FMA that uses it).
// COLS > 0 (ops with kFixCols): with b of that many columns in fixed point for FP64 rows.
template <typename A, int COLS>
struct BMat {
  A v[72];
  float unit;
  FixedMat fix;
};
template <typename A>
struct BMat<A, 0> {
  A v[72];
  float unit;
};

template <typename A, int COLS>
inline BMat<A, COLS> make_b(const double* b) {
  BMat<A, COLS> m;
  for (int i = 0; i < 72; ++i) m.v[i] = (A)b[i];
  m.unit = 1.0f;
  if constexpr (COLS > 0) {
    memset(&m.fix, 0, sizeof(m.fix));
    m.fix.range = fix_b<COLS>(b, m.fix.fx, m.fix.mag, m.fix.eb) ? kFixExpRange : 0;
    m.fix.k = fixed_const();
  }
  return m;
}

// b in shared memory: its 72 reals, and with COLS > 0 (FP64 rows in fixed point) fix_b's words.
template <typename A, int COLS>
struct BShared {
  alignas(16) A v[72];
  int fx[4][9][4];
  unsigned mag[4][kFixMags];
};
template <typename A>
struct BShared<A, 0> {
  A v[72];
};
template <typename A>
struct BShared<A, 1> {  // one column: its limbs with either sign (FixedB<1>)
  alignas(16) A v[72];
  int fx[3][2][4][4];
  unsigned mag[4][kFixMags];
};
template <class Op>
using BSharedOf = BShared<typename Op::BArg, Op::kFixCols>;

// Stages b in shared memory and lets each thread's op take its direction j = tid % 4.
template <class Op>
__device__ __forceinline__ void load_b_op(const BMat<typename Op::BArg, Op::kFixCols>& b, BSharedOf<Op>* bsh, Op& op,
                                          int native_warps) {
  for (int i = threadIdx.x; i < 72; i += blockDim.x) bsh->v[i] = b.v[i];
  if constexpr (Op::kFixCols == 1) {
    for (int i = threadIdx.x; i < 3 * 4 * 2; i += blockDim.x) {  // element, direction, re or im
      const int e = i >> 3, j = (i >> 1) & 3, c = 2 * (i & 1);
      const long long x = ((long long)b.fix.fx[j][e][c] << 32) + b.fix.fx[j][e][c + 1];
      for (int s = 0; s < 2; ++s) {
        const long long v = s ? -x : x;
        bsh->fx[e][s][j][c + 1] = (int)v;
        bsh->fx[e][s][j][c] = (int)((v - (int)v) >> 32);
      }
    }
  } else if constexpr (Op::kFixCols > 0) {
    for (int i = threadIdx.x; i < 4 * 9 * 4; i += blockDim.x) (&bsh->fx[0][0][0])[i] = (&b.fix.fx[0][0][0])[i];
  }
  if constexpr (Op::kFixCols > 0) {
    for (int i = threadIdx.x; i < 4 * kFixMags; i += blockDim.x) (&bsh->mag[0][0])[i] = (&b.fix.mag[0][0])[i];
  }
  __syncthreads();
  const int j = threadIdx.x & 3;
  op.init(bsh->v + 18 * j, native_warps);
  op.set_unit(b.unit);
  if constexpr (Op::kFixCols == 1) op.set_fixed(b.fix, bsh->fx[0][0][j], bsh->mag[j], j);
  else if constexpr (Op::kFixCols > 0) op.set_fixed(b.fix, bsh->fx[j], bsh->mag[j], j);
}

// ---- the link product -------------------------------------------------------------------------

// A link in registers: up to 9 complex elements, row major (e = 3*row + col).
template <typename T>
struct Link {
  T re[9], im[9];
};

// Row 2 of an SU(3) matrix from rows 0 and 1: conj(row0 x row1), with
// (u x v)_k = u_p v_q - u_q v_p, (p, q) = (k+1, k+2) mod 3. r0/r1 hold rows 0 and 1 (re, im).
template <typename T>
__device__ __forceinline__ void rebuild_row2_elems(const T (&r0re)[3], const T (&r0im)[3], const T (&r1re)[3],
                                                   const T (&r1im)[3], T (&ore)[3], T (&oim)[3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int p = (k + 1) % 3, q = (k + 2) % 3;
    T xr = r0re[p] * r1re[q];
    xr = fma(-r0im[p], r1im[q], xr);
    xr = fma(-r0re[q], r1re[p], xr);
    xr = fma(r0im[q], r1im[p], xr);
    T xi = r0re[p] * r1im[q];
    xi = fma(r0im[p], r1re[q], xi);
    xi = fma(-r0re[q], r1im[p], xi);
    xi = fma(-r0im[q], r1re[p], xi);
    ore[k] = xr;
    oim[k] = -xi;
  }
}

template <typename T>
__device__ __forceinline__ void rebuild_row2(Link<T>& a) {
  T r0re[3], r0im[3], r1re[3], r1im[3], ore[3], oim[3];
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    r0re[m] = a.re[m];
    r0im[m] = a.im[m];
    r1re[m] = a.re[3 + m];
    r1im[m] = a.im[3 + m];
  }
  rebuild_row2_elems(r0re, r0im, r1re, r1im, ore, oim);
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    a.re[6 + m] = ore[m];
    a.im[6 + m] = oim[m];
  }
}

// One output row: c[l] = sum_m a[m] b[m][l] (the SU3_Bench kernel's inner l, m loops for one k;
// 4 real FMAs per complex multiply-accumulate).
template <typename T>
__device__ __forceinline__ void row_mult(const T (&are)[3], const T (&aim)[3], const T (&bre)[9], const T (&bim)[9],
                                         T (&cre)[3], T (&cim)[3]) {
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    T re = are[0] * bre[l];
    T im = are[0] * bim[l];
    re = fma(-aim[0], bim[l], re);
    im = fma(aim[0], bre[l], im);
#pragma unroll
    for (int m = 1; m < 3; ++m) {
      re = fma(are[m], bre[3 * m + l], re);
      re = fma(-aim[m], bim[3 * m + l], re);
      im = fma(are[m], bim[3 * m + l], im);
      im = fma(aim[m], bre[3 * m + l], im);
    }
    cre[l] = re;
    cim[l] = im;
  }
}

// c[k][l] = sum_m a[k][m] b[m][l] for rows k < ROWS.
template <int ROWS, typename T>
__device__ __forceinline__ void link_mult(const Link<T>& a, const T (&bre)[9], const T (&bim)[9],
                                          Link<T>& c) {
#pragma unroll
  for (int k = 0; k < ROWS; ++k) {
    T are[3], aim[3], cre[3], cim[3];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      are[m] = a.re[3 * k + m];
      aim[m] = a.im[3 * k + m];
    }
    row_mult(are, aim, bre, bim, cre, cim);
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      c.re[3 * k + l] = cre[l];
      c.im[3 * k + l] = cim[l];
    }
  }
}

// ---- FP64 rows in fixed point -------------------------------------------------------------------
// One output row takes 36 FP64 FMAs, of which GB300 does 2 per clock and SM: by themselves they
// hold the FP64 product at 24 % of the memory bandwidth, with every other unit idle. The integer
// units do 32 multiply-adds of 32 x 32 + 64 bits per clock and SM beside them. So five of a row's
// six output reals are computed in fixed point while the FP64 pipe computes the sixth:
//  * a's row becomes 61-bit fixed point relative to its largest real, A = ah * 2^32 + al with a
//    29-bit ah and a sign, and al a signed 32-bit limb; b comes from the host in the same form
//    (fix_b). A real within 2^-8 of the largest is exact; a smaller one is cut at 2^-61 of it.
//  * an output is the sum of six products A * B: H = sum ah*bh, X = sum ah*bl and Y = sum al*bh,
//    in 64-bit accumulators that cannot overflow (6 * 2^58, 6 * 2^60), and T = H + X/2^32 + Y/2^32.
//    al*bl is left out (below 1.5 units of T). X and Y start at 2^63 + 2^31 (xbias): unsigned, their
//    high words need no sign extension, and they are rounded; hbias takes the 2 * 2^31 back.
//  * T becomes a double with one rounding (fixed_to_f64).
// T's unit is 2^-58 of full scale, (the row's largest real) x (b's), each rounded up to a power of
// two. T is off by at most 3.7 units (al*bl 1.5, X and Y 0.5 each, a's cut 0.75, b's rounding 0.4),
// as a rule by 0.5. Limbs of zero make no error: products of few enough bits for FP64 FMAs to be
// exact (integers, as a rule) are exact here too.
// The 3.7 units do not shrink with the terms, so every output real passes a gate: the sum S of its six
// |a||b| must be 1/16 of full scale (by the estimate below it is not for 3 of 10^5 with random SU(3) matrices). Then 3.7 units
// are at most 1.9 * 2^-53 S, and the output is off by at most 2^-53 |c| + 1.9 * 2^-53 S, against 6 *
// 2^-53 S for six FMAs; over the matrices tried (random and near the identity, reals spread over
// up to 31 binary orders, integers) at most 1.6 * 2^-53 S against 4.7, r.m.s. 0.24 to 0.42 against 0.45
// to 0.79. S is estimated from below by two dot products of bytes, from |a| cut to 5 bits and |b| to 8.
// An output real that does not pass, or is below 2^-26 of full scale (not normalised), is computed by
// FP64 FMAs; so are all of a row whose reals are spread over more than 2^31 (any zero), not finite or
// outside 2^-723 .. 2^677, and all rows when fix_b refuses b. A warp does FMAs for the output reals
// that any of its lanes needs and the sixth once for all, 36 of them at most: no mix of values takes
// longer than FMAs throughout do. Which way an output goes depends on its row's and b's values only,
// so results are the same for every launch shape and layout.
// Measured (AOS, 48^4 sites, GB/s): FP64 FMAs alone 1,585; random SU(3) 5,099-5,128, 5,395 without the
// gate; links exp(i e H) at e = 0.05 2,982; an identity or real a or b 1,575. The wide multiply-adds
// and the other integer instructions share their issue, so they set the rate (364 instructions per
// row, 90 of them wide multiply-adds). 4 of 18 output reals on the FP64 pipe instead of 3: 4,916.
// b is read from shared memory for each row: in registers 4,869, at 124 of them instead of 108. S in FP32,
// on the idle half of the FP32 pipe: 4,739.

// b[j] (or v[j]) of one thread in fixed point, in memory. COLS 3: element e = 3*m + l at limbs[e]. COLS 1:
// element m at limbs[8*m], its negative at limbs[8*m + 4] (the four directions' side by side, so that
// the addresses of a warp's load fall into different banks).
template <int COLS>
struct FixedB {
  const int4* limbs;  // (re_hi, re_lo, im_hi, im_lo)
  const uint4* mags;  // fix_b's magnitudes, two words per column
  unsigned kb, range;
  FixedConst k;
  __device__ __forceinline__ void take(const void* fx, const void* mag, int eb, unsigned exp_range, const FixedConst& c) {
    limbs = static_cast<const int4*>(fx);
    mags = static_cast<const uint4*>(mag);
    kb = (unsigned)(1085 - 1080 - 31 + eb) << 20;
    range = exp_range;
    k = c;
  }
};

// a * b + c with a 64-bit accumulator. The carry-linked pair is issued as one IMAD.WIDE; mad.wide
// was split into a product and 64-bit adds.
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
  long long d;
  asm("{.reg .b32 lo, hi;\n\t"
      "mov.b64 {lo, hi}, %3;\n\t"
      "mad.lo.cc.s32 lo, %1, %2, lo;\n\t"
      "madc.hi.s32 hi, %1, %2, hi;\n\t"
      "mov.b64 %0, {lo, hi};}"
      : "=l"(d)
      : "r"(a), "r"(b), "l"(c));
  return d;
}

// T in units of 2^k as a double, rounded once to nearest; `base` is (1054 + k) << 20. Valid while |T|'s
// high word is not 0; else `bad` gets bits above the low five. A negative T is worked on as its one's
// complement, shifted with ones: one unit of its 63 normalised bits below |T|, which only turns a tie.
__device__ __forceinline__ double fixed_to_f64(long long t, unsigned base, unsigned& bad) {
  int th, tl;
  asm("mov.b64 {%0, %1}, %2;" : "=r"(tl), "=r"(th) : "l"(t));
  const int s = th >> 31;
  const unsigned ah = (unsigned)(th ^ s), al = (unsigned)(tl ^ s);
  unsigned p, mh, ml, lo, hi;
  asm("bfind.u32 %0, %1;" : "=r"(p) : "r"(ah));  // ~0 for 0
  bad |= p;
  const unsigned n = p + 2;
  asm("shf.r.wrap.b32 %0, %1, %2, %3;" : "=r"(mh) : "r"(al), "r"(ah), "r"(n));
  asm("shf.r.wrap.b32 %0, %1, %2, %3;" : "=r"(ml) : "r"(s), "r"(al), "r"(n));
  asm("{add.cc.u32 %0, %0, 0x200; addc.u32 %1, %1, 0;}" : "+r"(ml), "+r"(mh));
  asm("shf.r.wrap.b32 %0, %1, %2, 10;" : "=r"(lo) : "r"(ml), "r"(mh));
  hi = (mh >> 10) + ((base | ((unsigned)th & 0x80000000u)) + (p << 20));
  return __hiloint2double((int)hi, (int)lo);
}

// A row's exponents (reals a[0..2].re, a[0..2].im): their distances d from the largest, and e0 = 0x7ff -
// the largest exponent field. The row suits the fixed-point form when take() is true and spread() has
// no bit above the low five.
struct FixedExps {
  int d[6], e0;
  __device__ __forceinline__ bool take(const double (&are)[3], const double (&aim)[3], unsigned range) {
    unsigned hn[6];  // the complement of |x|'s high word, so that its exponent field grows as |x| falls
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      hn[m] = ~(unsigned)__double2hiint(are[m]) & 0x7fffffffu;
      hn[3 + m] = ~(unsigned)__double2hiint(aim[m]) & 0x7fffffffu;
    }
    const unsigned lowest = min(min(min(hn[0], hn[1]), min(hn[2], hn[3])), min(hn[4], hn[5]));
    e0 = (int)(lowest >> 20);
#pragma unroll
    for (int q = 0; q < 6; ++q) d[q] = (int)(hn[q] >> 20) - e0;
    return (unsigned)(0x7ff - kFixExpMin) - (unsigned)e0 < range;
  }
  __device__ __forceinline__ unsigned spread() const { return (unsigned)(d[0] | d[1] | d[2] | d[3] | d[4] | d[5]); }
};

// Output real `out` = 2*l + (0 re, 1 im) of the row a[] times column l of b, by FP64 FMAs in row_mult's
// order; bj = b[j] in FP64 (re, im of element COLS*m + l).
template <int COLS>
__device__ __forceinline__ double fma_output(const double (&are)[3], const double (&aim)[3], const double* bj, int out) {
  const int l = out >> 1, im = out & 1;
  double c = are[0] * bj[2 * l + im];
  c = fma(im ? aim[0] : -aim[0], bj[2 * l + 1 - im], c);
#pragma unroll
  for (int m = 1; m < 3; ++m) {
    c = fma(are[m], bj[2 * (COLS * m + l) + im], c);
    c = fma(im ? aim[m] : -aim[m], bj[2 * (COLS * m + l) + 1 - im], c);
  }
  return c;
}

// a's real x in fixed point without its sign, d binary orders below its row's largest: hi * 2^32 + lo, hi
// of 29 bits.
__device__ __forceinline__ void cut_real(double x, int d, unsigned lead, unsigned& hi, unsigned& lo) {
  const unsigned l = (unsigned)__double2loint(x);
  const unsigned m = ((unsigned)__double2hiint(x) & 0xfffffu) | lead;
  const unsigned w = __funnelshift_l(l, m, 8);
  hi = w >> d;
  lo = __funnelshift_r(l << 8, w, d);
}

// The set of output reals (bit 2*l + im) that do not pass the gate; `mag`: |re| of a's three elements,
// then |im|, 29 bits each.
template <int COLS, int NAT>
__device__ __forceinline__ unsigned small_outputs(const unsigned (&mag)[6], const uint4* mags) {
  constexpr int kOut = 2 * COLS - NAT;
  // |re|, |im| of elements 0 and 1, then of 2, in bytes of 1/32 of full scale; im's sums take
  // them the other way round
  const unsigned r01 = __byte_perm(__byte_perm(mag[0], mag[3], 0x0073), __byte_perm(mag[1], mag[4], 0x0073), 0x5410);
  const unsigned r2 = __byte_perm(mag[2], mag[5], 0x0073);  // b's bytes 2 and 3 are 0 here
  const unsigned i01 = __byte_perm(r01, 0, 0x2301), i2 = __byte_perm(r2, 0, 0x2301);
  unsigned bm[(2 * COLS + 3) / 4 * 4], rest = 0;
#pragma unroll
  for (int i = 0; i < (2 * COLS + 3) / 4; ++i) {
    const uint4 v = mags[i];
    bm[4 * i] = v.x;
    bm[4 * i + 1] = v.y;
    bm[4 * i + 2] = v.z;
    bm[4 * i + 3] = v.w;
  }
#pragma unroll
  for (int o = kOut - 1; o >= 0; --o) {
    const unsigned sum = __dp4a(o & 1 ? i2 : r2, bm[o | 1], 0u - kFixMinSum);
    rest = __funnelshift_l(__dp4a(o & 1 ? i01 : r01, bm[o & ~1], sum), rest, 1);  // its sign
  }
  return rest;
}

// T from H, X and Y.
__device__ __forceinline__ long long sum_limbs(long long h, long long x, long long y) {
  return h + (long long)((unsigned long long)x >> 32) + (long long)((unsigned long long)y >> 32);
}

// The output reals of a row but for the last NAT: c[2*l] = re and c[2*l + 1] = im of sum_m a[m] b[m][l],
// l < COLS. Returns the set (bit 2*l + im) of those that FP64 FMAs have to do instead.
template <int COLS, int NAT>
__device__ __forceinline__ unsigned fixed_row(const double (&are)[3], const double (&aim)[3], const FixedExps& ex,
                                              const FixedB<COLS>& b, double (&c)[2 * COLS]) {
  constexpr int kOut = 2 * COLS - NAT;
  int ah[6], al[6], nh[3], nl[3];  // limbs of re, im and -im
  unsigned mag[6];                 // the magnitudes' high words: 29 bits
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    const double x = q < 3 ? are[q % 3] : aim[q % 3];
    unsigned vh, vl;
    cut_real(x, ex.d[q], b.k.lead, vh, vl);
    mag[q] = vh;
    const unsigned s = (unsigned)(__double2hiint(x) >> 31);
    vh ^= s;
    vl ^= s;
    asm("{sub.cc.u32 %0, %0, %2; subc.u32 %1, %1, %2;}" : "+r"(vl), "+r"(vh) : "r"(s));
    ah[q] = (int)(vh + (vl >> 31));
    al[q] = (int)vl;
    if (q >= 3) {
      asm("{sub.cc.u32 %0, %2, %0; subc.u32 %1, %2, %1;}" : "+r"(vl), "+r"(vh) : "r"(b.k.zero));
      nh[q - 3] = (int)(vh + (vl >> 31));
      nl[q - 3] = (int)vl;
    }
  }
  const unsigned rest = small_outputs<COLS, NAT>(mag, b.mags);
  const unsigned base = ((0x7ffu - (unsigned)ex.e0) << 20) + b.kb;
  unsigned bad = ex.spread();
#pragma unroll
  for (int l = 0; l < COLS; ++l) {
    // re and im together: six independent chains of multiply-adds
    long long hr = b.k.hbias, xr = b.k.xbias, yr = b.k.xbias, hi = b.k.hbias, xi = b.k.xbias, yi = b.k.xbias;
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const int4 w = b.limbs[COLS * m + l];
      hr = mad_wide(ah[m], w.x, hr);
      hr = mad_wide(nh[m], w.z, hr);
      xr = mad_wide(ah[m], w.y, xr);
      xr = mad_wide(nh[m], w.w, xr);
      yr = mad_wide(al[m], w.x, yr);
      yr = mad_wide(nl[m], w.z, yr);
      if (2 * l + 1 < kOut) {
        hi = mad_wide(ah[m], w.z, hi);
        hi = mad_wide(ah[3 + m], w.x, hi);
        xi = mad_wide(ah[m], w.w, xi);
        xi = mad_wide(ah[3 + m], w.y, xi);
        yi = mad_wide(al[m], w.z, yi);
        yi = mad_wide(al[3 + m], w.x, yi);
      }
    }
    c[2 * l] = fixed_to_f64(sum_limbs(hr, xr, yr), base, bad);
    if (2 * l + 1 < kOut) c[2 * l + 1] = fixed_to_f64(sum_limbs(hi, xi, yi), base, bad);
  }
  return bad & ~31u ? ~0u : rest;
}

// The same for one column, c[0] = re and c[1] = im: a's limbs without their signs, which choose b's
// instead. With two outputs a row, six sign changes and three negations cost more than the loads (a v
// at L=48 5,566 -> 6,158 GB/s, a^dagger v 5,246 -> 5,695; with three columns the loads cost more, 5,094 ->
// 4,808).
__device__ __forceinline__ unsigned fixed_row(const double (&are)[3], const double (&aim)[3], const FixedExps& ex,
                                              const FixedB<1>& b, double (&c)[2]) {
  unsigned mag[6], low[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) cut_real(q < 3 ? are[q % 3] : aim[q % 3], ex.d[q], b.k.lead, mag[q], low[q]);
  const unsigned rest = small_outputs<1, 0>(mag, b.mags);
  const unsigned base = ((0x7ffu - (unsigned)ex.e0) << 20) + b.kb;
  unsigned bad = ex.spread();
  long long hr = b.k.hbias, xr = b.k.xbias, yr = b.k.xbias, hi = b.k.hbias, xi = b.k.xbias, yi = b.k.xbias;
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    const int sr = (__double2hiint(are[m]) >> 31) & 4, si = (__double2hiint(aim[m]) >> 31) & 4;
    const int4 w = b.limbs[8 * m + sr];                                                   // b with re's sign
    const int2 u = reinterpret_cast<const int2*>(b.limbs)[2 * (8 * m + (si ^ 4)) + 1];  // im of b with -im's
    const int2 v = reinterpret_cast<const int2*>(b.limbs)[2 * (8 * m + si)];              // re of b with im's
    const int rh = (int)(mag[m] + (low[m] >> 31)), rl = (int)low[m];
    const int ih = (int)(mag[3 + m] + (low[3 + m] >> 31)), il = (int)low[3 + m];
    hr = mad_wide(rh, w.x, hr);
    hr = mad_wide(ih, u.x, hr);
    xr = mad_wide(rh, w.y, xr);
    xr = mad_wide(ih, u.y, xr);
    yr = mad_wide(rl, w.x, yr);
    yr = mad_wide(il, u.x, yr);
    hi = mad_wide(rh, w.z, hi);
    hi = mad_wide(ih, v.x, hi);
    xi = mad_wide(rh, w.w, xi);
    xi = mad_wide(ih, v.y, xi);
    yi = mad_wide(rl, w.z, yi);
    yi = mad_wide(il, v.x, yi);
  }
  c[0] = fixed_to_f64(sum_limbs(hr, xr, yr), base, bad);
  c[1] = fixed_to_f64(sum_limbs(hi, xi, yi), base, bad);
  return bad & ~31u ? ~0u : rest;
}

// A whole row c = a b (c as in fixed_row): its output reals in fixed point where that suits, the last
// NAT and the others by FP64 FMAs. bj = b[j] in FP64. The fixed-point part is run for every row, since a
// branch around it would run the last NAT twice in a warp whose rows differ (one link of four the
// identity, 2^21 sites: 1.78 ms with a branch, 1.53 so, 1.58 with FMAs throughout).
template <int COLS, int NAT>
__device__ __forceinline__ void row_f64(const double (&are)[3], const double (&aim)[3], const FixedB<COLS>& b,
                                        const double* bj, double (&c)[2 * COLS]) {
  constexpr int kOut = 2 * COLS - NAT;
  unsigned rest = ~0u;
  if (b.range) {  // else b does not suit: the same for every thread
    FixedExps ex;
    const bool ok = ex.take(are, aim, b.range);
    if constexpr (COLS == 1) rest = fixed_row(are, aim, ex, b, c);
    else rest = fixed_row<COLS, NAT>(are, aim, ex, b, c);
    rest = ok ? rest : ~0u;
#pragma unroll
    for (int o = kOut; o < 2 * COLS; ++o) c[o] = fma_output<COLS>(are, aim, bj, o);
  } else {
#pragma unroll
    for (int o = kOut; o < 2 * COLS; ++o) c[o] = fma_output<COLS>(are, aim, bj, o);
  }
  if (rest) {
#pragma unroll
    for (int o = 0; o < kOut; ++o)
      if (rest >> o & 1) c[o] = fma_output<COLS>(are, aim, bj, o);
  }
}

// ---- per-link operations used by the streaming kernels ----------------------------------------
// An op owns this thread's copy of b[j] (j = tid % 4) and turns one input link (NE_IN complex
// storage elements) into one output link (3*ROWS_OUT elements). `src` and `dst` may alias.
// Element e of the input link is src[e * ES_IN] and of the output link dst[e * ES_OUT]: 1 for a
// link stored contiguously (AOS), 32 inside an AOSOA32 block, the plane stride inside an SOA tile.
// Ops with kRowSplit also compute a single output row (apply_row), with the same operations as
// apply(), for launches with one thread per output row.

template <int DT, int NE_IN, int ROWS_OUT>
struct NativeOp {
  using S = Storage<DT>;
  using A = typename S::acc;   // FP64 for F64 storage, FP32 otherwise
  using V = typename S::vec;
  using BArg = A;              // precision of b in the kernel parameters
  static constexpr int kFixCols = 0, kMinCtas = 0;
  static constexpr int kNeIn = NE_IN, kNeOut = 3 * ROWS_OUT;
  static constexpr bool kRowSplit = true;  // has apply_row: one thread per output row is possible
  A bre[9], bim[9];
  __device__ __forceinline__ void begin_tile(int) {}
  __device__ __forceinline__ void set_unit(float) {}
  __device__ __forceinline__ void init(const BArg* bj, int /*native_warps*/) {
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      bre[e] = bj[2 * e];
      bim[e] = bj[2 * e + 1];
    }
  }
  template <int ES_IN = 1, int ES_OUT = 1>
  __device__ __forceinline__ void apply(const V* src, V* dst) const {
    Link<A> la, lc;
#pragma unroll
    for (int e = 0; e < NE_IN; ++e) S::unpack(src[e * ES_IN], la.re[e], la.im[e]);
    if (NE_IN == 6 && ROWS_OUT == 3) rebuild_row2(la);
    link_mult<ROWS_OUT>(la, bre, bim, lc);
#pragma unroll
    for (int e = 0; e < 3 * ROWS_OUT; ++e) dst[e * ES_OUT] = S::pack(lc.re[e], lc.im[e]);
  }
  // Output row k alone (row split: one thread per output row). Reads input row k only, except
  // that a rebuilt row 2 reads rows 0 and 1; the arithmetic is exactly that of apply().
  template <int ES_IN = 1, int ES_OUT = 1>
  __device__ __forceinline__ void apply_row(const V* src, V* dst, int k) const {
    A are[3], aim[3], cre[3], cim[3];
    if (NE_IN == 6 && ROWS_OUT == 3 && k == 2) {
      A r0re[3], r0im[3], r1re[3], r1im[3];
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        S::unpack(src[m * ES_IN], r0re[m], r0im[m]);
        S::unpack(src[(3 + m) * ES_IN], r1re[m], r1im[m]);
      }
      rebuild_row2_elems(r0re, r0im, r1re, r1im, are, aim);
    } else {
#pragma unroll
      for (int m = 0; m < 3; ++m) S::unpack(src[(3 * k + m) * ES_IN], are[m], aim[m]);
    }
    row_mult(are, aim, bre, bim, cre, cim);
#pragma unroll
    for (int l = 0; l < 3; ++l) dst[(3 * k + l) * ES_OUT] = S::pack(cre[l], cim[l]);
  }
};

// FP64 storage: rows in fixed point (fixed_row), or by FP64 FMAs where a row or b does not suit.
template <int NE_IN, int ROWS_OUT>
struct NativeOp<kF64, NE_IN, ROWS_OUT> {
  using S = Storage<kF64>;
  using V = double2;
  using BArg = double;
  static constexpr int kFixCols = 3;
    static constexpr int kMinCtas = NE_IN == 6 && ROWS_OUT == 3 ? 1 : 2;
  static constexpr int kNeIn = NE_IN, kNeOut = 3 * ROWS_OUT;
  static constexpr bool kRowSplit = true;
  // output reals per row on the FP64 pipe; two-row in, full out has its rebuild of row 2 there
  static constexpr int kNat = NE_IN == 6 && ROWS_OUT == 3 ? 0 : 1;
  FixedB<3> fix;
  const double* bm;  // b[j] in FP64, in shared memory
  __device__ __forceinline__ void begin_tile(int) {}
  __device__ __forceinline__ void set_unit(float) {}
  __device__ __forceinline__ void init(const BArg* bj, int /*native_warps*/) { bm = bj; }
  __device__ __forceinline__ void set_fixed(const FixedMat& f, const void* fx, const void* mag, int j) {
    fix.take(fx, mag, f.eb[j], f.range, f.k);
  }
  __device__ __forceinline__ void row(const double (&are)[3], const double (&aim)[3], double (&cre)[3],
                                      double (&cim)[3]) const {
    double c[6];
    row_f64<3, kNat>(are, aim, fix, bm, c);
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      cre[l] = c[2 * l];
      cim[l] = c[2 * l + 1];
    }
  }
  template <int ES_IN = 1, int ES_OUT = 1>
  __device__ __forceinline__ void apply(const V* src, V* dst) const {
    if constexpr (NE_IN == 6 && ROWS_OUT == 3) {
      // two-row in, full out (never in place): row 2 is rebuilt first, so that the FP64 pipe works on
      // it beside rows 0 and 1 (2,937 against 2,878 GB/s at L=48; the same operations as apply_row, so
      // the same bits)
      double r0re[3], r0im[3], r1re[3], r1im[3], r2re[3], r2im[3], cre[3], cim[3];
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        S::unpack(src[m * ES_IN], r0re[m], r0im[m]);
        S::unpack(src[(3 + m) * ES_IN], r1re[m], r1im[m]);
      }
      rebuild_row2_elems(r0re, r0im, r1re, r1im, r2re, r2im);
      auto put = [&](int k) {
#pragma unroll
        for (int l = 0; l < 3; ++l) dst[(3 * k + l) * ES_OUT] = S::pack(cre[l], cim[l]);
      };
      row(r0re, r0im, cre, cim);
      put(0);
      row(r1re, r1im, cre, cim);
      put(1);
      row(r2re, r2im, cre, cim);
      put(2);
      return;
    }
#pragma unroll
    for (int k = 0; k < ROWS_OUT; ++k) apply_row<ES_IN, ES_OUT>(src, dst, k);
  }
  // Output row k alone (row split: one thread per output row). Reads input row k only, except
  // that a rebuilt row 2 reads rows 0 and 1 (two-row in, full out is never in place).
  template <int ES_IN = 1, int ES_OUT = 1>
  __device__ __forceinline__ void apply_row(const V* src, V* dst, int k) const {
    double are[3], aim[3], cre[3], cim[3];
    if (NE_IN == 6 && ROWS_OUT == 3 && k == 2) {
      double r0re[3], r0im[3], r1re[3], r1im[3];
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        S::unpack(src[m * ES_IN], r0re[m], r0im[m]);
        S::unpack(src[(3 + m) * ES_IN], r1re[m], r1im[m]);
      }
      rebuild_row2_elems(r0re, r0im, r1re, r1im, are, aim);
    } else {
#pragma unroll
      for (int m = 0; m < 3; ++m) S::unpack(src[(3 * k + m) * ES_IN], are[m], aim[m]);
    }
    row(are, aim, cre, cim);
#pragma unroll
    for (int l = 0; l < 3; ++l) dst[(3 * k + l) * ES_OUT] = S::pack(cre[l], cim[l]);
  }
};

// ---- adjacent SU(3) operations ----------------------------------------------------------------
// The other per-link SU(3) products of lattice-QCD codes next to the benchmark's a x b: a^dagger x b (MILC's
// mult_su3_an) and the matrix x colour-vector products a v and a^dagger v (mult_su3_mat_vec and
// its adjoint), with b or v fixed per link direction exactly as in the SU3_Bench kernel.
// (a x b^dagger needs no kernel of its own: b^dagger is formed exactly on the host.)

template <int DT>
struct AnOp {  // c[k][l] = sum_m conj(a[m][k]) b[m][l]
  using S = Storage<DT>;
  using A = typename S::acc;
  using V = typename S::vec;
  using BArg = A;
  static constexpr int kFixCols = 0, kMinCtas = 0;
  static constexpr int kNeIn = 9, kNeOut = 9;
  static constexpr bool kRowSplit = false;  // row k of a^dagger b reads column k of a
  A bre[9], bim[9];
  __device__ __forceinline__ void begin_tile(int) {}
  __device__ __forceinline__ void set_unit(float) {}
  __device__ __forceinline__ void init(const BArg* bj, int) {
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      bre[e] = bj[2 * e];
      bim[e] = bj[2 * e + 1];
    }
  }
  template <int ES_IN = 1, int ES_OUT = 1>
  __device__ __forceinline__ void apply(const V* src, V* dst) const {
    Link<A> la;
#pragma unroll
    for (int e = 0; e < 9; ++e) S::unpack(src[e * ES_IN], la.re[e], la.im[e]);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
#pragma unroll
      for (int l = 0; l < 3; ++l) {
        // conj(a) = (ar, -ai): re += ar br + ai bi, im += ar bi - ai br
        A re = la.re[k] * bre[l];
        A im = la.re[k] * bim[l];
        re = fma(la.im[k], bim[l], re);
        im = fma(-la.im[k], bre[l], im);
#pragma unroll
        for (int m = 1; m < 3; ++m) {
          re = fma(la.re[3 * m + k], bre[3 * m + l], re);
          re = fma(la.im[3 * m + k], bim[3 * m + l], re);
          im = fma(la.re[3 * m + k], bim[3 * m + l], im);
          im = fma(-la.im[3 * m + k], bre[3 * m + l], im);
        }
        dst[(3 * k + l) * ES_OUT] = S::pack(re, im);
      }
    }
  }
};

template <int DT, bool ADJ>
struct MatVecOp {  // w[k] = sum_m a[k][m] v[m]   (ADJ: sum_m conj(a[m][k]) v[m])
  using S = Storage<DT>;
  using A = typename S::acc;
  using V = typename S::vec;
  using BArg = A;
  static constexpr int kFixCols = 0, kMinCtas = 0;
  static constexpr int kNeIn = 9, kNeOut = 3;
  static constexpr bool kRowSplit = false;  // one output vector per link
  A vre[3], vim[3];
  __device__ __forceinline__ void begin_tile(int) {}
  __device__ __forceinline__ void set_unit(float) {}
  __device__ __forceinline__ void init(const BArg* vj, int) {
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      vre[m] = vj[2 * m];
      vim[m] = vj[2 * m + 1];
    }
  }
  template <int ES_IN = 1, int ES_OUT = 1>
  __device__ __forceinline__ void apply(const V* src, V* dst) const {
    Link<A> la;
#pragma unroll
    for (int e = 0; e < 9; ++e) S::unpack(src[e * ES_IN], la.re[e], la.im[e]);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      A re = 0, im = 0;
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        const int e = ADJ ? 3 * m + k : 3 * k + m;
        const A ai = ADJ ? -la.im[e] : la.im[e];
        re = fma(la.re[e], vre[m], re);
        re = fma(-ai, vim[m], re);
        im = fma(la.re[e], vim[m], im);
        im = fma(ai, vre[m], im);
      }
      dst[k * ES_OUT] = S::pack(re, im);
    }
  }
};

// The same for FP64 storage, rows in fixed point (fixed_row): row k of a^dagger b is the conjugate of
// a's column k times b, and an element of a v is a's row k times the one column v (all in fixed point:
// with one of six on the FP64 pipe a^dagger v measured 9 % slower). At L=48, FP64 FMAs before:
// a^dagger b 1,568 -> 4,852 GB/s, a v 2,960 -> 6,158, a^dagger v 2,950 -> 5,695 (the products' launch shape).
template <>
struct AnOp<kF64> {
  using V = double2;
  using BArg = double;
  static constexpr int kFixCols = 3;
  static constexpr int kMinCtas = 2;  // 128 registers: 148 otherwise, which the product's 4 x 128 threads exceed
  static constexpr int kNeIn = 9, kNeOut = 9;
  static constexpr bool kRowSplit = false;  // row k of a^dagger b reads column k of a
  NativeOp<kF64, 9, 3> op;                  // b and the row routine
  __device__ __forceinline__ void begin_tile(int) {}
  __device__ __forceinline__ void set_unit(float) {}
  __device__ __forceinline__ void init(const BArg* bj, int w) { op.init(bj, w); }
  __device__ __forceinline__ void set_fixed(const FixedMat& f, const void* fx, const void* mag, int j) {
    op.set_fixed(f, fx, mag, j);
  }
  template <int ES_IN = 1, int ES_OUT = 1>
  __device__ __forceinline__ void apply(const V* src, V* dst) const {
    double2 a[9];  // all of a first: the output may overwrite it (in place)
#pragma unroll
    for (int e = 0; e < 9; ++e) a[e] = src[e * ES_IN];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      double are[3], aim[3], cre[3], cim[3];
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        are[m] = a[3 * m + k].x;
        aim[m] = -a[3 * m + k].y;
      }
      op.row(are, aim, cre, cim);
#pragma unroll
      for (int l = 0; l < 3; ++l) dst[(3 * k + l) * ES_OUT] = make_double2(cre[l], cim[l]);
    }
  }
};

template <bool ADJ>
struct MatVecOp<kF64, ADJ> {
  using V = double2;
  using BArg = double;
  static constexpr int kFixCols = 1;
  static constexpr int kMinCtas = 1;
  static constexpr int kNeIn = 9, kNeOut = 3;
  static constexpr bool kRowSplit = false;  // one output vector per link
  FixedB<1> fix;
  const double* vm;  // v[j] in FP64, in shared memory
  __device__ __forceinline__ void begin_tile(int) {}
  __device__ __forceinline__ void set_unit(float) {}
  __device__ __forceinline__ void init(const BArg* vj, int) { vm = vj; }
  __device__ __forceinline__ void set_fixed(const FixedMat& f, const void* fx, const void* mag, int j) {
    fix.take(fx, mag, f.eb[j], f.range, f.k);
  }
  template <int ES_IN, int ES_OUT>
  __device__ __forceinline__ void element(const V* src, V* dst, int k) const {
    double are[3], aim[3], w[2];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const double2 x = src[(ADJ ? 3 * m + k : 3 * k + m) * ES_IN];
      are[m] = x.x;
      aim[m] = ADJ ? -x.y : x.y;
    }
    row_f64<1, 0>(are, aim, fix, vm, w);
    dst[k * ES_OUT] = make_double2(w[0], w[1]);
  }
  template <int ES_IN = 1, int ES_OUT = 1>
  __device__ __forceinline__ void apply(const V* src, V* dst) const {
#pragma unroll
    for (int k = 0; k < 3; ++k) element<ES_IN, ES_OUT>(src, dst, k);
  }
};

// ---- FP64 storage with FP32-pair ("double-float") arithmetic ----------------------------------
// GB300 issues FP64 FMAs at 1/64 of the FP32 rate, and even double<->float conversions run on the
// FP64 pipe. This op keeps FP64 in memory but computes with unevaluated pairs of FP32 numbers:
//  * split: a double x becomes hi + lo, hi = x truncated to 24 significant bits (integer bit
//    operations on the exponent and mantissa), lo = the remaining 29 mantissa bits, converted with
//    one rounding (I2F) and scaled by 2^(e-52). |x - hi - lo| <= 2^-48 |x|. Valid for
//    2^-74 <= |x| < 2^127; smaller magnitudes (including 0) are replaced by a value below 2^-73.
//  * each real output is a 6-term dot product (Ogita, Rump and Oishi's Dot2 scheme, SIAM J. Sci.
//    Comput. 26 (2005)): products x_hi*y_hi are split exactly into p + e by an FMA (TwoProduct),
//    the p's are summed with Knuth's TwoSum, and every error term (e, the TwoSum errors and the
//    cross products x_hi*y_lo + x_lo*y_hi) is accumulated in a second FP32 number;
//  * the real and imaginary parts of each complex output run as the two lanes of Blackwell's
//    packed FP32x2 add/mul/fma, halving the FP32 instruction count;
//  * the pair (s, L) becomes a double by building both halves' FP64 bit patterns with integer
//    operations (exact for normal floats) and one FP64 add. (Assembling it with integer
//    operations only, to leave the FP64 pipe idle, measured slower: the extra integer work costs
//    more issue slots than the FP64 add.)
// Measured error against the FP64 oracle on random SU(3) data: max ~3e-14, RMS ~2e-15.

struct FF {
  float h, l;
};

__device__ __forceinline__ FF split_f64(double x) {
  const unsigned H = (unsigned)__double2hiint(x);
  const unsigned Lw = (unsigned)__double2loint(x);
  unsigned ax = H & 0x7FFFFFFFu;
  ax = max(ax, (949u << 20));  // |x| >= 2^-74 keeps every exponent below in range
  const unsigned hb = __funnelshift_l(Lw, ax - (896u << 20), 3) | (H & 0x80000000u);
  const unsigned sb = (hb & 0xFF800000u) - (52u << 23);  // sign | 2^(e-52)
  FF r;
  r.h = __uint_as_float(hb);
  r.l = __uint2float_rn(Lw & 0x1FFFFFFFu) * __uint_as_float(sb);
  return r;
}

// Exact FP64 value of a normal float, built from its bits (zero maps to 2^-127). The arithmetic
// shift copies the sign into bits 28-31; the mask keeps bit 31 and the exponent and mantissa in
// bits 0-27, and adding the exponent bias difference (1023 - 127) << 20 cannot carry into the
// sign. Four integer operations (one fewer than or-ing the sign back in: 1.3 % faster measured).
__device__ __forceinline__ double f32_bits_to_f64(float f) {
  const int b = __float_as_int(f);
  const unsigned hi = ((unsigned)(b >> 3) & 0x8FFFFFFFu) + (896u << 20);
  return __hiloint2double((int)hi, (int)((unsigned)b << 29));
}

// Packed FP32x2 arithmetic (Blackwell's add/mul/fma.f32x2: two independent, individually
// rounded FP32 operations per instruction). a - b is computed as fma(b, -1, a), which rounds
// exactly like a subtraction.
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

// The real and imaginary parts of one complex output as two lanes of FP32x2 operations:
// sum_{t<N} x_t * y_t with x = (xh, xl) broadcast to both lanes and y = (yh, yl) per lane, in the
// manner of Ogita, Rump and Oishi's Dot2. Per term t: the product p = fl(xh*yh), Knuth's TwoSum
// s2 = s + p with its two exact error parts t1 (s's share) and t2 = p - z (p's share, z = s2 - s),
// and the product error e = xh*yh - p. Since e and t2 are always added together and
// e + t2 = xh*yh - z exactly, one FMA gives their sum with a single rounding of a value of size
// ~ulp(s2) (so ~2^-48 of the sum); t1 and that FMA go to one error accumulator, the cross
// products xh*yl + xl*yh to another. That is 10 FP32x2 operations per term instead of 12.
// The add s + p is written as fma(p, unit, s) with unit = 1.0 passed as a kernel parameter: p's
// only use is then inside an FMA's multiplicand, which the compiler cannot merge with p's multiply.
// (As a plain add of a single-use product it was contracted into fma(xh, yh, s), which rounds
// s2 differently from the TwoSum's p and loses the error term: ~2^-24 results, measured.)
// The result is the unevaluated pair s + L per lane.
template <int N>
__device__ __forceinline__ void dot_pair2(const float (&xh)[N], const float (&xl)[N], const float2 (&yh)[N],
                                          const float2 (&yl)[N], float2 one, float2& s_out, float2& L_out) {
  float2 x0h = make_float2(xh[0], xh[0]), x0l = make_float2(xl[0], xl[0]);
  float2 s = mul2(x0h, yh[0]);
  float2 Lt = fma2(x0h, yh[0], make_float2(-s.x, -s.y));  // e of the first product
  float2 Lc = fma2(x0h, yl[0], mul2(x0l, yh[0]));
#pragma unroll
  for (int t = 1; t < N; ++t) {
    const float2 xth = make_float2(xh[t], xh[t]), xtl = make_float2(xl[t], xl[t]);
    const float2 p = mul2(xth, yh[t]);
    const float2 s2 = fma2(p, one, s);
    const float2 z = sub2(s2, s);
    const float2 t1 = sub2(s, sub2(s2, z));
    s = s2;
    Lt = add2(Lt, t1);
    Lt = add2(Lt, fma2(xth, yh[t], make_float2(-z.x, -z.y)));  // e + t2 in one rounding
    Lc = fma2(xth, yl[t], Lc);
    Lc = fma2(xtl, yh[t], Lc);
  }
  s_out = s;
  L_out = add2(Lt, Lc);
}

// One complex output of the product: the 6-term pair dot product, assembled into FP64.
__device__ __forceinline__ double2 dot6_pair2(const float (&xh)[6], const float (&xl)[6], const float2 (&yh)[6],
                                              const float2 (&yl)[6], float2 one) {
  float2 s, L;
  dot_pair2<6>(xh, xl, yh, yl, one, s, L);
  return make_double2(f32_bits_to_f64(s.x) + f32_bits_to_f64(L.x), f32_bits_to_f64(s.y) + f32_bits_to_f64(L.y));
}

// Row 2 of a two-row link, conj(u x v) with u = row 0 and v = row 1, in FP32-pair arithmetic: from
// the pair splits of the two rows (terms 2m = re, 2m+1 = im of element m) to the pair (wh, wl)
// of each real of row 2. Element k is conj(u_p v_q - u_q v_p), (p, q) = (k+1, k+2) mod 3; its
// (re, im) lanes are one 4-term dot product with a's row-0 reals broadcast and row-1 reals,
// negated or swapped, per lane:
//   re = up.re vq.re - up.im vq.im - uq.re vp.re + uq.im vp.im
//   im = -up.re vq.im - up.im vq.re + uq.re vp.im + uq.im vp.re
// The pair (s, L) of a Dot2 is itself a split of the value (s carries 24 bits, L the rest), so
// row 2 goes into the product with no FP64 operation.
__device__ __forceinline__ void rebuild_row2_pair(const float (&uh)[6], const float (&ul)[6], const float (&vh)[6],
                                                  const float (&vl)[6], float2 one, float (&wh)[6], float (&wl)[6]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int p = (k + 1) % 3, q = (k + 2) % 3;
    const float xh[4] = {uh[2 * p], uh[2 * p + 1], uh[2 * q], uh[2 * q + 1]};
    const float xl[4] = {ul[2 * p], ul[2 * p + 1], ul[2 * q], ul[2 * q + 1]};
    const float2 yh[4] = {make_float2(vh[2 * q], -vh[2 * q + 1]), make_float2(-vh[2 * q + 1], -vh[2 * q]),
                          make_float2(-vh[2 * p], vh[2 * p + 1]), make_float2(vh[2 * p + 1], vh[2 * p])};
    const float2 yl[4] = {make_float2(vl[2 * q], -vl[2 * q + 1]), make_float2(-vl[2 * q + 1], -vl[2 * q]),
                          make_float2(-vl[2 * p], vl[2 * p + 1]), make_float2(vl[2 * p + 1], vl[2 * p])};
    float2 sv, Lv;
    dot_pair2<4>(xh, xl, yh, yl, one, sv, Lv);
    wh[2 * k] = sv.x;
    wl[2 * k] = Lv.x;
    wh[2 * k + 1] = sv.y;
    wl[2 * k + 1] = Lv.y;
  }
}

template <int NE_IN, int ROWS_OUT>
struct PairF64Op {
  using V = double2;
  using BArg = double;
  static constexpr int kFixCols = 0, kMinCtas = 0;
  static constexpr int kNeIn = NE_IN, kNeOut = 3 * ROWS_OUT;
  static constexpr bool kRowSplit = true;
  // b[j] split once per thread, as lane pairs for the two terms of each (m, l):
  // (re, im) lanes of ar*(br, bi) and of ai*(-bi, br), high and low parts.
  float2 ya[9], yb[9], yla[9], ylb[9];
  float2 one;  // (1, 1), from the kernel parameters (dot_pair2)
  __device__ __forceinline__ void begin_tile(int) {}
  __device__ __forceinline__ void set_unit(float u) { one = make_float2(u, u); }
  __device__ __forceinline__ void init(const double* bj, int /*native_warps*/) {
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      const double r = bj[2 * e], i = bj[2 * e + 1];
      const float rh = __double2float_rn(r), ih = __double2float_rn(i);
      const float rl = __double2float_rn(r - (double)rh), il = __double2float_rn(i - (double)ih);
      ya[e] = make_float2(rh, ih);
      yb[e] = make_float2(-ih, rh);
      yla[e] = make_float2(rl, il);
      ylb[e] = make_float2(-il, rl);
    }
  }
  // The same constants from a host-side split: pre[4e..4e+3] = (re_hi, im_hi, re_lo, im_lo).
  __device__ __forceinline__ void init_pre(const float* pre) {
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      const float rh = __ldg(pre + 4 * e), ih = __ldg(pre + 4 * e + 1);
      const float rl = __ldg(pre + 4 * e + 2), il = __ldg(pre + 4 * e + 3);
      ya[e] = make_float2(rh, ih);
      yb[e] = make_float2(-ih, rh);
      yla[e] = make_float2(rl, il);
      ylb[e] = make_float2(-il, rl);
    }
  }
  // The pair split of input row r (terms 2m: re, 2m+1: im of element m).
  template <int ES_IN>
  __device__ __forceinline__ void split_row(const V* src, int r, float (&xh)[6], float (&xl)[6]) const {
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const double2 v = src[(3 * r + m) * ES_IN];
      const FF re = split_f64(v.x), im = split_f64(v.y);
      xh[2 * m] = re.h;
      xl[2 * m] = re.l;
      xh[2 * m + 1] = im.h;
      xl[2 * m + 1] = im.l;
    }
  }
  // Output row k from the pair split (xh, xl) of the input row.
  template <int ES_OUT>
  __device__ __forceinline__ void row_out(const float (&xh)[6], const float (&xl)[6], V* dst, int k) const {
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      float2 yh[6], yl[6];
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        yh[2 * m] = ya[3 * m + l];
        yl[2 * m] = yla[3 * m + l];
        yh[2 * m + 1] = yb[3 * m + l];
        yl[2 * m + 1] = ylb[3 * m + l];
      }
      dst[(3 * k + l) * ES_OUT] = dot6_pair2(xh, xl, yh, yl, one);
    }
  }
  // Output row k: reads input row k and writes output row k (so src and dst may alias). Row 2 of
  // a two-row input is first rebuilt from rows 0 and 1 in pair arithmetic (rebuild_row2_pair).
  template <int ES_IN = 1, int ES_OUT = 1>
  __device__ __forceinline__ void apply_row(const V* src, V* dst, int k) const {
    float xh[6], xl[6];
    if (NE_IN == 6 && ROWS_OUT == 3 && k == 2) {
      float uh[6], ul[6], vh[6], vl[6];
      split_row<ES_IN>(src, 0, uh, ul);
      split_row<ES_IN>(src, 1, vh, vl);
      rebuild_row2_pair(uh, ul, vh, vl, one, xh, xl);
    } else {
      split_row<ES_IN>(src, k, xh, xl);
    }
    row_out<ES_OUT>(xh, xl, dst, k);
  }
  template <int ES_IN = 1, int ES_OUT = 1>
  __device__ __forceinline__ void apply(const V* src, V* dst) const {
    if constexpr (NE_IN == 6 && ROWS_OUT == 3) {
      // two-row in, full out (never in place): rows 0 and 1 are split once and serve both their
      // own outputs and the rebuild of row 2 (the same operations as apply_row, so the same bits)
      float uh[6], ul[6], vh[6], vl[6], wh[6], wl[6];
      split_row<ES_IN>(src, 0, uh, ul);
      split_row<ES_IN>(src, 1, vh, vl);
      rebuild_row2_pair(uh, ul, vh, vl, one, wh, wl);
      row_out<ES_OUT>(uh, ul, dst, 0);
      row_out<ES_OUT>(vh, vl, dst, 1);
      row_out<ES_OUT>(wh, wl, dst, 2);
    } else {
#pragma unroll
      for (int k = 0; k < ROWS_OUT; ++k) apply_row<ES_IN, ES_OUT>(src, dst, k);
    }
  }
};


// The adjacent products in FP32-pair arithmetic (FP64 storage, FP64-accurate results):
// a^dagger b, whose output row k is the product's row routine applied to column k of a
// conjugated (the imaginary parts' splits change sign, exactly), with the same b pairs.
struct PairAnOp {
  using V = double2;
  using BArg = double;
  static constexpr int kFixCols = 0, kMinCtas = 0;
  static constexpr int kNeIn = 9, kNeOut = 9;
  static constexpr bool kRowSplit = false;  // row k of a^dagger b reads column k of a
  PairF64Op<9, 3> pair;                     // b as FP32 pairs and the row routine
  __device__ __forceinline__ void begin_tile(int) {}
  __device__ __forceinline__ void set_unit(float u) { pair.set_unit(u); }
  __device__ __forceinline__ void init(const double* bj, int w) { pair.init(bj, w); }
  template <int ES_IN = 1, int ES_OUT = 1>
  __device__ __forceinline__ void apply(const V* src, V* dst) const {
    double2 a[9];  // all of a first: the output may overwrite it (in place)
#pragma unroll
    for (int e = 0; e < 9; ++e) a[e] = src[e * ES_IN];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      float xh[6], xl[6];  // conj(a[m][k]), terms 2m: re, 2m+1: im
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        const FF re = split_f64(a[3 * m + k].x), im = split_f64(a[3 * m + k].y);
        xh[2 * m] = re.h;
        xl[2 * m] = re.l;
        xh[2 * m + 1] = -im.h;
        xl[2 * m + 1] = -im.l;
      }
      pair.template row_out<ES_OUT>(xh, xl, dst, k);
    }
  }
};

// a v and a^dagger v in FP32-pair arithmetic: each output element is one 6-term pair dot product
// of row k of a (ADJ: column k, conjugated) with v[j] held as FP32 pairs.
template <bool ADJ>
struct PairMatVecOp {
  using V = double2;
  using BArg = double;
  static constexpr int kFixCols = 0, kMinCtas = 0;
  static constexpr int kNeIn = 9, kNeOut = 3;
  static constexpr bool kRowSplit = false;  // one output vector per link
  float2 ya[3], yb[3], yla[3], ylb[3];      // v[m]: (re, im), (-im, re), and their low parts
  float2 one;
  __device__ __forceinline__ void begin_tile(int) {}
  __device__ __forceinline__ void set_unit(float u) { one = make_float2(u, u); }
  __device__ __forceinline__ void init(const double* vj, int) {
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const double r = vj[2 * m], i = vj[2 * m + 1];
      const float rh = __double2float_rn(r), ih = __double2float_rn(i);
      const float rl = __double2float_rn(r - (double)rh), il = __double2float_rn(i - (double)ih);
      ya[m] = make_float2(rh, ih);
      yb[m] = make_float2(-ih, rh);
      yla[m] = make_float2(rl, il);
      ylb[m] = make_float2(-il, rl);
    }
  }
  template <int ES_IN = 1, int ES_OUT = 1>
  __device__ __forceinline__ void apply(const V* src, V* dst) const {
    const float2 yh[6] = {ya[0], yb[0], ya[1], yb[1], ya[2], yb[2]};
    const float2 yl[6] = {yla[0], ylb[0], yla[1], ylb[1], yla[2], ylb[2]};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      float xh[6], xl[6];
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        const double2 v = src[(ADJ ? 3 * m + k : 3 * k + m) * ES_IN];
        const FF re = split_f64(v.x), im = split_f64(v.y);
        xh[2 * m] = re.h;
        xl[2 * m] = re.l;
        xh[2 * m + 1] = ADJ ? -im.h : im.h;
        xl[2 * m + 1] = ADJ ? -im.l : im.l;
      }
      dst[k * ES_OUT] = dot6_pair2(xh, xl, yh, yl, one);
    }
  }
};

// HYBRID: per tile, warp w uses the FP64 pipe (NATIVE) when (tile + w) % period == 0 and FP32
// pairs otherwise, period = warps / native_warps. The native work rotates over all warps, so it
// is spread over every SM sub-partition's FP64 unit. Each thread keeps both forms of its b[j].
template <int NE_IN, int ROWS_OUT>
struct HybridF64Op {
  using V = double2;
  using BArg = double;
  static constexpr int kFixCols = 3, kMinCtas = 0;
  static constexpr int kNeIn = NE_IN, kNeOut = 3 * ROWS_OUT;
  static constexpr bool kRowSplit = true;
  NativeOp<kF64, NE_IN, ROWS_OUT> nat;
  PairF64Op<NE_IN, ROWS_OUT> pair;
  int period;  // 0: never native
  bool native;
  __device__ __forceinline__ void init(const double* bj, int native_warps) {
    nat.init(bj, 0);
    pair.init(bj, 0);
    const int warps = (int)(blockDim.x >> 5);
    period = native_warps > 0 ? max(1, warps / native_warps) : 0;
    native = false;
  }
  __device__ __forceinline__ void begin_tile(int k) {
    native = period > 0 && ((k + (int)(threadIdx.x >> 5)) % period) == 0;
  }
  __device__ __forceinline__ void set_unit(float u) { pair.set_unit(u); }
  __device__ __forceinline__ void set_fixed(const FixedMat& f, const void* fx, const void* mag, int j) {
    nat.set_fixed(f, fx, mag, j);
  }
  template <int ES_IN = 1, int ES_OUT = 1>
  __device__ __forceinline__ void apply(const V* src, V* dst) const {
    if (native) nat.template apply<ES_IN, ES_OUT>(src, dst);
    else pair.template apply<ES_IN, ES_OUT>(src, dst);
  }
  template <int ES_IN = 1, int ES_OUT = 1>
  __device__ __forceinline__ void apply_row(const V* src, V* dst, int k) const {
    if (native) nat.template apply_row<ES_IN, ES_OUT>(src, dst, k);
    else pair.template apply_row<ES_IN, ES_OUT>(src, dst, k);
  }
};

}  // namespace su3
