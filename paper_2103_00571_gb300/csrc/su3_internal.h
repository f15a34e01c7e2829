// Host-side internals shared by the libsu3 translation units (not part of the C ABI).
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stddef.h>
#include <stdint.h>

#include <string>

#include "su3.h"

namespace su3 {

// Device status word bits (the handle's status word; su3_sync reads and clears it).
enum : unsigned { kDevErrTimeout = 1u };

// A fully validated form: what a kernel instantiation is selected by.
struct Form {
  int dtype;      // su3_dtype
  int repr_in;    // su3_repr of a
  int repr_out;   // su3_repr of c
  int layout;     // su3_layout
  int arith;      // su3_arith
  int64_t n_sites;
  int64_t a_stride;  // AOS: bytes between sites of a (resolved, never 0)
  int64_t c_stride;  // AOS: bytes between sites of c
};

struct LaunchCfg {
  int block;
  int tile_sites;
  int stages;
  int ctas_per_sm;
  int native_permille;  // HYBRID: share of tiles on the FP64 pipe
  int threads_per_link = 1;  // AOS: 1, or 3 = one thread per output row (2 per link for two-row output)
  bool is_default = false;   // not set by the caller: the launch may change threads_per_link and widen block
};

// Everything a launcher needs from the handle.
struct LaunchCtx {
  cudaStream_t stream;
  unsigned* status;  // device status word
  int num_sms;
  int smem_per_sm = 0;    // shared memory per SM in bytes (0: unknown, no fitting)
  int smem_reserved = 0;  // shared memory the system reserves per CTA
  int64_t* launches;  // incremented per kernel launch
  std::string* err;
};

inline int real_bytes(int dtype) { return dtype == SU3_F64 ? 8 : dtype == SU3_F32 ? 4 : 2; }
inline int n_elem(int repr) { return repr == SU3_REPR_FULL18 ? 9 : 6; }
inline int64_t link_bytes(int dtype, int repr) { return (int64_t)n_elem(repr) * 2 * real_bytes(dtype); }

// Default launch configuration of a form (used until the autotuner sets one).
LaunchCfg default_cfg(const Form& f);
// The same for su3_mult_op's a^dagger b and su3_mat_vec.
LaunchCfg default_adjacent_cfg(const Form& f);
// What su3_set_launch_cfg fills a partial configuration up with: independent of the array's size, and
// shallow enough that any one field can be set beside it.
LaunchCfg general_cfg(const Form& f);

// An array with fewer tiles of *ts sites than SMs: narrower tiles (multiples of `quantum` sites), in
// CTAs just wide enough for them, spread it over more SMs, so that its warps do not queue on a few SMs'
// pipes. `rows`: output rows per link that may have a thread each. `split` (FP64 in fixed point): by
// default one thread per output row while a tile's rows fit one CTA, since a whole link is a chain of
// three rows (per launch at 64 sites 5.8 -> 3.7 us, 1,000 sites 5.9 -> 4.3, 2,000 sites 5.3 -> 4.7; with
// more rows than threads, at 4,096 sites, 5.5 either way). A shape that the caller set keeps its
// threads per link and at most its block. Every launch shape gives the same bits.
inline void spread_small(LaunchCfg* cfg, long long* ts, long long n_sites, int num_sms, long long quantum, int rows,
                         bool split) {
  if (n_sites <= 0 || (n_sites + *ts - 1) / *ts >= num_sms) return;
  long long t = (n_sites + num_sms - 1) / num_sms;
  t = (t + quantum - 1) / quantum * quantum;
  if (t < quantum) t = quantum;
  if (t >= *ts) return;
  *ts = t;
  split = split && cfg->is_default && t * 4 * rows <= 256;
  if (split) cfg->threads_per_link = 3;
  const long long items = t * 4 * (cfg->threads_per_link == 1 ? 1 : rows);
  const long long need = items < 32 ? 32 : (items + 31) / 32 * 32, limit = split ? 256 : cfg->block;
  cfg->block = (int)(need < limit ? need : limit);
}

// HYBRID: warps per CTA on the FP64 pipe, the nearest to native_permille of the CTA's warps.
inline int native_warps(const Form& f, const LaunchCfg& cfg) {
  if (f.arith != SU3_ARITH_HYBRID) return 0;
  const int warps = cfg.block / 32;
  const int n = (warps * cfg.native_permille + 500) / 1000;
  return n < warps ? n : warps;
}

// c = a x b over one lattice (the streaming kernels). b is FP64 on the host.
su3_status launch_mult(const Form& f, const LaunchCfg& cfg, const void* a, const double* b, void* c,
                       const LaunchCtx& ctx);

// c = a x b with a and c in host memory the device can address (pinned, or any host memory on a
// device with pageable-memory access): the kernel streams both over the host link itself.
su3_status launch_mult_host_direct(const Form& f, const LaunchCfg& cfg, const void* a, const double* b, void* c,
                                   const LaunchCtx& ctx);

// a^dagger b (which 0), a v (1), a^dagger v (2): AOS FULL18 NATIVE; v[j] at bv[18*j .. 18*j+5].
su3_status launch_adjacent(int which, const Form& f, const LaunchCfg& cfg, const void* a, const double* bv, void* c,
                           const LaunchCtx& ctx);

// One CTA whose bounded mbarrier wait runs out after limit_ms (failure-path self test).
su3_status launch_selftest_wait(int limit_ms, const LaunchCtx& ctx);

// Packed FP64 AOS <-> the form's storage.
su3_status launch_pack(const Form& dst, const double* src, void* dst_dev, const LaunchCtx& ctx);
su3_status launch_unpack(const Form& src, const void* src_dev, double* dst, const LaunchCtx& ctx);

// ---- b of the FP64 product in fixed point (the device side is fixed_row in su3_device.cuh) -------

// Constants of the fixed-point rows that must be unknown to the compiler. With them known it turns
// products by -x into negated multiplies and splits multiply-accumulates into a product and 64-bit
// adds (19 more integer adds per output: 4,142 against 4,732 GB/s at 2^21 sites).
struct FixedConst {
  int zero;
  unsigned lead;           // 2^20: the implicit leading bit of an FP64 mantissa, in its high word
  long long hbias, xbias;  // start values of the accumulators
};
inline FixedConst fixed_const() {
  return FixedConst{0, 1u << 20, -(1ll << 32), (long long)((1ull << 63) + (1ull << 31))};
}

// Biased exponents of a row's largest |real| that the form takes: 2^-723 <= |a| < 2^677.
constexpr unsigned kFixExpMin = 300, kFixExpRange = 1400;
// Least sum of the |a||b| of an output real's six terms, in 2^-13 of full scale: 1/16 (fixed_row).
constexpr unsigned kFixMinSum = 512;
// Words per direction of fix_b's magnitudes: 6, padded to 16-byte words.
constexpr int kFixMags = 8;

// Element e of b[j] as two signed 32-bit limbs for re and two for im, fx[j][e] = (re_hi, re_lo,
// im_hi, im_lo), value (hi * 2^32 + lo) * 2^(eb[j] - 61) with |b[j]| < 2^eb[j]. `range`: the number of
// exponents of a row's largest real that the fixed-point form takes, 0 when b does not suit it.
struct FixedMat {
  alignas(16) int fx[4][9][4];
  unsigned mag[4][kFixMags];
  int eb[4];
  unsigned range;
  FixedConst k;
};

// Fills fx, mag (column l: |re| and |im| of rows 0 and 1 in bytes of 2^(eb - 8), then of row 2) and eb
// from b (COLS 3: [j][row][col]; 1: one colour vector per j at the start of b's j-th 18 reals). Returns
// whether b suits the form: every value finite, the largest of each matrix within 1e-30 .. 1e30, and
// in every column at least three of the six reals within 2^-5 of that largest, since with fewer most
// output reals would not pass fixed_row's gate. 99.9 % of sets of four random SU(3) matrices do; when one
// matrix does not, every row takes FP64 FMAs.
template <int COLS>
inline bool fix_b(const double* b, int (*fx)[9][4], unsigned (*mag)[kFixMags], int* eb) {
  for (int j = 0; j < 4; ++j) {
    const double* m = b + 18 * j;
    double top = 0;
    for (int q = 0; q < 6 * COLS; ++q) {
      if (!(fabs(m[q]) <= 1e30)) return false;  // also NaN
      top = fabs(m[q]) > top ? fabs(m[q]) : top;
    }
    if (top < 1e-30) return false;
    frexp(top, &eb[j]);  // top < 2^eb
    const double large = ldexp(1.0, eb[j] - 5);
    for (int l = 0; l < COLS; ++l) {
      int n = 0;
      for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 2; ++c) n += fabs(m[2 * (COLS * r + l) + c]) >= large;
      if (n < 3) return false;
    }
    const double scale = ldexp(1.0, 61 - eb[j]), bytes = ldexp(1.0, 8 - eb[j]);
    for (int q = 0; q < 6 * COLS; ++q) {
      const long long v = (long long)rint(m[q] * scale);
      const int lo = (int)(unsigned)((unsigned long long)v & 0xffffffffull);
      fx[j][q >> 1][2 * (q & 1)] = (int)((v - lo) >> 32);
      fx[j][q >> 1][2 * (q & 1) + 1] = lo;
    }
    for (int l = 0; l < COLS; ++l) {
      unsigned w[3];  // an element's |re| and |im| as bytes, rounded down
      for (int r = 0; r < 3; ++r)
        w[r] = (unsigned)(fabs(m[2 * (COLS * r + l)]) * bytes) | (unsigned)(fabs(m[2 * (COLS * r + l) + 1]) * bytes) << 8;
      mag[j][2 * l] = w[0] | w[1] << 16;
      mag[j][2 * l + 1] = w[2];
    }
  }
  return true;
}

// Device descriptor of one lattice in a batched launch.
struct BatchDesc {
  const void* a;
  void* c;
  long long n_sites;
  int dtype;           // SU3_F64 or SU3_F32
  int first_tile;      // exclusive prefix sum of tile counts
  short arith;         // SU3_ARITH_NATIVE, or SU3_ARITH_F32PAIR for F64 lattices
  short fixed;         // F64 NATIVE: whether b suits the fixed-point form (fix_b)
  signed char eb[4];   // F64 NATIVE: exponents of the four matrices (fix_b)
  double b[72];        // FP64 b (F32 lattices round it in the kernel)
  union {
    alignas(16) float bpair[144];  // F32PAIR: b[j][e] split as (re_hi, im_hi, re_lo, im_lo), [j][e][4]
    int bfix[4][9][4];             // F64 NATIVE: b in fixed point (fix_b)
  };
  unsigned bmag[4][kFixMags];  // F64 NATIVE: fix_b's magnitudes
};
static_assert(offsetof(BatchDesc, bfix) % 16 == 0 && offsetof(BatchDesc, bmag) % 16 == 0 && sizeof(BatchDesc) % 16 == 0,
              "bfix and bmag are read as 16-byte words");

// Fills BatchDesc::bpair from the FP64 b (hi = b rounded to FP32, lo = the rest rounded to FP32).
inline void split_b_pairs(const double* b, float* out) {
  for (int q = 0; q < 36; ++q) {
    const double r = b[2 * q], i = b[2 * q + 1];
    const float rh = (float)r, ih = (float)i;
    out[4 * q] = rh;
    out[4 * q + 1] = ih;
    out[4 * q + 2] = (float)(r - (double)rh);
    out[4 * q + 3] = (float)(i - (double)ih);
  }
}

// Fills the descriptor's arithmetic and b from an item's.
inline void fill_batch_b(BatchDesc* o, int dtype, int arith, const double* b) {
  o->arith = (short)arith;
  o->fixed = 0;
  for (int j = 0; j < 4; ++j) o->eb[j] = 0;
  for (int i = 0; i < 72; ++i) o->b[i] = b[i];
  for (int i = 0; i < 4 * kFixMags; ++i) (&o->bmag[0][0])[i] = 0;
  if (dtype == SU3_F64 && arith == SU3_ARITH_NATIVE) {
    int eb[4] = {0, 0, 0, 0};
    for (int i = 0; i < 144; ++i) o->bpair[i] = 0;
    o->fixed = fix_b<3>(b, o->bfix, o->bmag, eb) ? 1 : 0;
    for (int j = 0; j < 4; ++j) o->eb[j] = (signed char)eb[j];  // |eb| <= 101
  } else {
    split_b_pairs(b, o->bpair);
  }
}

struct BatchCfg {
  int block;
  int tile_sites;
  int stages;
  int ctas_per_sm;
  int threads_per_link = 1;  // 1, or 3: one thread per output row
};

BatchCfg default_batch_cfg();
// Tiles are sized in bytes: tile_sites FP64 sites, or 2 * tile_sites FP32 sites (576 B vs 288 B each).
__host__ __device__ inline int batch_tile_sites(int dtype, int tile_sites) { return dtype == SU3_F64 ? tile_sites : 2 * tile_sites; }
int batch_tile_count(long long n_sites, int dtype, int tile_sites);

// Validates a batched configuration and sets the kernel's shared-memory attribute.
su3_status prepare_batched(const BatchCfg& cfg, std::string* err);

// One persistent launch over `n` lattices whose descriptors are already in device memory.
su3_status launch_batched(const BatchDesc* descs_dev, int n, int total_tiles, const BatchCfg& cfg,
                          const LaunchCtx& ctx);

}  // namespace su3
