// FP64 GEMM tasks (energies, environments, fused operators, truncations and
// sigma products of the FP64 path).
//
// GB300's FP64 pipe issues two fused multiply-adds per clock and SM (1.25
// TFLOP/s for the chip), about 1/1800 of its BF16 tensor rate.  So large tasks
// run as exact integer products on the tensor cores (Ozaki's splitting): every
// row of an operand is scaled by a power of two to 62-bit integers, each
// integer is cut into eight balanced digits of eight bits, digits are exact in
// FP16, and products of digit planes accumulate exactly in FP32 (at most 8 x
// 128 products of 2^14).  The 36 plane pairs whose weight is at least 2^-56 of
// the largest are formed; pairs of equal weight share one accumulator, the
// accumulators are combined in integers and rounded to FP64 once per 1024 K
// values.  What is lost is the cut of an operand (below 2^-61 of its row's
// largest value) and the pairs left out (at most 2^-57.2 of the product of the
// two rows' largest values per term, typically 2^-60).  Both go with the rows'
// largest values, not with the terms: where the large values of two rows meet
// the small ones of the other, an output's error would pass that of a chain of
// FP64 multiply-adds.  So every output is checked against a lower bound of sum
// |x y| (sum_magnitudes), and those that might pass the chain's bound, n 2^-53
// sum |x y|, are summed in FP64 instead (gemm_f64_again_kernel).  Without the check
// operands graded over 2^40 in opposite directions are off by 1e-8 of sum |x y|.
// Few outputs of states with even spectra are in doubt (0 to 13 %), but most of
// those of large converged states, whose rows are graded by their Schmidt values:
// there the FP64 pipe bounds the product as it did before (a window of four
// positions at M1 = 2000: 24 s; 6.5 s unchecked; 40 to 45 s on the FP64 pipe alone).
//
// Tasks of few multiply-adds run on the FP64 pipe (gemm_f64_pipe_kernel).
//
// Measured against the 64 x 64 FP64-pipe tiles that did all of this before
// (3-band model, middle position, M1 = 500): sigma phases 27.0 + 28.8 ms ->
// 2.8 + 3.0 ms (2.4 + 2.8 without the check), error against 64-bit contraction
// 2.4e-15 -> 1.0e-15; all products of the energies at M1 = 400, 790 ms -> 55 ms.
// A tile's time is its chain (loads, cutting, products, check, drain, conversion,
// stores), of which the integer pipe carries most; the tensor pipe is busy a
// tenth of it.
#include <algorithm>
#include <atomic>
#include <vector>
#include <cstring>
#include <type_traits>

#include "engine.hpp"
#include "tcgen05.cuh"

namespace mpslcc {

namespace {

constexpr int TM = 128;                // rows of X in a tensor-core tile
constexpr int KB = 1024;               // K values per scaling block
constexpr int KS = 32;                 // K values per step (64 bytes of FP16)
constexpr int CHUNK = 4;               // steps between two drains: 128 K values
constexpr int PLANES = 8;
constexpr int MAX_DEV = 128;
constexpr uint32_t ENOUGH = 1156, ENOUGH_B = 255;   // see sum_magnitudes
constexpr int ZERO_ROW = 63;           // exponent in the scale of a row of zeros (others: 64 and more)

// Two shapes.  TN = 64, one CTA of 16 warps per SM: two step buffers, so that
// digits are cut while the previous step multiplies; 8 x 64 accumulator columns
// take all of tensor memory.  TN = 32, two CTAs of 8 warps per SM, one step
// buffer each: for short sums, whose time is the chain load - cut - multiply -
// drain - write of a tile, one CTA's chain fills the other's gaps.
template <int TN_> struct F64Cfg {
  static constexpr int TN = TN_;
  static constexpr int WARPS = TN == 64 ? 16 : 8, THREADS = 32 * WARPS, CTAS = TN == 64 ? 1 : 2;
  static constexpr int NBUF = TN == 64 ? 2 : 1;
  static constexpr int ROW = 64 * NBUF;                        // bytes of a plane's row
  static constexpr int XPLANE = TM * ROW, YPLANE = TN * ROW;
  static constexpr int OPER = PLANES * (XPLANE + YPLANE);      // 192 or 80 KB
  static constexpr int XU = 16 / WARPS;                        // loader units of X per warp
  static constexpr int YU0 = WARPS - TN / 8;                   // first warp that loads Y
  // Leading magnitudes, a byte each: MW steps, 16-byte groups of a row swizzled.
  // (Four steps at TN = 32 would take the chip from 196 to 228 KB of shared
  // memory per SM, and the loads' share of L1 from 60 to 28 KB: 9.7 instead of
  // 8.7 ms for a sigma of the 3-band model at M1 = 500.)
  static constexpr int MW = TN == 64 ? 4 : 2, MROW = KS * MW;
  static constexpr int MAGS = (TM + TN) * MROW;
  static constexpr int ALIGN = 8 * ROW;                        // of the planes: a swizzle atom
};
template <class F> __device__ __forceinline__ int mag_at(int row, int group) {
  return row * F::MROW + ((group ^ (F::MW == 4 ? row & 7 : row >> 1 & 3)) << 4);
}
// Tiles with outputs in doubt (see the head of the file), and for each of a tile's
// blocks of 1024 K values a bit per output, 16 columns of a row a word.
struct F64Doubt {
  int* count;
  long long* rec;
  uint16_t* mask;
  int cap, blocks;
};
constexpr size_t F64_SCRATCH_HEAD = 256;   // two counts
inline size_t f64_record_bytes(int tn, int blocks) { return sizeof(long long) + (size_t)blocks * TM * tn / 8; }
// Tiles of one launch where there are more: 64 MB of records, and no less than some
// milliseconds of products.
inline long long f64_launch_tiles(int tn, int blocks) {
  return (long long)((64u << 20) / f64_record_bytes(tn, blocks));
}
constexpr int F64_MAX_BLOCKS = 32;         // outputs in doubt of longer sums are summed in place

struct F64Slot {
  F64Task t;
  int b, ks, ix, iy;
};
template <bool MULTI> constexpr int TAB = MULTI ? KB : KS * CHUNK;   // K values of a block
template <class F, bool MULTI> constexpr int f64_smem() {
  return F::OPER + F::ALIGN + F::MAGS + TAB<MULTI> * 4 + (TM + F::TN) * 4 + 64 + 2 * (int)sizeof(F64Slot) +
         (TM + F::TN) * 8;
}
// see F64Cfg
static_assert(2 * (f64_smem<F64Cfg<32>, true>() + 1024) <= 196 * 1024, "two CTAs in 196 KB");

struct F64Tile { int b, ks, ix, iy; };
__device__ __forceinline__ F64Tile tile_of(const F64Task& T, long long tile) {
  const long long local = tile - T.tile0;
  const long long txy = (long long)T.tx * T.ty, per_b = txy * T.ksplit;
  F64Tile t;
  unsigned q;
  if (local < (1LL << 31) && per_b < (1LL << 31)) {   // 64-bit divisions cost hundreds of instructions
    t.b = (int)((unsigned)local / (unsigned)per_b);
    const unsigned r = (unsigned)local - (unsigned)t.b * (unsigned)per_b;
    t.ks = (int)(r / (unsigned)txy);
    q = r - (unsigned)t.ks * (unsigned)txy;
  } else {
    t.b = (int)(local / per_b);
    const long long r = local - (long long)t.b * per_b;
    t.ks = (int)(r / txy);
    q = (unsigned)(r - (long long)t.ks * txy);
  }
  t.ix = (int)(q / (unsigned)T.ty);
  t.iy = (int)(q - (unsigned)t.ix * (unsigned)T.ty);
  return t;
}

// Task of `tile`, found by a whole warp from task `prev` on (a CTA's tiles
// ascend): the next 32 tasks, then 32-fold steps.
__device__ __forceinline__ int warp_find(const F64Task* t, int n, long long tile, int prev) {
  const int lane = threadIdx.x & 31;
  int lo = prev, hi = min(n, prev + 33), step = 1;   // t[lo] starts at or before the tile
  for (;;) {
    const int i = lo + (lane + 1) * step;
    const int c = __popc(__ballot_sync(0xffffffffu, i < hi && t[i].tile0 <= tile));
    lo += c * step;
    if (step == 1 && (c < 32 || lo + 1 >= n)) return lo;
    hi = step == 1 ? n : min(hi, lo + step);
    step = (hi - lo + 31) / 32;
    if (step < 1) step = 1;
  }
}
// Fills a slot with tile's task and coordinates (a whole warp); returns the task.
__device__ __forceinline__ int fetch_slot(F64Slot* s, const F64Task* t, int n, long long tile, int prev) {
  const int lane = threadIdx.x & 31;
  const int i = warp_find(t, n, tile, prev);
  static_assert(sizeof(F64Task) % 8 == 0 && sizeof(F64Task) <= 512, "task copy");
#pragma unroll
  for (int w = lane; w < (int)(sizeof(F64Task) / 8); w += 32) ((long long*)&s->t)[w] = ((const long long*)(t + i))[w];
  __syncwarp();
  if (lane == 0) {
    const F64Tile c = tile_of(s->t, tile);
    s->b = c.b; s->ks = c.ks; s->ix = c.ix; s->iy = c.iy;
  }
  return i;
}

// Offset of row i of a folded operand: rows run over (batch entry, row).
__device__ __forceinline__ long long row_off(int i, int inner, long long is, long long bs) {
  const int b = i / inner;
  return (long long)b * bs + (long long)(i - b * inner) * is;
}

// Operand column of summed index v (K runs, or v itself).
__device__ __forceinline__ int k_col(const F64Task& T, int v) {
  if (!T.kr) return v;
  int lo = 0, hi = T.nkr - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(T.kr + 2 * mid + 1) <= v) lo = mid;
    else hi = mid - 1;
  }
  return __ldg(T.kr + 2 * lo) + (v - __ldg(T.kr + 2 * lo + 1));
}

// How a tile is written: C = alpha v + beta C.  The cases that need the FP64
// pipe are told apart once per tile (a comparison of doubles runs there too,
// and two per element took 20 % of the tensor-core kernel's time).
enum { PUT_SCALE = 1, PUT_BETA = 2, PUT_ADD = 4 };
__device__ __forceinline__ int put_mode(const F64Task& T, bool first) {
  return (T.alpha != 1.0 ? PUT_SCALE : 0) | (!first ? PUT_ADD : (T.beta != 0.0 ? PUT_BETA : 0));
}
// of a sum that joins what lies there
__device__ __forceinline__ int sum_mode(const F64Task& T) { return (T.alpha != 1.0 ? PUT_SCALE : 0) | PUT_ADD; }
__device__ __forceinline__ void put(const F64Task& T, int mode, double* c, double v) {
  if (mode) {
    if (mode & PUT_SCALE) v *= T.alpha;
    if (mode & PUT_ADD) v += *c;
    else if (mode & PUT_BETA) v += T.beta * (*c);
  }
  *c = v;
}

// ---------------------------------------------------------------------------
// tensor-core kernel
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tmem_ld2(uint32_t taddr, uint32_t* v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(v[0]), "=r"(v[1]) : "r"(taddr));
}

// One loader unit: up to 32 x 8 or 8 x 32 elements of an operand tile; a
// thread holds eight K values of one row's step: q, q + 2, ..., q + 14 for q =
// 0, 1, and 16 more for q = 2, 3 (so that a step of up to 16 values has an
// empty second half).
struct Unit {
  const double* p;
  int row, q;
  bool ok;
};

// Values below nk of the unit's row; tab holds the operand columns, or is null
// where they are base, base + 1, ...
__device__ __forceinline__ void load_unit(const Unit& u, long long ks, const int* tab, int base, int nk,
                                          double (&v)[8]) {
  const int q0 = u.q < 2 ? u.q : 14 + u.q;
  const int left = u.ok ? nk - q0 : 0;
  if (tab) {
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = 2 * j < left ? __ldg(u.p + (long long)tab[q0 + 2 * j] * ks) : 0.0;
  } else {
    const double* p = u.p + (base + q0) * ks;
    const long long st = 2 * ks;
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = 2 * j < left ? __ldg(p + j * st) : 0.0;
  }
}

// Largest magnitude of the unit's values as high words; a value whose high
// word is zero but that is not zero counts as the smallest subnormal.
__device__ __forceinline__ uint32_t unit_max(const double (&v)[8], uint32_t m) {
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint32_t h = (uint32_t)__double2hiint(v[j]) & 0x7fffffffu;
    m = max(m, h | (__double2loint(v[j]) != 0 ? 1u : 0u));
  }
  return m;
}

// v as an integer of 62 bits relative to the row exponent (cut towards zero:
// 2^-61 of the row's largest value at most), offset by 128 in every digit:
// byte i of the result is digit i plus 128.  The top byte of `mag` gets the
// integer's magnitude over 2^54, cut.
__device__ __forceinline__ unsigned long long digits(double v, int emax, uint32_t& mag) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  const int d = min(emax - (int)((hi >> 20) & 0x7ffu), 63);   // 63 clears zeros too: emax >= 63
  unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
  m = (m << 9) >> d;
  mag = (uint32_t)(m >> 32) << 2;
  const long long s = (long long)((int)hi >> 31);
  return (m ^ (unsigned long long)s) + (0x8080808080808080ull - (unsigned long long)s);
}

// Exponent of a row scale (exponent of the row's largest value, times two, plus
// one if its values are taken 2^512-fold).
__device__ __forceinline__ int scale_exp(int scale) { return (scale >> 1) - ((scale & 1) << 9); }

// Writes the unit's eight values as 16 bytes in each digit plane: rows of two
// steps with 128-byte swizzle (16-byte chunk xor row mod 8), or rows of one
// step with 64-byte swizzle (chunk xor row / 2 mod 4).  A digit's byte under
// the FP16 exponent of 1024 is 1024 + digit + 128; one subtraction leaves it.
// (Bound by the integer pipe: two byte permutations per pair of digits, where
// BF16's shorter significand needed four operations.)
template <class F>
__device__ __forceinline__ void store_unit(const Unit& u, double (&v)[8], int scale, uint8_t* planes, int plane,
                                           int half, uint8_t* mags, int mrow, int step) {
  const int emax = scale >> 1;
  if (scale & 1) {
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] *= 0x1p512;
  }
  uint32_t t0[8], t1[8], mg[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const unsigned long long t = digits(v[j], emax, mg[j]);
    t0[j] = (uint32_t)t;
    t1[j] = (uint32_t)(t >> 32);
  }
  auto tops = [](uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    return __byte_perm(__byte_perm(a, b, 0x0073), __byte_perm(c, d, 0x0073), 0x5410);
  };
  *reinterpret_cast<uint2*>(mags + mag_at<F>(mrow + u.row, 2 * (step & (F::MW - 1)) + (u.q >> 1)) + (u.q & 1) * 8) =
      make_uint2(tops(mg[0], mg[1], mg[2], mg[3]), tops(mg[4], mg[5], mg[6], mg[7]));
  uint8_t* dst = F::NBUF == 2 ? planes + u.row * 128 + (((half * 4 + u.q) ^ (u.row & 7)) << 4)
                           : planes + u.row * 64 + ((u.q ^ ((u.row >> 1) & 3)) << 4);
#pragma unroll
  for (int p = 0; p < PLANES; p += 2) {
    // planes p and p + 1 (plane 0 the most significant) are bytes s + 1 and s
    // of the same word
    const int s = (PLANES - 2 - p) & 3;
    uint32_t w0[4], w1[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t a = p < 4 ? t1[2 * j] : t0[2 * j], b = p < 4 ? t1[2 * j + 1] : t0[2 * j + 1];
      const uint32_t x = __byte_perm(a, b, s | (s + 4) << 4 | (s + 1) << 8 | (s + 5) << 12);   // a_s b_s a_s+1 b_s+1
      const uint32_t lo = __byte_perm(x, 0x64646464u, 0x4140), hi = __byte_perm(x, 0x64646464u, 0x4342);
      asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(w1[j]) : "r"(lo), "r"(0x64806480u));
      asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(w0[j]) : "r"(hi), "r"(0x64806480u));
    }
    *reinterpret_cast<uint4*>(dst + p * plane) = make_uint4(w0[0], w0[1], w0[2], w0[3]);
    *reinterpret_cast<uint4*>(dst + (p + 1) * plane) = make_uint4(w1[0], w1[1], w1[2], w1[3]);
  }
}

// Whether a digit product may stand.  With |X|, |Y| < 2^62 a term loses less
// than 2 x 2^62 to the cut of its operands and 7.03 x 2^62 to the plane pairs
// left out, in units of X Y, so the error of an output is below that of a chain
// of n FP64 multiply-adds, n 2^-53 sum |x y|, if sum |X Y| >= 9.03 x 2^115.  The
// leading eight bits of the operands bound that sum from below: sum (|X| >>
// 54)(|Y| >> 54) >= 1156 = 9.03 x 2^7 will do.  Where x and y have their large
// values at different k it may fail, and the output is summed again in FP64
// (gemm_f64_again_kernel).  A thread adds up its row's outputs of 16 columns, four
// at a time, over `steps` of a window and stops with its warp once all have enough
// (mostly after 32 values); `sums` holds a byte per output, its sum / 16 so far or
// ENOUGH_B.
template <class F>
__device__ __forceinline__ void sum_magnitudes(const uint8_t* mags, int row, int col0, int steps, uint32_t (&sums)[4]) {
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    if (!__any_sync(0xffffffffu, sums[g] != ~0u)) continue;
    uint32_t acc[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const uint32_t b = sums[g] >> (8 * c) & 255u;
      acc[c] = b == ENOUGH_B ? ENOUGH : b << 4;
    }
#pragma unroll 1
    for (int st = 0; st < steps; ++st) {
#pragma unroll
      for (int w = 2 * st; w < 2 * st + 2; ++w) {
        const uint4 a = *reinterpret_cast<const uint4*>(mags + mag_at<F>(row, w));
#pragma unroll
        for (int c = 0; c < 4; ++c) {   // rows TM + col0 + ...: a multiple of 16
          const uint4 b = *reinterpret_cast<const uint4*>(mags + (TM + col0) * F::MROW + mag_at<F>(4 * g + c, w));
          acc[c] = __dp4a(a.w, b.w, __dp4a(a.z, b.z, __dp4a(a.y, b.y, __dp4a(a.x, b.x, acc[c]))));
        }
      }
      if (__all_sync(0xffffffffu, min(min(acc[0], acc[1]), min(acc[2], acc[3])) >= ENOUGH)) break;
    }
    sums[g] = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) sums[g] |= (acc[c] >= ENOUGH ? ENOUGH_B : acc[c] >> 4) << (8 * c);
  }
}

// hi 2^32 + lo, in units of 2^(eab - 2112), as FP64 rounded to nearest.
__device__ __forceinline__ double to_f64(long long hi, long long lo, int eab) {
  const long long h = hi + (lo >> 32);
  uint32_t a2 = (uint32_t)((unsigned long long)h >> 32), a1 = (uint32_t)h, a0 = (uint32_t)lo;
  const uint32_t neg = (uint32_t)((int)a2 >> 31);
  // magnitude of the 96-bit value
  asm("xor.b32 %0, %0, %3;\n xor.b32 %1, %1, %3;\n xor.b32 %2, %2, %3;\n"
      "sub.cc.u32 %0, %0, %3;\n subc.cc.u32 %1, %1, %3;\n subc.u32 %2, %2, %3;"
      : "+r"(a0), "+r"(a1), "+r"(a2)
      : "r"(neg));
  int e = eab + 95 - 1089;
  if (a2 == 0) {
    a2 = a1; a1 = a0; a0 = 0;
    e -= 32;
    if (a2 == 0) {
      a2 = a1; a1 = 0;
      e -= 32;
      if (a2 == 0) return 0.0;
    }
  }
  const int lz = __clz((int)a2);
  e -= lz;
  const uint32_t m1 = __funnelshift_l(a1, a2, lz), m0 = __funnelshift_l(a0, a1, lz);
  uint32_t rl = __funnelshift_r(m0, m1, 11), rh = m1 >> 11;   // 53 bits, then the rounding bit
  asm("add.cc.u32 %0, %0, %2;\n addc.u32 %1, %1, 0;" : "+r"(rl), "+r"(rh) : "r"((m0 >> 10) & 1u));
  if (e < 1 || e > 2045) {
    const double v = scalbn((double)(((unsigned long long)rh << 32) | rl), e - 1075);
    return neg ? -v : v;
  }
  return __hiloint2double((int)((rh + ((uint32_t)(e - 1) << 20)) | (neg & 0x80000000u)), (int)rl);
}

__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}

// With MULTI = false every task sums at most one chunk (128 K values): the
// accumulators go straight to the output, and the registers can hold two steps'
// values.  With MULTI = true the chunks' sums stay in 64 registers a thread and
// a step's values are loaded when they are cut (more than 128 registers all the
// same: 670 bytes a thread are spilled; with MULTI = false 160 at TN = 64, 80 at 32).
template <int TN, bool MULTI>
__global__ void __launch_bounds__(F64Cfg<TN>::THREADS, F64Cfg<TN>::CTAS)
    gemm_f64_tc_kernel(const F64Task* __restrict__ tasks, int ntasks, long long tile0, long long total, int* err,
                       unsigned long long wait_ns, F64Doubt w) {   // tiles tile0 .. total - 1
  using F = F64Cfg<TN>;
  constexpr int THREADS = F::THREADS, XU = F::XU, NBUF = F::NBUF;
  constexpr bool PAIR = !MULTI && XU == 1;            // registers hold two steps' values
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + F::ALIGN - 1) & ~(uintptr_t)(F::ALIGN - 1));
  uint8_t* yplanes = smem + PLANES * F::XPLANE;
  uint8_t* mags = smem + F::OPER;                     // leading magnitudes of a window; then outputs to sum here
  int* tab = (int*)(mags + F::MAGS);                  // operand column of each K value of the block
  uint32_t* rmax = (uint32_t*)(tab + TAB<MULTI>);     // largest high word per row: X, then Y
  int* rscale = (int*)rmax;                           // then the rows' scales in its place
  uint64_t* bar = (uint64_t*)(rscale + TM + TN);      // [2] products of a buffer done, [1] drain
  volatile uint32_t* tslot = (volatile uint32_t*)(bar + 3);
  int* nagain = (int*)(bar + 4);                      // a block's outputs in doubt; a tile's record
  F64Slot* slots = (F64Slot*)(bar + 8);               // this tile's task and the next one's
  long long* coff = (long long*)(slots + 2);          // output offset of each column
  long long* roff = coff + TN;                        // and of each row
  uint16_t* list = (uint16_t*)mags;                   // outputs to sum here (after a block's products)
  static_assert(TM * TN * 2 <= F::MAGS, "list");
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_init(&bar[2], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32((const void*)tslot)),
                 "r"(8 * TN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  int ti = 0;                                         // warp 1: task of the last slot filled
  if (warp == 1 && tile0 + blockIdx.x < total) ti = fetch_slot(&slots[0], tasks, ntasks, tile0 + blockIdx.x, 0);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tslot;
  const int quarter = warp & 3, colq = warp >> 2;     // this warp's part of a drain
  const uint32_t tdrain = tmem + ((uint32_t)(quarter * 32) << 16) + colq * 16;
  const int orow = quarter * 32 + lane;               // this thread's row of a drain
  uint32_t it = 0;                                    // steps issued so far
  bool abort = false;
  int cur = 0;

  for (long long tile = tile0 + blockIdx.x; tile < total && !abort; tile += gridDim.x, cur ^= 1) {
    const F64Task& T = slots[cur].t;
    const int x0 = slots[cur].ix * TM, y0 = slots[cur].iy * TN;
    const int nx = min(TM, T.mx - x0), ny = min(TN, T.my - y0);
    const int k0 = slots[cur].ks * T.kchunk, k1 = min(T.k, k0 + T.kchunk);
    const bool next = tile + gridDim.x < total;
    bool fetched = false;
    // loader units: 16 of X over all warps, TN / 8 of Y over the last ones
    Unit ux[XU], uy;
#pragma unroll
    for (int u = 0; u < XU; ++u) {
      const int n = warp + u * F::WARPS;
      if (T.xks == 1) { ux[u].row = n * 8 + (lane & 7); ux[u].q = lane >> 3; }
      else { ux[u].row = (n >> 2) * 32 + lane; ux[u].q = n & 3; }
      ux[u].ok = ux[u].row < nx;
      ux[u].p = T.x + (long long)slots[cur].b * T.xub + (ux[u].ok ? row_off(x0 + ux[u].row, T.nx, T.xrs, T.xbs) : 0);
    }
    const int wy = warp - F::YU0;
    if (T.yks == 1) { uy.row = wy * 8 + (lane & 7); uy.q = lane >> 3; }
    else { uy.row = (wy >> 2) * 32 + lane; uy.q = wy & 3; }
    uy.ok = wy >= 0 && uy.row < ny;
    uy.p = T.y + (long long)slots[cur].b * T.yub + (uy.ok ? row_off(y0 + uy.row, T.ny, T.yrs, T.ybs) : 0);
    if (tid < ny) coff[tid] = row_off(y0 + tid, T.ny, T.cys, T.cyb);
    if (tid >= THREADS - nx) roff[tid - (THREADS - nx)] = row_off(x0 + tid - (THREADS - nx), T.nx, T.cxs, T.cxb);
    const bool mine = quarter * 32 < nx && colq * 16 < ny;
    int rec = -1;                                     // the tile's record of outputs in doubt
    int kb = k0;
    do {
      const int len = max(0, min(KB, k1 - kb));
      const int nst = (len + KS - 1) / KS;
      if (tid < TM + TN) rmax[tid] = 0;
      if (tid == 0) *nagain = 0;
      if (T.kr)
        for (int i = tid; i < len; i += THREADS) tab[i] = k_col(T, kb + i);
      __syncthreads();
      struct Vals { double x[XU][8], y[8]; };
      auto load = [&](int s, Vals& v) {
        const int* tb = T.kr ? tab + s * KS : nullptr;
#pragma unroll
        for (int u = 0; u < XU; ++u) load_unit(ux[u], T.xks, tb, kb + s * KS, len - s * KS, v.x[u]);
        load_unit(uy, T.yks, tb, kb + s * KS, len - s * KS, v.y);
      };
      // largest magnitude of each row over the block
      uint32_t mx[XU] = {}, my = 0;
      auto widest = [&](const Vals& v) {
#pragma unroll
        for (int u = 0; u < XU; ++u) mx[u] = unit_max(v.x[u], mx[u]);
        my = unit_max(v.y, my);
      };
      Vals v0, v1;   // PAIR: the values of the next even and odd step
      if (!PAIR) {
        for (int s = nst - 1; s >= 0; --s) {
          load(s, v0);
          widest(v0);
        }
      } else {
        for (int s = (nst - 1) & ~1; s >= 0; s -= 2) {
          load(s, v0);
          if (s + 1 < nst) load(s + 1, v1);
          widest(v0);
          if (s + 1 < nst) widest(v1);
        }
      }
#pragma unroll
      for (int u = 0; u < XU; ++u)
        if (mx[u]) atomicMax(&rmax[ux[u].row], mx[u]);
      if (my) atomicMax(&rmax[TM + uy.row], my);
      __syncthreads();
      // Row scales.  A row with an infinity or a NaN sends the tile through
      // plain multiply-adds; a row of nothing but values below 2^-959 (noise to
      // the power of the chain's length is met in earnest) is taken 2^512-fold.
      bool bad = false;
      if (tid < TM + TN) {
        const uint32_t h = rmax[tid];
        bad = (h >> 20) == 0x7ffu;
        int e = (int)(h >> 20), tiny = 0;
        if (e < 64) {
          tiny = h != 0;
          e = tiny ? (int)((uint32_t)__double2hiint(__hiloint2double((int)h + 1, 0) * 0x1p512) >> 20) : ZERO_ROW;
        }
        rscale[tid] = e << 1 | tiny;
      }
      const bool plain = __syncthreads_or(bad);
      int nsum = plain ? nx * ny : 0;   // outputs to sum here
      const int pm = put_mode(T, kb == k0);
      double* C = T.c + (long long)slots[cur].b * T.cub + (long long)slots[cur].ks * T.sK;
      long long ahi[MULTI ? 16 : 1], alo[MULTI ? 16 : 1];   // sums of accumulators 0 .. 3 and 4 .. 7
      if (MULTI) {
#pragma unroll
        for (int j = 0; j < 16; ++j) ahi[j] = alo[j] = 0;
      }
      // accumulators of columns cb and cb + 1 of this thread's row, added to hi and lo
      auto drain2 = [&](int cb, long long* hi, long long* lo) {
        uint32_t v[8][2];
#pragma unroll
        for (int g = 0; g < 8; ++g) tmem_ld2(tdrain + cb + g * TN, v[g]);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          int c[8];
#pragma unroll
          for (int g = 0; g < 8; ++g) c[g] = __float2int_rn(__uint_as_float(v[g][j]));
          // |c0| <= 2^19, |c2| <= 2^22: 256 times them plus the next fits 32 bits
          hi[j] = mad_wide(c[0] * 256 + c[1], 1 << 16, mad_wide(c[2] * 256 + c[3], 1, hi[j]));
          lo[j] = mad_wide(c[4], 1 << 24, mad_wide(c[5], 1 << 16, mad_wide(c[6], 256, mad_wide(c[7], 1, lo[j]))));
        }
      };
      if (!plain) {
        // outputs to be checked: those of non-zero rows
        uint32_t sums[4] = {~0u, ~0u, ~0u, ~0u};
        if (mine && orow < nx && rscale[orow] != ZERO_ROW << 1) {
#pragma unroll
          for (int c = 0; c < 16; ++c)
            if (colq * 16 + c < ny && rscale[TM + colq * 16 + c] != ZERO_ROW << 1) sums[c >> 2] ^= ENOUGH_B << (8 * (c & 3));
        }
        auto step = [&](int s, Vals& v) -> bool {
          const uint32_t h = NBUF == 2 ? it & 1u : 0u, use = NBUF == 2 ? it >> 1 : it;   // buffer, its use count
          if (!PAIR && nst > 1) load(s, v);
          bool ok = !abort;   // a wait of the last chunk ran out: no more of them
          if (ok && use >= 1) ok = mbar_wait(&bar[h], (use - 1) & 1u, err, 11, wait_ns);
          if (ok) {
#pragma unroll
            for (int u = 0; u < XU; ++u)
              if (ux[u].ok) store_unit<F>(ux[u], v.x[u], rscale[ux[u].row], smem, F::XPLANE, h, mags, 0, s);
            if (uy.ok) store_unit<F>(uy, v.y, rscale[TM + uy.row], yplanes, F::YPLANE, h, mags, TM, s);
          }
          if (PAIR && s + 2 < nst) load(s + 2, v);
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          fence_before();
          if (!__syncthreads_and(ok)) return false;
          if (tid == 0) {
            fence_after();
            const uint64_t dx = sdesc_k<F::ROW>(smem + h * 64), dy = sdesc_k<F::ROW>(yplanes + h * 64);
            constexpr uint64_t PX = F::XPLANE >> 4, PY = F::YPLANE >> 4;
            const bool fresh = (s & (CHUNK - 1)) == 0;
#pragma unroll
            for (int kk = 0; kk < 2; ++kk) {
              if (kk == 1 && len - s * KS <= KS / 2) break;   // empty second half
              const uint64_t a = dx + 2 * kk, b = dy + 2 * kk;
              // plane pair (i, j) adds to accumulator i + j <= 7: for one i the
              // Y planes lie one after the other, and so do their accumulators
              const uint32_t keep = fresh && kk == 0 ? 0u : 1u;
#pragma unroll
              for (int i = 0; i < PLANES; ++i) {
                const int n = (PLANES - i) * TN;   // columns
                umma<MPSLCC_BF16>(tmem + i * TN, a + i * PX, b, idesc_f16(TM, n < 256 ? n : 256), i == 0 ? keep : 1u);
                if (n > 256)
                  umma<MPSLCC_BF16>(tmem + i * TN + 256, a + i * PX, b + (256 / TN) * PY, idesc_f16(TM, n - 256),
                                    i == 0 ? keep : 1u);
              }
            }
            umma_commit(&bar[h]);
          }
          if (warp == 1 && next && !fetched) {   // while the products run
            ti = fetch_slot(&slots[cur ^ 1], tasks, ntasks, tile + gridDim.x, ti);
            fetched = true;
          }
          // a window of several: checked while the products run
          const bool window = F::MW < CHUNK && (s + 1 == nst || (s & (F::MW - 1)) == F::MW - 1);
          if (window) sum_magnitudes<F>(mags, orow, colq * 16, (s & (F::MW - 1)) + 1, sums);
          if (MULTI && (s + 1 == nst || (s & (CHUNK - 1)) == CHUNK - 1)) {
            // all products up to this step are done
            if (!mbar_wait(&bar[h], use & 1u, err, 12, wait_ns)) abort = true;
            fence_after();
            if (mine) {
#pragma unroll
              for (int cb = 0; cb < 16; cb += 2) drain2(cb, ahi + (MULTI ? cb : 0), alo + (MULTI ? cb : 0));
            }
            fence_before();
          }
          if (window && s + 1 < nst) __syncthreads();   // the next step overwrites the magnitudes
          ++it;
          return true;
        };
        if (!PAIR) {
          for (int s = 0; s < nst; ++s)
            if (!step(s, v0)) { abort = true; break; }
        } else {
          for (int s = 0; s < nst; s += 2) {
            if (!step(s, v0)) { abort = true; break; }
            if (s + 1 < nst && !step(s + 1, v1)) { abort = true; break; }
          }
        }
        // one window: checked where no step's values hold registers
        static_assert(F::MW < CHUNK || !MULTI, "windows");
        if (F::MW == CHUNK) sum_magnitudes<F>(mags, orow, colq * 16, nst, sums);
        if (!MULTI && nst > 0 && !abort) {   // the last step's products
          const uint32_t use = it - 1;
          const uint32_t parity = (NBUF == 2 ? use >> 1 : use) & 1u;
          if (!mbar_wait(&bar[NBUF == 2 ? use & 1u : 0], parity, err, 12, wait_ns)) abort = true;
          fence_after();
        }
        uint32_t open = 0;   // outputs to sum again
#pragma unroll
        for (int c = 0; c < 16; ++c) open |= ((sums[c >> 2] >> (8 * (c & 3)) & 255u) != ENOUGH_B ? 1u : 0u) << c;
        int at = 0;
        if (open) at = atomicAdd(nagain, __popc(open));
        abort = __syncthreads_or(abort);
        // Outputs in doubt are left to the second kernel, or summed below where there
        // is no room for their record.
        nsum = abort ? 0 : *nagain;
        if (nsum > 0 && w.cap > 0) {
          if (rec < 0) {   // the tile's first
            __syncthreads();
            if (tid == 0) *nagain = atomicAdd(w.count, 1);
            __syncthreads();
            rec = *nagain;
            __syncthreads();
            if (rec < w.cap) {
              if (tid == 0) w.rec[rec] = tile;
              for (int b = 0; MULTI && b < w.blocks; ++b)
                w.mask[((long long)rec * w.blocks + b) * THREADS + orow * (TN / 16) + colq] = 0;
            } else {
              if (tid == 0) *nagain = 0;
              __syncthreads();
              at = open ? atomicAdd(nagain, __popc(open)) : 0;
            }
          }
          if (rec < w.cap) {
            const int b = MULTI ? (kb - k0) / KB : 0;
            w.mask[((long long)rec * w.blocks + b) * THREADS + orow * (TN / 16) + colq] = (uint16_t)open;
            nsum = 0;
          }
        }
        if (nsum > 0)
          for (uint32_t o = open; o; o &= o - 1) list[at++] = (uint16_t)(orow << 6 | (colq * 16 + __ffs(o) - 1));
        // A warp holds 32 rows (one a lane) of 16 columns.  Where rows are
        // contiguous in memory it stores them column by column; else it turns
        // its piece in shared memory (its own part: the products are done) and
        // stores two rows of 16 columns at a time, instead of 32 rows of one.
        // Outputs in doubt get a zero: their sums are added.
        if (mine && !abort) {
          const int exr = scale_exp(rscale[orow]);
          const bool lanes = T.cxs == 1;
          double* r = C + (orow < nx ? roff[orow] : 0);
          double* st = (double*)smem + warp * (32 * 17);
#pragma unroll
          for (int cb = 0; cb < 16; cb += 2) {
            long long hi[2], lo[2];
            if (MULTI) {
#pragma unroll
              for (int j = 0; j < 2; ++j) { hi[j] = ahi[cb + j]; lo[j] = alo[cb + j]; }
            } else {
              hi[0] = hi[1] = lo[0] = lo[1] = 0;
              if (nst > 0) drain2(cb, hi, lo);
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              const int col = colq * 16 + cb + j;
              double x = to_f64(hi[j], lo[j], exr + scale_exp(rscale[TM + col]));
              if (open >> (cb + j) & 1) x = 0.0;
              if (!lanes) st[lane * 17 + cb + j] = x;
              else if (col < ny && orow < nx) put(T, pm, r + coff[col], x);
            }
          }
          if (!lanes) {
            __syncwarp();
            const int col = colq * 16 + (lane & 15);
            double* c = C + (col < ny ? coff[col] : 0);
#pragma unroll 4
            for (int i = lane >> 4; i < 32; i += 2) {
              const int row = quarter * 32 + i;
              if (row < nx && col < ny) put(T, pm, c + roff[row], st[i * 17 + (lane & 15)]);
            }
          }
        }
        if (!MULTI) fence_before();
      }
      // The listed outputs, or all of a block with a row that is not finite, as plain
      // sums: eight lanes an output, each every eighth K value.
      if (nsum > 0) {
        __syncthreads();   // the list
        const int sm = plain ? pm : sum_mode(T);
        const double* X = T.x + (long long)slots[cur].b * T.xub;
        const double* Y = T.y + (long long)slots[cur].b * T.yub;
        for (int e0 = warp * 4; e0 < nsum; e0 += THREADS / 8) {
          const int e = min(e0 + (lane >> 3), nsum - 1);
          const int i = plain ? e / ny : list[e] >> 6, j = plain ? e - i * ny : list[e] & 63;
          const double* px = X + row_off(x0 + i, T.nx, T.xrs, T.xbs);
          const double* py = Y + row_off(y0 + j, T.ny, T.yrs, T.ybs);
          double s = 0.0;
#pragma unroll 4
          for (int k = lane & 7; k < len; k += 8) {
            const int col = T.kr ? tab[k] : kb + k;
            s = fma(__ldg(px + (long long)col * T.xks), __ldg(py + (long long)col * T.yks), s);
          }
#pragma unroll
          for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
          if ((lane & 7) == 0 && e0 + (lane >> 3) < nsum) put(T, sm, C + roff[i] + coff[j], s);
        }
      }
      if (warp == 1 && next && !fetched && kb + KB >= k1) {
        ti = fetch_slot(&slots[cur ^ 1], tasks, ntasks, tile + gridDim.x, ti);
        fetched = true;
      }
      abort = __syncthreads_or(abort);
      kb += KB;
    } while (MULTI && kb < k1 && !abort);   // a short sum is one block
  }
  if (abort && tid == 0) {
    // products already issued read shared and tensor memory: wait for them
    umma_commit(&bar[2]);
    mbar_wait(&bar[2], 0u, err, 13, DRAIN_NS);
  }
  __syncthreads();
  fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(8 * TN) : "memory");
}

// ---------------------------------------------------------------------------
// Outputs that the digit products leave in doubt, summed in FP64 and added: a record
// is a tile and a bit per output and block.  A kernel of its own: inlined or called,
// this code made the tensor-core kernel's loops spill (phase 2 of the M1 = 500 sigma
// 3.0 -> 4.4 ms without one output in doubt), and several CTAs an SM hide one
// another's loads.  Bound by the FP64 pipe (two multiply-adds a clock and SM) where
// most of a tile is in doubt, and by its loads otherwise.  The rows that hold such
// outputs are staged 32 values at a time; many are sparse (5 of 48 terms in the
// operator sums at M1 = 1500), so their terms are found from bit masks of the
// non-zero values.  Against sums in the tensor-core kernel that read their operands
// directly: 28.6 -> 24.0 s for the window above, 6.0 -> 4.6 s for the energies.
// ---------------------------------------------------------------------------
template <int TN> struct AgainCfg {
  static constexpr int THREADS = 256, LD = KS + 1, CTAS = TN == 64 ? 3 : 4, ENTRIES = TM * TN / 16;
  static constexpr int SMEM =
      (TM + TN) * (LD * 8 + 2 * 8) + TM * TN * 2 + 2 * (TM + TN) * 4 + KS * 4 + 64 + (int)sizeof(F64Slot);
};
template <int TN>
__global__ void __launch_bounds__(AgainCfg<TN>::THREADS, AgainCfg<TN>::CTAS)
    gemm_f64_again_kernel(const F64Task* __restrict__ tasks, int ntasks, F64Doubt w, int* next_count) {
  using A = AgainCfg<TN>;
  constexpr int THREADS = A::THREADS, LD = A::LD, U = 4;
  extern __shared__ uint8_t smem_raw[];
  double* xs = (double*)smem_raw;                       // [row][k]
  double* ys = xs + TM * LD;
  long long* xo = (long long*)(ys + TN * LD);           // operand and output offsets of the rows
  long long* yo = xo + TM;
  long long* roff = yo + TN;
  long long* coff = roff + TM;
  F64Slot* slot = (F64Slot*)(coff + TN);
  uint32_t* masks = (uint32_t*)(slot + 1);              // two sets, of this step's values and the next one's
  uint32_t* need = masks + 2 * (TM + TN);               // rows of X, then of Y, that hold outputs of the list
  int* kcol = (int*)(need + 8);
  int* count = kcol + KS;
  uint16_t* list = (uint16_t*)(count + 2);              // row << 6 | column
  const int tid = threadIdx.x;
  if (blockIdx.x == 0 && tid == 0) *next_count = 0;     // of the launch after this one
  const int nrec = min(*w.count, w.cap);
  for (int r = blockIdx.x; r < nrec; r += gridDim.x) {
    __syncthreads();
    if (tid < 32) fetch_slot(slot, tasks, ntasks, w.rec[r], 0);
    if (tid < 2 * (TM + TN)) masks[tid] = 0;
    if (TM + TN > THREADS / 2 && tid + THREADS < 2 * (TM + TN)) masks[tid + THREADS] = 0;
    __syncthreads();
    const F64Task& T = slot->t;
    const int x0 = slot->ix * TM, y0 = slot->iy * TN;
    const int nx = min(TM, T.mx - x0), ny = min(TN, T.my - y0);
    const int k0 = slot->ks * T.kchunk, k1 = min(T.k, k0 + T.kchunk);
    if (tid < nx) {
      xo[tid] = row_off(x0 + tid, T.nx, T.xrs, T.xbs);
      roff[tid] = row_off(x0 + tid, T.nx, T.cxs, T.cxb);
    }
    if (tid >= THREADS - ny) {
      const int c = tid - (THREADS - ny);
      yo[c] = row_off(y0 + c, T.ny, T.yrs, T.ybs);
      coff[c] = row_off(y0 + c, T.ny, T.cys, T.cyb);
    }
    const double* X = T.x + (long long)slot->b * T.xub;
    const double* Y = T.y + (long long)slot->b * T.yub;
    double* C = T.c + (long long)slot->b * T.cub + (long long)slot->ks * T.sK;
    const bool xk = T.xks == 1, yk = T.yks == 1;
    const int mode = sum_mode(T);
    uint32_t set = 0;
    for (int blk = 0; blk < w.blocks; ++blk) {
      const int ka = k0 + blk * KB, kz = min(k1, ka + KB);
      __syncthreads();
      if (tid < 8) need[tid] = 0;
      if (tid == 8) *count = 0;
      __syncthreads();
      for (int e = tid; e < A::ENTRIES; e += THREADS) {
        uint32_t bits = w.mask[((long long)r * w.blocks + blk) * A::ENTRIES + e];
        const int row = e / (TN / 16), c0 = e % (TN / 16) * 16;
        if (!bits) continue;
        atomicOr(&need[row >> 5], 1u << (row & 31));
        atomicOr(&need[4 + (c0 >> 5)], bits << (c0 & 31));
        int at = atomicAdd(count, __popc(bits));
        for (; bits; bits &= bits - 1) list[at++] = (uint16_t)(row << 6 | (c0 + __ffs(bits) - 1));
      }
      __syncthreads();
      const int n = *count;
      for (int base = 0; base < n; base += U * THREADS) {
        int at[U];
        double acc[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int e = base + u * THREADS + tid;
          at[u] = e < n ? list[e] : -1;
          acc[u] = 0.0;
        }
        for (int kk = ka; kk < kz; kk += KS, set ^= 1u) {
          const int nk = min(KS, kz - kk);
          uint32_t* mx = masks + set * (TM + TN);
          uint32_t* my = mx + TM;
          if (tid < nk) kcol[tid] = k_col(T, kk + tid);
          __syncthreads();
          // rows in need of it; values of other rows are not read
          auto stage = [&](auto cols, const double* P, const long long* off, const uint32_t* nd, int nr, bool alongk,
                           long long ks, double* dst, uint32_t* mk) {
            constexpr int R = decltype(cols)::value, N = R * KS / THREADS;
#pragma unroll 1
            for (int i0 = 0; i0 < N; i0 += 8 < N ? 8 : N) {
              constexpr int B = 8 < N ? 8 : N;
              double v[B];
#pragma unroll
              for (int i = 0; i < B; ++i) {
                const int e = tid + (i0 + i) * THREADS, rr = alongk ? e / KS : e % R, q = alongk ? e % KS : e / R;
                const bool on = rr < nr && q < nk && (nd[rr >> 5] >> (rr & 31) & 1u);
                v[i] = on ? __ldg(P + off[rr] + (long long)kcol[q] * ks) : 0.0;
              }
#pragma unroll
              for (int i = 0; i < B; ++i) {
                const int e = tid + (i0 + i) * THREADS, rr = alongk ? e / KS : e % R, q = alongk ? e % KS : e / R;
                dst[rr * LD + q] = v[i];
                if (v[i] != 0.0) atomicOr(&mk[rr], 1u << q);
              }
            }
          };
          stage(std::integral_constant<int, TM>(), X, xo, need, nx, xk, T.xks, xs, mx);
          stage(std::integral_constant<int, TN>(), Y, yo, need + 4, ny, yk, T.yks, ys, my);
          __syncthreads();
          if (tid < TM + TN) masks[(set ^ 1u) * (TM + TN) + tid] = 0;
#pragma unroll
          for (int u = 0; u < U; ++u) {
            if (at[u] < 0) continue;
            const int i = at[u] >> 6, j = at[u] & 63;
            const double* px = xs + i * LD;
            const double* py = ys + j * LD;
            double a = acc[u];
            const uint32_t m0 = mx[i] & my[j];
            if (__popc(m0) > nk / 2) {
#pragma unroll 4
              for (int q = 0; q < nk; ++q) a = fma(px[q], py[q], a);
            } else {
              for (uint32_t m = m0; m; m &= m - 1) {
                const int q = __ffs(m) - 1;
                a = fma(px[q], py[q], a);
              }
            }
            acc[u] = a;
          }
          __syncthreads();
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (at[u] >= 0) put(T, mode, C + roff[at[u] >> 6] + coff[at[u] & 63], acc[u]);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// FP64-pipe kernel: 32 x 32 output tiles, outputs dense over the threads (no
// multiply-add is issued for padding), or thin tiles; each output is summed in
// ascending K.  (One warp a tile without shared memory, 32 of them on an SM,
// measured slower: 18.9 against 15.5 ms over the energies at M1 = 400, and 3x
// on long sums of few outputs, whose loads then lie on the chain.)
// ---------------------------------------------------------------------------
constexpr int SM_T = 32, THIN_X = 8, THIN_Y = 256, THIN_K = 64;

// A tile of up to 8 rows of X (kept in shared memory) and 256 rows of Y, one a
// thread: Y is read once, coalesced where its rows are contiguous.  Sums of a
// few matrices with coefficients (the operators' dense blocks) are of this
// form: 8 x k multiply-adds per value read.  As 128-row tensor-core tiles 2 %
// full they took 35 of the energies' 88 ms at M1 = 400.
template <int N>
__device__ __forceinline__ void thin_sum(const double* xs, const double* y, long long yks, const int* kcol, int nk,
                                         double (&acc)[THIN_X]) {
#pragma unroll 4
  for (int q = 0; q < nk; ++q) {
    const double v = __ldg(y + (long long)kcol[q] * yks);
#pragma unroll
    for (int i = 0; i < N; ++i) acc[i] = fma(xs[q * THIN_X + i], v, acc[i]);
  }
}

__device__ __forceinline__ void thin_tile(const F64Task& T, const F64Tile& tc, double* xs, int* kcol) {
  const int tid = threadIdx.x;
  const int x0 = tc.ix * THIN_X, y0 = tc.iy * THIN_Y;
  const int nx = min(THIN_X, T.mx - x0), ny = min(THIN_Y, T.my - y0);
  const int k0 = tc.ks * T.kchunk, k1 = min(T.k, k0 + T.kchunk);
  const double* X = T.x + (long long)tc.b * T.xub;
  double* C = T.c + (long long)tc.b * T.cub + (long long)tc.ks * T.sK;
  const bool ok = tid < ny;
  const double* y = T.y + (long long)tc.b * T.yub + (ok ? row_off(y0 + tid, T.ny, T.yrs, T.ybs) : 0);
  double acc[THIN_X];
#pragma unroll
  for (int i = 0; i < THIN_X; ++i) acc[i] = 0.0;
  for (int kk = k0; kk < k1; kk += THIN_K) {
    const int nk = min(THIN_K, k1 - kk);
    if (tid < nk) kcol[tid] = k_col(T, kk + tid);
    __syncthreads();
    for (int e = tid; e < nk * THIN_X; e += 256) {
      const int q = e / THIN_X, i = e - q * THIN_X;
      xs[e] = i < nx ? X[row_off(x0 + i, T.nx, T.xrs, T.xbs) + (long long)kcol[q] * T.xks] : 0.0;
    }
    __syncthreads();
    if (ok) {
      if (nx == 1) thin_sum<1>(xs, y, T.yks, kcol, nk, acc);
      else if (nx == 2) thin_sum<2>(xs, y, T.yks, kcol, nk, acc);
      else if (nx <= 4) thin_sum<4>(xs, y, T.yks, kcol, nk, acc);
      else thin_sum<8>(xs, y, T.yks, kcol, nk, acc);
    }
    __syncthreads();
  }
  if (!ok) return;
  const int pm = put_mode(T, true);
  const long long c = row_off(y0 + tid, T.ny, T.cys, T.cyb);
#pragma unroll
  for (int i = 0; i < THIN_X; ++i)
    if (i < nx) put(T, pm, C + row_off(x0 + i, T.nx, T.cxs, T.cxb) + c, acc[i]);
}

__global__ void __launch_bounds__(256) gemm_f64_pipe_kernel(const F64Task* __restrict__ tasks, int ntasks,
                                                             long long total) {
  __shared__ double xs[SM_T][SM_T + 1], ys[SM_T][SM_T + 1];   // [k][row]
  __shared__ int kcol[THIN_K];
  const int tid = threadIdx.x;
  int ti = 0;
  for (long long tile = blockIdx.x; tile < total; tile += gridDim.x) {
    ti = warp_find(tasks, ntasks, tile, ti);
    const F64Task T = tasks[ti];
    const F64Tile tc = tile_of(T, tile);
    if (T.thin) {
      thin_tile(T, tc, &xs[0][0], kcol);
      continue;
    }
    const int x0 = tc.ix * SM_T, y0 = tc.iy * SM_T;
    const int nx = min(SM_T, T.mx - x0), ny = min(SM_T, T.my - y0);
    const int k0 = tc.ks * T.kchunk, k1 = min(T.k, k0 + T.kchunk);
    const double* X = T.x + (long long)tc.b * T.xub;
    const double* Y = T.y + (long long)tc.b * T.yub;
    double* C = T.c + (long long)tc.b * T.cub + (long long)tc.ks * T.sK;
    const int nout = nx * ny;
    int oi[4], oj[4];
    double acc[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = tid + u * 256;
      oi[u] = e < nout ? e / ny : -1;
      oj[u] = e < nout ? e - oi[u] * ny : 0;
      acc[u] = 0.0;
    }
    // each thread loads four elements of either operand per step
    const int xa = tid & 31, xb = tid >> 5;   // fast and slow index of the load
    const long long xrow = T.xks == 1 ? 0 : (xa < nx ? row_off(x0 + xa, T.nx, T.xrs, T.xbs) : 0);
    const long long yrow = T.yks == 1 ? 0 : (xa < ny ? row_off(y0 + xa, T.ny, T.yrs, T.ybs) : 0);
    long long xr4[4], yr4[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = xb + 8 * u;
      xr4[u] = T.xks == 1 && r < nx ? row_off(x0 + r, T.nx, T.xrs, T.xbs) : 0;
      yr4[u] = T.yks == 1 && r < ny ? row_off(y0 + r, T.ny, T.yrs, T.ybs) : 0;
    }
    for (int kk = k0; kk < k1; kk += SM_T) {
      const int nk = min(SM_T, k1 - kk);
      const int kf = T.kr && xa < nk ? k_col(T, kk + xa) : kk + xa;   // column of the fast index
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int s = xb + 8 * u;
        int col = kk + s;
        if (T.kr && (T.xks != 1 || T.yks != 1) && s < nk) col = k_col(T, col);
        if (T.xks == 1) xs[xa][s] = (s < nx && xa < nk) ? X[xr4[u] + kf] : 0.0;
        else xs[s][xa] = (xa < nx && s < nk) ? X[xrow + (long long)col * T.xks] : 0.0;
        if (T.yks == 1) ys[xa][s] = (s < ny && xa < nk) ? Y[yr4[u] + kf] : 0.0;
        else ys[s][xa] = (xa < ny && s < nk) ? Y[yrow + (long long)col * T.yks] : 0.0;
      }
      __syncthreads();
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (oi[u] < 0) continue;
        double a = acc[u];
        for (int q = 0; q < nk; ++q) a = fma(xs[q][oi[u]], ys[q][oj[u]], a);
        acc[u] = a;
      }
      __syncthreads();
    }
    const int pm = put_mode(T, true);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (oi[u] >= 0)
        put(T, pm, C + row_off(x0 + oi[u], T.nx, T.cxs, T.cxb) + row_off(y0 + oj[u], T.ny, T.cys, T.cyb), acc[u]);
  }
}

inline long long cdiv(long long a, long long b) { return (a + b - 1) / b; }

}  // namespace

// Rows and K of a task in the kernels' form.  A batch that shares one operand
// becomes rows of the other (their tiles then fill up whatever the batch's own
// size): fold 1 along A's rows, 2 along B's.
struct F64Dims {
  long long ma, mb;   // rows of op(A), columns of op(B), folded
  int fold, k, kc, batch, ksplit;
};
static F64Dims f64_dims(const GemmTask& g) {
  F64Dims d;
  const long long big = 1LL << 30;
  d.ma = g.m;
  d.mb = g.n;
  d.batch = g.batch;
  d.fold = 0;
  if (g.batch > 1 && g.sB == 0 && g.batch * d.ma < big) { d.fold = 1; d.ma *= g.batch; d.batch = 1; }
  else if (g.batch > 1 && g.sA == 0 && g.batch * d.mb < big) { d.fold = 2; d.mb *= g.batch; d.batch = 1; }
  d.k = g.kr ? g.kv : g.k;
  d.ksplit = std::max(1, g.ksplit);
  d.kc = (int)(cdiv(cdiv(std::max(d.k, 1), d.ksplit), 16) * 16);
  return d;
}

// How a task runs on the FP64 pipe or on the tensor cores: its operands as given
// or exchanged, with the estimated SM clocks of the whole task and the longest
// tile.
struct F64Form {
  double clocks, tile;
  int swap, bx, by;   // exchanged operands; tile
  bool thin;
};

// A multiply-add instruction of the FP64 pipe takes 16 clocks a warp whatever
// its operands.
static F64Form pipe_form(const F64Dims& d) {
  const double kc = std::max(1, std::min(d.k, d.kc));
  const double reps = (double)d.batch * d.ksplit;
  const double o = (double)std::min<long long>(d.ma, SM_T) * std::min<long long>(d.mb, SM_T);
  const double sq = 700.0 + (300.0 / SM_T) * (kc + SM_T) + 0.5 * kc * (o + 31.0);
  F64Form f{sq * reps * cdiv(d.ma, SM_T) * cdiv(d.mb, SM_T), sq, 0, SM_T, SM_T, false};
  for (int w = 0; w < 2; ++w) {
    const long long x = w ? d.mb : d.ma, y = w ? d.ma : d.mb;
    const int n = x == 1 ? 1 : (x == 2 ? 2 : (x <= 4 ? 4 : 8));
    const double t = 400.0 + std::max(0.5 * kc * n * (std::min<long long>(y, THIN_Y) + 31), 60.0 * (kc + n));
    const double all = t * reps * cdiv(x, THIN_X) * cdiv(y, THIN_Y);
    if (all < f.clocks) f = {all, t, w, THIN_X, THIN_Y, true};
  }
  return f;
}

// Tensor-core tile: set-up, a step's products and barriers, the cutting of its
// rows' digits, the drain and the write-out of its 32 x 16 pieces.  Measured
// with clocks on the device at K = 56, M1 = 500: about 45000 a full tile of 128
// x 64.
static F64Form tc_form(const F64Dims& d, const GemmTask& g, int tn) {
  const double kc = std::max(1, std::min(d.k, d.kc)), steps = (double)(((long long)kc + KS - 1) / KS);
  F64Form best{1e300, 0, 0, TM, tn, false};
  for (int w = 0; w < 2; ++w) {
    const long long x = w ? d.mb : d.ma, y = w ? d.ma : d.mb;
    const double tx = (double)cdiv(x, TM), ty = (double)cdiv(y, tn);
    const double px = 0.5 + x / 32.0, py = 0.5 + y / 16.0;   // pieces along each side, all tiles
    const bool lanes = (w ? 1 : g.ldc) == 1;                  // rows contiguous in memory
    const double tile = tn == 64 ? 8500.0 + 4200.0 * steps : 4500.0 + 2200.0 * steps;
    const double rows = steps * (steps > 1 ? 140.0 : 80.0) * (ty * x + tx * y) / 8.0;
    const double out = px * py * (330.0 * ((long long)(kc / 128) + 1) + (lanes ? 300.0 : 450.0));
    const double all = (tx * ty * tile + rows + out) * d.batch * d.ksplit;
    if (all < best.clocks) best = {all, tile, w, TM, tn, false};
  }
  return best;
}

static bool is_long(const F64Dims& d) { return std::min(d.k, d.kc) > KS * CHUNK; }

static F64Task make_task(const GemmTask& g, const F64Dims& d, const F64Form& f) {
  F64Task t;
  std::memset(&t, 0, sizeof(t));
  const bool ta = g.flags & GEMM_TA, tb = g.flags & GEMM_TB;
  t.x = g.A; t.y = g.B; t.c = g.C;
  t.xrs = ta ? 1 : g.lda; t.xks = ta ? g.lda : 1;
  t.yrs = tb ? g.ldb : 1; t.yks = tb ? 1 : g.ldb;
  t.nx = g.m; t.mx = (int)d.ma;
  t.ny = g.n; t.my = (int)d.mb;
  t.cxs = g.ldc; t.cys = 1;
  t.batch = d.batch;
  if (d.fold == 1) { t.xbs = g.sA; t.cxb = g.sC; }
  else if (d.fold == 2) { t.ybs = g.sB; t.cyb = g.sC; }
  else { t.xub = g.sA; t.yub = g.sB; t.cub = g.sC; }
  t.k = d.k;
  t.kr = g.kr;
  t.nkr = g.nkr;
  t.alpha = g.alpha;
  t.beta = d.ksplit > 1 ? 0.0 : g.beta;   // partial sums: what lies there is not C
  t.ksplit = d.ksplit;
  MPSLCC_REQUIRE(t.ksplit == 1 || g.sK > 0, ST_INTERNAL, "FP64 task split over K without partial offsets");
  t.sK = t.ksplit > 1 ? g.sK : 0;
  t.kchunk = d.kc;
  if (f.swap) {
    std::swap(t.x, t.y);
    std::swap(t.xrs, t.yrs); std::swap(t.xks, t.yks); std::swap(t.xbs, t.ybs); std::swap(t.xub, t.yub);
    std::swap(t.nx, t.ny); std::swap(t.mx, t.my);
    std::swap(t.cxs, t.cys); std::swap(t.cxb, t.cyb);
  }
  t.thin = f.thin;
  t.tx = (int)cdiv(t.mx, f.bx);
  t.ty = (int)cdiv(t.my, f.by);
  return t;
}

// A launch whose multiply-adds keep the FP64 pipes busy for no longer than a
// tensor-core launch takes to fill and drain (about 10 us; 30 us for the
// longest tile) runs there whole: one launch instead of two, and its sums are
// plain FP64 chains.
static bool short_launch(double clocks, double longest) { return clocks <= 152 * 20e3 && longest <= 60e3; }

static bool f64_empty(const GemmTask& g) { return g.m <= 0 || g.n <= 0 || g.batch <= 0; }

bool f64_on_pipe(const GemmTask* g, int n) {
  double sum = 0, longest = 0;
  for (int i = 0; i < n; ++i) {
    if (f64_empty(g[i])) continue;
    const F64Form f = pipe_form(f64_dims(g[i]));
    sum += f.clocks;
    longest = std::max(longest, f.tile);
  }
  return short_launch(sum, longest);
}

// Splits a task list between the kernels, by estimated clocks, and fills the
// tile counts.  The short sums of a launch share one tile shape; long ones take
// 128 x 32 (two CTAs per SM overlap the cutting and the drains: 2.8 against 3.4
// ms for phase 2 of the M1 = 500 sigma, K = 2900).
void plan_f64(const GemmTask* g, int n, F64Plan& p) {
  p = F64Plan();
  struct Opt { F64Dims d; F64Form pipe, tc[2]; };
  std::vector<Opt> o((size_t)n);
  double sum = 0, longest = 0, cost[2] = {0, 0};
  for (int i = 0; i < n; ++i) {
    if (f64_empty(g[i])) continue;
    o[i].d = f64_dims(g[i]);
    o[i].pipe = pipe_form(o[i].d);
    sum += o[i].pipe.clocks;
    longest = std::max(longest, o[i].pipe.tile);
  }
  const bool all_pipe = short_launch(sum, longest);
  if (!all_pipe) {
    for (int i = 0; i < n; ++i) {
      if (f64_empty(g[i])) continue;
      for (int w = 0; w < 2; ++w) {
        o[i].tc[w] = tc_form(o[i].d, g[i], w || is_long(o[i].d) ? 32 : 64);
        cost[w] += std::min(o[i].pipe.clocks, o[i].tc[w].clocks);
      }
    }
    p.tn = cost[1] < cost[0] ? 32 : 64;
  }
  const int w = p.tn == 32 ? 1 : 0;
  for (int i = 0; i < n; ++i) {
    if (f64_empty(g[i])) continue;
    const bool pipe = all_pipe || o[i].pipe.clocks <= o[i].tc[w].clocks;
    const int list = pipe ? F64_PIPE : (is_long(o[i].d) ? F64_LONG : F64_SHORT);
    F64Task t = make_task(g[i], o[i].d, pipe ? o[i].pipe : o[i].tc[w]);
    t.tile0 = p.tiles[list];
    p.tiles[list] += (long long)t.batch * t.ksplit * t.tx * t.ty;
    if (list == F64_LONG) p.blocks = std::max(p.blocks, (int)cdiv(std::min(t.k, t.kchunk), KB));
    p.t[list].push_back(t);
  }
  for (int l = 0; l < F64_LISTS; ++l) p.n[l] = (int)p.t[l].size();
}

size_t f64_plan_bytes(const F64Plan& p) {
  size_t n = 0;
  for (const auto& l : p.t) n += l.size();
  return n * sizeof(F64Task);
}

// Copies the plan's tasks to device memory at d (f64_plan_bytes of it).
void upload_f64(const F64Plan& p, void* d, cudaStream_t s) {
  for (const auto& l : p.t) {
    if (l.empty()) continue;
    cuda_check(cudaMemcpyAsync(d, l.data(), l.size() * sizeof(F64Task), cudaMemcpyHostToDevice, s), "upload FP64 tasks");
    d = (char*)d + l.size() * sizeof(F64Task);
  }
}

template <int TN, bool MULTI>
static int launch_f64_tc(const F64Task* d, int n, long long tiles, int device, int sms, int* err, cudaStream_t s,
                         unsigned long long wait_ns, F64Scratch* scratch, int nblocks = 1) {
  using F = F64Cfg<TN>;
  static std::atomic<bool> attr[MAX_DEV];
  MPSLCC_REQUIRE(device >= 0 && device < MAX_DEV, ST_ARG, "device ordinal out of range");
  if (!attr[device].load(std::memory_order_acquire)) {
    cuda_check(cudaFuncSetAttribute(gemm_f64_tc_kernel<TN, MULTI>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    f64_smem<F, MULTI>()),
               "smem attr");
    cuda_check(cudaFuncSetAttribute(gemm_f64_again_kernel<TN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    AgainCfg<TN>::SMEM),
               "smem attr");
    attr[device].store(true, std::memory_order_release);
  }
  // Tiles in pairs of launches that the records have room for.  Two counts take
  // turns: the second kernel of one pair clears the next one's.
  const int blocks = MULTI ? nblocks : 1;
  const size_t bytes = f64_record_bytes(TN, blocks);
  const bool room = blocks <= F64_MAX_BLOCKS && scratch && scratch->bytes >= F64_SCRATCH_HEAD + bytes;
  F64Doubt w = {nullptr, nullptr, nullptr, 0, blocks};
  long long step = tiles;
  if (room) {
    const long long most = f64_launch_tiles(TN, blocks);
    w.cap = (int)std::min((long long)((scratch->bytes - F64_SCRATCH_HEAD) / bytes), most);
    w.rec = (long long*)((char*)scratch->p + F64_SCRATCH_HEAD);
    w.mask = (uint16_t*)(w.rec + w.cap);
    if (w.cap == most) step = most;
  }
  int launches = 0;
  for (long long t0 = 0; t0 < tiles; t0 += step) {
    const long long t1 = std::min(tiles, t0 + step);
    int* counts = room ? (int*)scratch->p : nullptr;
    if (room) w.count = counts + (scratch->turn++ & 1);
    const int grid = (int)std::min<long long>(t1 - t0, (long long)std::max(1, sms) * F::CTAS);
    gemm_f64_tc_kernel<TN, MULTI><<<grid, F::THREADS, f64_smem<F, MULTI>(), s>>>(d, n, t0, t1, err, wait_ns, w);
    ++launches;
    if (!room) continue;
    const int g2 = (int)std::min<long long>(t1 - t0, (long long)std::max(1, sms) * AgainCfg<TN>::CTAS);
    gemm_f64_again_kernel<TN>
        <<<g2, AgainCfg<TN>::THREADS, AgainCfg<TN>::SMEM, s>>>(d, n, w, counts + (scratch->turn & 1));
    ++launches;
  }
  return launches;
}

size_t f64_scratch_bytes(const F64Launch& l) {
  const auto need = [](long long tiles, int tn, int blocks) {
    if (blocks > F64_MAX_BLOCKS) return (size_t)0;
    return (size_t)std::min(tiles, f64_launch_tiles(tn, blocks)) * f64_record_bytes(tn, blocks);
  };
  const size_t n = std::max(need(l.tiles[F64_SHORT], l.tn, 1), need(l.tiles[F64_LONG], 32, l.blocks));
  return n ? F64_SCRATCH_HEAD + n : 0;
}

int launch_f64(const F64Launch& l, const void* d, int device, int sms, int* err, cudaStream_t s,
               unsigned long long wait_ns, F64Scratch* scratch) {
  int launches = 0;
  const F64Task* t = (const F64Task*)d;
  for (int i = 0; i < F64_LISTS; ++i) {
    const int n = l.n[i];
    const long long tiles = l.tiles[i];
    MPSLCC_REQUIRE((tiles > 0) == (n > 0), ST_INTERNAL, "FP64 task list without its counts");
    if (n == 0) continue;
    if (i == F64_PIPE) {
      gemm_f64_pipe_kernel<<<(int)std::min<long long>(tiles, 152LL * 8), 256, 0, s>>>(t, n, tiles);
      ++launches;
    } else if (i == F64_SHORT && l.tn == 32) {
      launches += launch_f64_tc<32, false>(t, n, tiles, device, sms, err, s, wait_ns, scratch);
    } else if (i == F64_SHORT) {
      launches += launch_f64_tc<64, false>(t, n, tiles, device, sms, err, s, wait_ns, scratch);
    } else {
      launches += launch_f64_tc<32, true>(t, n, tiles, device, sms, err, s, wait_ns, scratch, l.blocks);
    }
    t += n;
  }
  return launches;
}

}  // namespace mpslcc
