// FP64 GEMM tasks (energies, environments, fused operators, truncations and
// sigma products of the FP64 path).
//
// GB300's FP64 pipe issues two fused multiply-adds per clock and SM (1.25
// TFLOP/s for the chip), about 1/1800 of its BF16 tensor rate.  So large tasks
// run as exact integer products on the tensor cores (Ozaki's splitting): every
// row of an operand is scaled by a power of two to 62-bit integers, each
// integer is cut into eight balanced digits of eight bits, digits are exact in
// BF16, and products of digit planes accumulate exactly in FP32 (at most 8 x
// 128 products of 2^14).  The 36 plane pairs whose weight is at least 2^-56 of
// the largest are formed; pairs of equal weight share one accumulator, the
// accumulators are combined in integers and rounded to FP64 once per 1024 K
// values.  Against a chain of FP64 multiply-adds, whose error grows with K,
// what is lost is the rounding of an operand to 2^-62 of its row's largest
// value and the pairs left out (2^-60 of a product of two such values).
//
// Tasks of few multiply-adds run on the FP64 pipe (gemm_f64_small_kernel).
//
// Measured against the 64 x 64 FP64-pipe tiles that did all of this before
// (3-band model, M1 = 500, middle position): sigma phases 27.0 + 28.8 ms ->
// 3.8 + 3.4 ms, error against 64-bit contraction 2.4e-15 -> 1.0e-15; the
// environment passes of the energies at M1 = 400, 790 ms -> 120 ms.
#include <algorithm>
#include <atomic>
#include <cstring>

#include "engine.hpp"
#include "tcgen05.cuh"

namespace mpslcc {

namespace {

constexpr int TM = 128, TN = 64;       // tensor-core tile (rows of X, rows of Y)
constexpr int KB = 1024;               // K values per scaling block
constexpr int KS = 32;                 // K values per step (half a 128-byte row of BF16)
constexpr int CHUNK = 4;               // steps between two drains: 128 K values
constexpr int PLANES = 8;
constexpr int THREADS = 512;
constexpr int XPLANE = TM * 128, YPLANE = TN * 128;          // bytes of a digit plane (64 K values)
constexpr int OPER = PLANES * (XPLANE + YPLANE);             // 192 KB
constexpr int STG_LD = TN + 1;                               // staging pitch of the result tile, doubles
constexpr int SMEM_TC = OPER + 1024 + KB * 4 + (TM + TN) * 4 + 64 + (int)sizeof(F64Task);
constexpr int SM_T = 32;               // tile of the FP64-pipe kernel
constexpr int MAX_DEV = 128;

__device__ __forceinline__ int find_f64(const F64Task* t, int n, long long tile) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (t[mid].tile0 <= tile) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

struct F64Tile { int b, ks, ix, iy; };
__device__ __forceinline__ F64Tile tile_of(const F64Task& T, long long tile) {
  const long long local = tile - T.tile0;
  const long long txy = (long long)T.tx * T.ty, per_b = txy * T.ksplit;
  F64Tile t;
  t.b = (int)(local / per_b);
  const long long r = local - (long long)t.b * per_b;
  t.ks = (int)(r / txy);
  const int q = (int)(r - (long long)t.ks * txy);
  t.ix = q / T.ty;
  t.iy = q - t.ix * T.ty;
  return t;
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
// thread holds the eight K values q, q + 4, ..., q + 28 of one row's step.
struct Unit {
  const double* p;
  long long ks;
  int row, q;
  bool ok;
};

__device__ __forceinline__ void load_unit(const Unit& u, const int* tab, int nk, double (&v)[8]) {
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int k = u.q + 4 * j;
    v[j] = (u.ok && k < nk) ? __ldg(u.p + (long long)tab[k] * u.ks) : 0.0;
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

// v as an integer of 62 bits relative to the row exponent, offset by 128 in
// every digit: byte i of the result is digit i plus 128.
__device__ __forceinline__ unsigned long long digits(double v, int emax) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  const int e = (hi >> 20) & 0x7ff;
  unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
  int d = min(emax - e, 62);
  m <<= 10;                          // one guard bit below the 62-bit grid
  m = ((m >> d) + 1) >> 1;           // round half up in magnitude
  if (e == 0) m = 0;
  const unsigned long long s = (unsigned long long)((long long)(int)hi >> 63);
  return ((m ^ s) - s) + 0x8080808080808080ull;
}

// Writes the unit's eight values as 16 bytes in each digit plane (128-byte
// swizzle: 16-byte chunk index xor row within the 8-row group).
__device__ __forceinline__ void store_unit(const Unit& u, const double (&v)[8], int emax, uint8_t* planes, int plane,
                                           int half) {
  unsigned long long t[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) t[j] = digits(v[j], emax);
  uint8_t* dst = planes + u.row * 128 + (((half * 4 + u.q) ^ (u.row & 7)) << 4);
#pragma unroll
  for (int p = 0; p < PLANES; ++p) {
    const int dg = PLANES - 1 - p;   // plane 0 holds the most significant digit
    uint32_t w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t a = dg < 4 ? (uint32_t)t[2 * j] : (uint32_t)(t[2 * j] >> 32);
      const uint32_t b = dg < 4 ? (uint32_t)t[2 * j + 1] : (uint32_t)(t[2 * j + 1] >> 32);
      const int s = dg & 3;
      // the digits plus 128 in the low bytes of two 16-bit halves
      const uint32_t y = __byte_perm(a, b, s | (s + 4) << 8);
      // BF16 128 + (y mod 128), minus 128 or 256: the digit, exactly
      const uint32_t f = (y & 0x007f007fu) | 0x43004300u;
      const uint32_t g = (y & 0x00800080u) ^ 0x43804380u;
      uint32_t r;
      asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(f), "r"(g));
      w[j] = r;
    }
    *reinterpret_cast<uint4*>(dst + p * plane) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// hi 2^32 + lo, in units of 2^(eab - 2112), as FP64 rounded to nearest.
__device__ __forceinline__ double to_f64(long long hi, long long lo, int eab) {
  unsigned long long w0 = ((unsigned long long)hi << 32) + (unsigned long long)lo;
  long long w1 = (hi >> 32) + (lo >> 63) + (w0 < (unsigned long long)lo ? 1 : 0);
  const unsigned long long s = (unsigned long long)(w1 >> 63);
  w0 ^= s;
  w1 ^= (long long)s;
  w0 -= s;
  if (s && w0 == 0) ++w1;
  int lz, top;
  unsigned long long nrm;
  if (w1 != 0) {
    lz = __clzll(w1);
    nrm = (unsigned long long)w1 << lz;
    if (lz) nrm |= w0 >> (64 - lz);
    top = 127 - lz;
  } else {
    if (w0 == 0) return 0.0;
    lz = __clzll((long long)w0);
    nrm = w0 << lz;
    top = 63 - lz;
  }
  const int e = eab + top - 1089;
  const unsigned long long mant = (nrm >> 11) + ((nrm >> 10) & 1);   // in [2^52, 2^53]
  if (e < 1 || e > 2045) {
    const double v = scalbn((double)mant, eab + top - 52 - 2112);
    return s ? -v : v;
  }
  return __longlong_as_double((long long)(((((unsigned long long)(e - 1)) << 52) + mant) | (s << 63)));
}

__global__ void __launch_bounds__(THREADS, 1)
    gemm_f64_tc_kernel(const F64Task* __restrict__ tasks, int ntasks, long long total, int* err,
                       unsigned long long wait_ns) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* yplanes = smem + PLANES * XPLANE;
  int* tab = (int*)(smem + OPER);                     // operand column of each K value of the block
  uint32_t* rmax = (uint32_t*)(tab + KB);             // largest high word per row: X, then Y
  uint64_t* bar = (uint64_t*)(rmax + TM + TN);        // [2] products of a half done, [1] drain
  volatile uint32_t* tslot = (volatile uint32_t*)(bar + 3);
  F64Task* task = (F64Task*)(bar + 8);                // the tile's task
  double* stg = (double*)smem;                        // result tile (after the products)
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
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tslot;
  const int quarter = warp & 3, colq = warp >> 2;     // this warp's part of a drain
  uint32_t it = 0;                                    // steps issued so far
  bool abort = false;

  for (long long tile = blockIdx.x; tile < total && !abort; tile += gridDim.x) {
    if (tid < (int)(sizeof(F64Task) / 8))
      ((long long*)task)[tid] = ((const long long*)(tasks + find_f64(tasks, ntasks, tile)))[tid];
    __syncthreads();
    const F64Task& T = *task;
    const F64Tile tc = tile_of(T, tile);
    const int x0 = tc.ix * TM, y0 = tc.iy * TN;
    const int nx = min(TM, T.mx - x0), ny = min(TN, T.my - y0);
    const int k0 = tc.ks * T.kchunk, k1 = min(T.k, k0 + T.kchunk);
    const double* X = T.x + (long long)tc.b * T.xub;
    const double* Y = T.y + (long long)tc.b * T.yub;
    double* C = T.c + (long long)tc.b * T.cub + (long long)tc.ks * T.sK;
    // loader units: one of X per warp, one of Y in warps 8 .. 15
    Unit ux, uy;
    if (T.xks == 1) { ux.row = warp * 8 + (lane & 7); ux.q = lane >> 3; }
    else { ux.row = (warp >> 2) * 32 + lane; ux.q = warp & 3; }
    ux.ks = T.xks;
    ux.ok = ux.row < nx;
    ux.p = X + (ux.ok ? row_off(x0 + ux.row, T.nx, T.xrs, T.xbs) : 0);
    const int w8 = warp & 7;
    if (T.yks == 1) { uy.row = w8 * 8 + (lane & 7); uy.q = lane >> 3; }
    else { uy.row = (w8 >> 2) * 32 + lane; uy.q = w8 & 3; }
    uy.ks = T.yks;
    uy.ok = warp >= 8 && uy.row < ny;
    uy.p = Y + (uy.ok ? row_off(y0 + uy.row, T.ny, T.yrs, T.ybs) : 0);

    int kb = k0;
    do {
      const int len = max(0, min(KB, k1 - kb));
      const int nst = (len + KS - 1) / KS;
      if (tid < TM + TN) rmax[tid] = 0;
      for (int i = tid; i < len; i += THREADS) tab[i] = k_col(T, kb + i);
      __syncthreads();
      // row exponents of this block; the last step visited stays in registers
      double vx[8], vy[8];
      uint32_t mx = 0, my = 0;
      for (int s = nst - 1; s >= 0; --s) {
        load_unit(ux, tab + s * KS, len - s * KS, vx);
        load_unit(uy, tab + s * KS, len - s * KS, vy);
        mx = unit_max(vx, mx);
        my = unit_max(vy, my);
      }
      if (mx) atomicMax(&rmax[ux.row], mx);
      if (my) atomicMax(&rmax[TM + uy.row], my);
      __syncthreads();
      // rows that hold an infinity, a NaN or nothing but values near the
      // subnormal range go through plain multiply-adds
      bool bad = false;
      if (tid < TM + TN) {
        const uint32_t h = rmax[tid];
        bad = (h >> 20) == 0x7ffu || (h != 0 && (h >> 20) < 64u);
      }
      const bool plain = __syncthreads_or(bad);
      long long ahi[16], alo[16];   // sums of accumulators 0 .. 3 and 4 .. 7
#pragma unroll
      for (int j = 0; j < 16; ++j) ahi[j] = alo[j] = 0;
      const bool mine = quarter * 32 < nx && colq * 16 < ny;
      if (!plain) {
        const int ex = ux.ok ? (int)(rmax[ux.row] >> 20) : 0, ey = uy.ok ? (int)(rmax[TM + uy.row] >> 20) : 0;
        for (int s = 0; s < nst; ++s, ++it) {
          const uint32_t h = it & 1u;
          bool ok = true;
          if (it >= 2) ok = mbar_wait(&bar[h], ((it >> 1) - 1) & 1u, err, 11, wait_ns);
          if (ok) {
            if (ux.ok) store_unit(ux, vx, ex, smem, XPLANE, h);
            if (uy.ok) store_unit(uy, vy, ey, yplanes, YPLANE, h);
          }
          if (s + 1 < nst) {
            load_unit(ux, tab + (s + 1) * KS, len - (s + 1) * KS, vx);
            load_unit(uy, tab + (s + 1) * KS, len - (s + 1) * KS, vy);
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          fence_before();
          if (!__syncthreads_and(ok)) { abort = true; break; }
          const bool chunk_end = s + 1 == nst || (s & (CHUNK - 1)) == CHUNK - 1;
          if (tid == 0) {
            fence_after();
            const uint64_t dx = sdesc(smem + h * 64), dy = sdesc(yplanes + h * 64);
            constexpr uint64_t PX = XPLANE >> 4, PY = YPLANE >> 4;
            const bool fresh = (s & (CHUNK - 1)) == 0;
#pragma unroll
            for (int kk = 0; kk < 2; ++kk) {
              const uint64_t a = dx + 2 * kk, b = dy + 2 * kk;
              // plane pair (i, j) adds to accumulator i + j <= 7: for one i the
              // Y planes lie one after the other, and so do their accumulators
              const uint32_t keep = fresh && kk == 0 ? 0u : 1u;
#pragma unroll
              for (int i = 0; i < PLANES; ++i) {
                const int n = (PLANES - i) * TN;   // columns
                umma<MPSLCC_BF16>(tmem + i * TN, a + i * PX, b, idesc<MPSLCC_BF16>(TM, n < 256 ? n : 256),
                                  i == 0 ? keep : 1u);
                if (n > 256)
                  umma<MPSLCC_BF16>(tmem + i * TN + 256, a + i * PX, b + 4 * PY, idesc<MPSLCC_BF16>(TM, n - 256),
                                    i == 0 ? keep : 1u);
              }
            }
            umma_commit(&bar[h]);
          }
          if (chunk_end) {
            // all products up to this step are done: combine the weights
            if (!mbar_wait(&bar[h], (it >> 1) & 1u, err, 12, wait_ns)) abort = true;
            fence_after();
            if (mine) {
#pragma unroll
              for (int cb = 0; cb < 16; cb += 2) {
                uint32_t v[8][2];
                const uint32_t ta = tmem + ((uint32_t)(quarter * 32) << 16) + colq * 16 + cb;
#pragma unroll
                for (int g = 0; g < 8; ++g) tmem_ld2(ta + g * TN, v[g]);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                  int c[8];
#pragma unroll
                  for (int g = 0; g < 8; ++g) c[g] = __float2int_rn(__uint_as_float(v[g][j]));
                  ahi[cb + j] += (long long)c[0] * (1 << 24) + (long long)c[1] * (1 << 16) + (long long)c[2] * 256 + c[3];
                  alo[cb + j] += (long long)c[4] * (1 << 24) + (long long)c[5] * (1 << 16) + (long long)c[6] * 256 + c[7];
                }
              }
            }
            fence_before();
          }
        }
        abort = __syncthreads_or(abort);
        if (abort) break;
        if (mine) {
          const int exr = (int)(rmax[quarter * 32 + lane] >> 20);
#pragma unroll
          for (int j = 0; j < 16; ++j)
            stg[(quarter * 32 + lane) * STG_LD + colq * 16 + j] =
                to_f64(ahi[j], alo[j], exr + (int)(rmax[TM + colq * 16 + j] >> 20));
        }
      } else {
        for (int e = tid; e < nx * ny; e += THREADS) {
          const int i = e / ny, j = e - i * ny;
          const double* px = X + row_off(x0 + i, T.nx, T.xrs, T.xbs);
          const double* py = Y + row_off(y0 + j, T.ny, T.yrs, T.ybs);
          double s = 0.0;
          for (int k = 0; k < len; ++k) s = fma(px[tab[k] * T.xks], py[tab[k] * T.yks], s);
          stg[i * STG_LD + j] = s;
        }
      }
      __syncthreads();
      // write-out along the direction that is contiguous in memory
      const int pm = put_mode(T, kb == k0);
      if (T.cys == 1) {
        const bool o0 = lane < ny, o1 = lane + 32 < ny;
        const long long c0 = o0 ? row_off(y0 + lane, T.ny, 1, T.cyb) : 0;
        const long long c1 = o1 ? row_off(y0 + lane + 32, T.ny, 1, T.cyb) : 0;
        for (int i = warp; i < nx; i += THREADS / 32) {
          double* r = C + row_off(x0 + i, T.nx, T.cxs, T.cxb);
          if (o0) put(T, pm, r + c0, stg[i * STG_LD + lane]);
          if (o1) put(T, pm, r + c1, stg[i * STG_LD + lane + 32]);
        }
      } else {
        for (int i0 = 0; i0 < nx; i0 += 32) {
          const int i = i0 + lane;
          const long long ci = i < nx ? row_off(x0 + i, T.nx, T.cxs, T.cxb) : 0;
          for (int j = warp; j < ny; j += THREADS / 32)
            if (i < nx) put(T, pm, C + ci + row_off(y0 + j, T.ny, T.cys, T.cyb), stg[i * STG_LD + j]);
        }
      }
      __syncthreads();
      kb += KB;
    } while (kb < k1);
  }
  if (abort && tid == 0) {
    // products already issued read shared and tensor memory: wait for them
    umma_commit(&bar[2]);
    mbar_wait(&bar[2], 0u, err, 13, DRAIN_NS);
  }
  __syncthreads();
  fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

// ---------------------------------------------------------------------------
// FP64-pipe kernel: 32 x 32 output tiles, outputs dense over the threads (no
// multiply-add is issued for padding), each summed in ascending K.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) gemm_f64_small_kernel(const F64Task* __restrict__ tasks, int ntasks,
                                                             long long total) {
  __shared__ double xs[SM_T][SM_T + 1], ys[SM_T][SM_T + 1];   // [k][row]
  const int tid = threadIdx.x;
  for (long long tile = blockIdx.x; tile < total; tile += gridDim.x) {
    const F64Task T = tasks[find_f64(tasks, ntasks, tile)];
    const F64Tile tc = tile_of(T, tile);
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

// A task in the kernels' form.  A batch that shares one operand becomes rows
// of the other (their tiles then fill up whatever the batch's own size), and
// the operand with more rows lies along the tile's long side.
static F64Task make_f64_task(const GemmTask& g) {
  F64Task t;
  std::memset(&t, 0, sizeof(t));
  const bool ta = g.flags & GEMM_TA, tb = g.flags & GEMM_TB;
  t.x = g.A; t.y = g.B; t.c = g.C;
  t.xrs = ta ? 1 : g.lda; t.xks = ta ? g.lda : 1;
  t.yrs = tb ? g.ldb : 1; t.yks = tb ? 1 : g.ldb;
  t.nx = t.mx = g.m;
  t.ny = t.my = g.n;
  t.cxs = g.ldc; t.cys = 1;
  t.batch = g.batch;
  const long long big = 1LL << 30;
  if (g.batch > 1 && g.sB == 0 && (long long)g.batch * g.m < big) {
    t.mx = g.batch * g.m; t.xbs = g.sA; t.cxb = g.sC; t.batch = 1;
  } else if (g.batch > 1 && g.sA == 0 && (long long)g.batch * g.n < big) {
    t.my = g.batch * g.n; t.ybs = g.sB; t.cyb = g.sC; t.batch = 1;
  } else {
    t.xub = g.sA; t.yub = g.sB; t.cub = g.sC;
  }
  t.k = g.kr ? g.kv : g.k;
  t.kr = g.kr;
  t.nkr = g.nkr;
  t.alpha = g.alpha;
  t.beta = g.beta;
  t.ksplit = std::max(1, g.ksplit);
  MPSLCC_REQUIRE(t.ksplit == 1 || g.sK > 0, ST_INTERNAL, "FP64 task split over K without partial offsets");
  t.sK = t.ksplit > 1 ? g.sK : 0;
  t.kchunk = (int)(cdiv(cdiv(std::max(t.k, 1), t.ksplit), 16) * 16);
  if (cdiv(t.my, TM) * cdiv(t.mx, TN) < cdiv(t.mx, TM) * cdiv(t.my, TN)) {
    std::swap(t.x, t.y);
    std::swap(t.xrs, t.yrs); std::swap(t.xks, t.yks); std::swap(t.xbs, t.ybs); std::swap(t.xub, t.yub);
    std::swap(t.nx, t.ny); std::swap(t.mx, t.my);
    std::swap(t.cxs, t.cys); std::swap(t.cxb, t.cyb);
  }
  return t;
}

// Estimated SM clocks of a task's largest tile: a multiply-add instruction of
// the FP64 pipe takes 16 clocks a warp; a tensor-core tile takes about 4000
// for its set-up and write-out, 2400 a step of 32 K values and 1500 a drain
// whatever part of it is used.
static double pipe_clocks(const F64Task& t) {
  const long long kc = std::max(1, std::min(t.k, t.kchunk));
  return 1500.0 + 600.0 * cdiv(kc, SM_T) +
         16.0 * kc * cdiv(std::min<long long>(t.mx, SM_T) * std::min<long long>(t.my, SM_T), 32);
}
static double tc_clocks(const F64Task& t) {
  const long long kc = std::max(1, std::min(t.k, t.kchunk));
  return 4000.0 * cdiv(kc, KB) + 2400.0 * cdiv(kc, KS) + 1500.0 * cdiv(kc, KS * CHUNK);
}
static long long tiles_of(const F64Task& t, int bx, int by) {
  return (long long)t.batch * t.ksplit * cdiv(t.mx, bx) * cdiv(t.my, by);
}

// A launch whose multiply-adds keep the FP64 pipes busy for no longer than a
// tensor-core launch takes to fill and drain (about 10 us; 30 us for the
// longest tile) runs there whole: one launch instead of two, and its sums are
// plain FP64 chains.
static bool pipe_launch(const std::vector<F64Task>& t) {
  double sum = 0;
  for (const auto& x : t) {
    const double c = pipe_clocks(x);
    if (c > 60e3) return false;
    sum += c * tiles_of(x, SM_T, SM_T);
  }
  return sum <= 152 * 20e3;
}

static std::vector<F64Task> f64_tasks(const GemmTask* g, int n) {
  std::vector<F64Task> v;
  v.reserve(n);
  for (int i = 0; i < n; ++i)
    if (g[i].m > 0 && g[i].n > 0 && g[i].batch > 0) v.push_back(make_f64_task(g[i]));
  return v;
}

bool f64_on_pipe(const GemmTask* g, int n) { return pipe_launch(f64_tasks(g, n)); }

// Splits a task list between the two kernels (the one with fewer estimated
// clocks over the task's tiles) and fills the tile counts.
void plan_f64(const GemmTask* g, int n, F64Plan& p) {
  p = F64Plan();
  const std::vector<F64Task> v = f64_tasks(g, n);
  const bool all_small = pipe_launch(v);
  for (F64Task t : v) {
    const bool small =
        all_small || pipe_clocks(t) * tiles_of(t, SM_T, SM_T) <= tc_clocks(t) * tiles_of(t, TM, TN);
    const int bx = small ? SM_T : TM, by = small ? SM_T : TN;
    t.tx = (int)cdiv(t.mx, bx);
    t.ty = (int)cdiv(t.my, by);
    long long& tot = small ? p.tiles_small : p.tiles_tc;
    t.tile0 = tot;
    tot += (long long)t.batch * t.ksplit * t.tx * t.ty;
    (small ? p.small : p.tc).push_back(t);
  }
  p.n_tc = (int)p.tc.size();
  p.n_small = (int)p.small.size();
}

size_t f64_plan_bytes(const F64Plan& p) { return (p.tc.size() + p.small.size()) * sizeof(F64Task); }

// Copies the plan's tasks to device memory at d (f64_plan_bytes of it).
void upload_f64(const F64Plan& p, void* d, cudaStream_t s) {
  if (!p.tc.empty())
    cuda_check(cudaMemcpyAsync(d, p.tc.data(), p.tc.size() * sizeof(F64Task), cudaMemcpyHostToDevice, s),
               "upload FP64 tasks");
  if (!p.small.empty())
    cuda_check(cudaMemcpyAsync((char*)d + p.tc.size() * sizeof(F64Task), p.small.data(),
                               p.small.size() * sizeof(F64Task), cudaMemcpyHostToDevice, s),
               "upload FP64 tasks");
}

int launch_f64(const F64Launch& l, const void* d, int device, int sms, int* err, cudaStream_t s) {
  int n = 0;
  MPSLCC_REQUIRE((l.tiles_tc > 0) == (l.n_tc > 0) && (l.tiles_small > 0) == (l.n_small > 0), ST_INTERNAL,
                 "FP64 task list without its counts");
  if (l.tiles_tc > 0) {
    static std::atomic<bool> attr[MAX_DEV];
    MPSLCC_REQUIRE(device >= 0 && device < MAX_DEV, ST_ARG, "device ordinal out of range");
    if (!attr[device].load(std::memory_order_acquire)) {
      cuda_check(cudaFuncSetAttribute(gemm_f64_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_TC),
                 "smem attr");
      attr[device].store(true, std::memory_order_release);
    }
    const int grid = (int)std::min<long long>(l.tiles_tc, std::max(1, sms));
    gemm_f64_tc_kernel<<<grid, THREADS, SMEM_TC, s>>>((const F64Task*)d, l.n_tc, l.tiles_tc, err, WAIT_NS);
    ++n;
  }
  if (l.tiles_small > 0) {
    const int grid = (int)std::min<long long>(l.tiles_small, 152LL * 8);
    gemm_f64_small_kernel<<<grid, 256, 0, s>>>((const F64Task*)d + l.n_tc, l.n_small, l.tiles_small);
    ++n;
  }
  return n;
}

}  // namespace mpslcc
