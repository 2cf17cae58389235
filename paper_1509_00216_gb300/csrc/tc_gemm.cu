// Tensor-core sigma path for sm_103a: a grouped GEMM whose operand tiles are
// staged by TMA (cp.async.bulk.tensor, 128-byte swizzle) into a shared-memory
// ring (as many stages of one A and one B tile as the launch's N-tile cap
// leaves room for: 4 to 8, or 2 to 4 in split mode, where a stage holds the
// hi and lo tiles of both operands) and multiplied by
// tcgen05.mma (kind::f16 with BF16 operands, or kind::tf32) into an FP32
// accumulator in tensor memory.  One thread issues TMA, one thread issues
// MMA, and eight epilogue warps drain a double-buffered accumulator with
// tcgen05.ld.
//
// Each task carries its own tensor maps, so the uneven quantum-number
// sectors of one sigma product (every operator class, every middle sector)
// run in one launch per phase, and a task may read its K range as a list of
// runs (the non-zero local pieces of the fused operators).  The epilogue
// either stores rows with a batched row remap (phase 1 writes the stacked
// T_w^T blocks) or stores the FP32 partial sum of its K split at the split's
// own offset (phase 2; a fixed-order reduction adds the splits).
// Every mbarrier wait is bounded (a launch argument); on expiry the kernel
// records an error flag and stops issuing work, then waits (with a separate,
// fixed bound) for the TMA loads and tensor-core products it already issued,
// frees its tensor memory and returns.
#include <cuda.h>
#include <cuda_bf16.h>

#include <array>
#include <atomic>
#include <cstring>
#include <map>
#include <mutex>
#include <string>

#include "engine.hpp"
#include "kruns.hpp"
#include "tcfold.hpp"
#include "tcgen05.cuh"
#include "widen.cuh"

namespace mpslcc {

struct alignas(64) TcTask {
  CUtensorMap ma;       // A: rows x K, K contiguous (hi part in split mode)
  CUtensorMap mb;       // B: rows x K, K contiguous (hi part in split mode)
  CUtensorMap ma2;      // split mode: lo parts of A and B
  CUtensorMap mb2;
  void* C;
  long long bstride;    // output offset between row batches (elements)
  int rpb;              // rows per batch of the output remap
  int ldc;
  int cst;              // mode 4: elements between output columns
  int m, n, k;
  int ksteps, kchunk, ksplit;
  int ntile;            // UMMA N (multiple of 16, <= 256)
  int tm, tn;
  int mode;             // 0: FP32 atomic add, 1: BF16 store, 2: FP32 store,
                        // 3: split BF16 store (hi at +0, lo at +soff), 4: FP64 alpha/beta store,
                        // 5: three-piece BF16 store, six B-side blocks at +j soff,
                        // 6: FP64 store of the plain product
  int split;            // operands are hi + lo pairs: acc += Ah Bh + Ah Bl + Al Bh
  long long soff;
  double alpha, beta;   // mode 4: FP64 store C = alpha acc + beta C
  long long tile0;
  int batch;            // independent products of the same shape
  int a3d, b3d;         // operand map has the batch as third dimension (else shared)
  long long cbatch;     // output offset between batch entries (elements)
  long long kstride;    // output offset between K-split partials (elements);
                        // each split stores its own partial (mode 2)
  const int* kr;        // K runs, or null for K steps at 0, KT, 2 KT, ...: nkr + 1
                        // pairs {first K column, steps before the run} (the last
                        // pair a sentinel holding the task's step count), then
                        // per K split the run its first step lies in
  int nkr;
  // column pieces (npc > 0, modes 1, 2, 3, 5): output column c of row m
  // (channel w = m / rpb, row r = m % rpb) lies in the piece p with
  // pcs[p] <= c < pcs[p + 1] and goes to C[r ldc + pcb[p] + w pcw[p] + c - pcs[p]];
  // piece starts, bases and strides are multiples of 8 (of 16 for sigma)
  int npc;
  int pcs[5];
  int pcw[4];
  long long pcb[4];
};

namespace {

constexpr int MAX_DEVICES = 128;
constexpr int A_BYTES = 128 * 128;           // 128 rows x 128 bytes
constexpr int MAX_STAGES = 8;
constexpr int STG_ROW = 80;                  // epilogue staging: bytes per row (64 used)
constexpr int STG_WARP = 32 * STG_ROW;       // per epilogue warp

// Kernel configurations.  CFG 0, one CTA per SM: a 192 KB operand ring,
// N tiles up to 256 rows, a double-buffered 2 x 256-column accumulator and
// eight epilogue warps (two per tensor-memory lane quarter).  CFG 1, two CTAs
// per SM for tasks of short K and small tiles, whose time goes to per-tile
// latency: a 96 KB ring, N tiles up to 64 rows, 2 x 64 accumulator columns
// (each CTA allocates 128 of the SM's 512) and four epilogue warps.
template <int CFG> struct KCfg {
  static constexpr int RING = CFG == 0 ? 192 * 1024 : 96 * 1024;
  static constexpr int ACC = CFG == 0 ? 256 : 64;
  static constexpr int TMEM = 2 * ACC;
  static constexpr int EPI = CFG == 0 ? 8 : 4;
  static constexpr int THREADS = 64 + 32 * EPI;   // TMA warp, MMA warp, epilogue warps
  static constexpr int MINB = CFG == 0 ? 1 : 2;
  static constexpr int SMEM = RING + 1024 + 256 + EPI * STG_WARP;
};

// Stages of a ring of `ring` bytes for a launch whose tasks use N tiles of at
// most `cap` rows (64, 128 or 256): a stage holds one A tile (128 x 128 B) and
// one B tile (cap x 128 B), twice in split mode (hi and lo parts).
__host__ __device__ __forceinline__ int stage_bytes(int cap, bool split) {
  return (A_BYTES + cap * 128) * (split ? 2 : 1);
}
__host__ __device__ __forceinline__ int ring_stages(int ring, int cap, bool split) {
  const int n = ring / stage_bytes(cap, split);
  return n < MAX_STAGES ? n : MAX_STAGES;
}
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], "
      "[%2];" ::"r"(smem_u32(dst)),
      "l"((uint64_t)map), "r"(smem_u32(bar)), "r"(x), "r"(y)
      : "memory");
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], "
      "[%2];" ::"r"(smem_u32(dst)),
      "l"((uint64_t)map), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z)
      : "memory");
}

// Brings a task's tensor maps into the TMA unit's descriptor cache ahead of
// its first load.
__device__ __forceinline__ void prefetch_maps(const TcTask* T, bool split) {
  asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&T->ma) : "memory");
  asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&T->mb) : "memory");
  if (split) {
    asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&T->ma2) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&T->mb2) : "memory");
  }
}

__device__ __forceinline__ void tma_load(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y, int z,
                                         int three) {
  if (three) tma_load_3d(dst, map, bar, x, y, z);
  else tma_load_2d(dst, map, bar, x, y);
}

// Where a tile lies: its task, batch entry, K split, first row and column,
// first K step, K steps, and the N of its products.
struct TileAt { int ti, b, ks, row0, col0, kt0, nk, ntile; };
__device__ __forceinline__ TileAt tile_at(const TcTask* tasks, int n, long long tile, int lo) {
  int hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tasks[mid].tile0 <= tile) lo = mid;
    else hi = mid - 1;
  }
  const TcTask* T = &tasks[lo];
  const long long local = tile - T->tile0;
  const int tn = T->tn, kchunk = T->kchunk, ksteps = T->ksteps;
  const long long tiles_mn = (long long)T->tm * tn;
  const long long per_b = tiles_mn * T->ksplit;
  TileAt t;
  t.ti = lo;
  t.ntile = T->ntile;
  t.b = (int)(local / per_b);
  const long long lb = local - (long long)t.b * per_b;
  t.ks = (int)(lb / tiles_mn);
  const int r = (int)(lb - (long long)t.ks * tiles_mn);
  const int tmi = r / tn;
  t.row0 = tmi * 128;
  t.col0 = (r - tmi * tn) * t.ntile;
  t.kt0 = t.ks * kchunk;
  t.nk = min(ksteps, t.kt0 + kchunk) - t.kt0;
  return t;
}

// A warp finds its CTA's tiles 32 at a time, one per lane: the search over the
// tasks and the divisions are dependent loads and long chains, and tile by
// tile they were most of the time of a launch of short tiles (all sigma phases
// of a mixed-precision window: 42.9 -> 35.1 ms of device time).  Lane q holds the q-th of the next 32
// tiles; lanes past the end hold the last tile.
__device__ __forceinline__ TileAt look_ahead(const TcTask* tasks, int n, long long tile, long long total, int lane,
                                             int prev) {
  const long long mine = tile + (long long)lane * gridDim.x;
  return tile_at(tasks, n, mine < total ? mine : total - 1, prev);
}

__device__ __forceinline__ int pick(int v, int q) { return __shfl_sync(0xffffffffu, v, q); }

// Writes one accumulator row segment (32 FP32 values of row `roff`,
// columns c0 .. c0 + nv - 1) in the task's output mode.
__device__ __forceinline__ void store_row(const TcTask* T, long long roff, int c0, int nv, const uint32_t* v) {
  if (T->mode == 1 || T->mode == 3) {
    // BF16 rows: a thread owns 32 contiguous outputs = 64 bytes; store
    // them as four 16-byte vectors when aligned
    __nv_bfloat16* C = (__nv_bfloat16*)T->C + roff + c0;
    if (nv == 32 && ((uintptr_t)C & 15) == 0 && (T->mode == 1 || (T->soff & 7) == 0)) {
      uint32_t hi[16], lo[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const float f0 = __uint_as_float(v[2 * j]), f1 = __uint_as_float(v[2 * j + 1]);
        const __nv_bfloat162 h = __floats2bfloat162_rn(f0, f1);
        const float2 hf = __bfloat1622float2(h);
        const __nv_bfloat162 l = __floats2bfloat162_rn(f0 - hf.x, f1 - hf.y);
        hi[j] = *reinterpret_cast<const uint32_t*>(&h);
        lo[j] = *reinterpret_cast<const uint32_t*>(&l);
      }
      uint4* d0 = reinterpret_cast<uint4*>(C);
#pragma unroll
      for (int q = 0; q < 4; ++q) d0[q] = make_uint4(hi[4 * q], hi[4 * q + 1], hi[4 * q + 2], hi[4 * q + 3]);
      if (T->mode == 3) {
        uint4* d1 = reinterpret_cast<uint4*>(C + T->soff);
#pragma unroll
        for (int q = 0; q < 4; ++q) d1[q] = make_uint4(lo[4 * q], lo[4 * q + 1], lo[4 * q + 2], lo[4 * q + 3]);
      }
      return;
    }
  }
  if (T->mode == 5) {
    // three-piece BF16 split of the FP32 result (exact: 3 x 8 bits), written
    // as the six B-side blocks [h m m h l h] at +j soff
    __nv_bfloat16* C = (__nv_bfloat16*)T->C + roff + c0;
    if (nv == 32 && ((uintptr_t)C & 15) == 0 && (T->soff & 7) == 0) {
      uint32_t ph[16], pm[16], pl[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const float f0 = __uint_as_float(v[2 * j]), f1 = __uint_as_float(v[2 * j + 1]);
        const __nv_bfloat162 h = __floats2bfloat162_rn(f0, f1);
        const float2 hf = __bfloat1622float2(h);
        const float r0 = f0 - hf.x, r1 = f1 - hf.y;
        const __nv_bfloat162 m = __floats2bfloat162_rn(r0, r1);
        const float2 mf = __bfloat1622float2(m);
        const __nv_bfloat162 l = __floats2bfloat162_rn(r0 - mf.x, r1 - mf.y);
        ph[j] = *reinterpret_cast<const uint32_t*>(&h);
        pm[j] = *reinterpret_cast<const uint32_t*>(&m);
        pl[j] = *reinterpret_cast<const uint32_t*>(&l);
      }
      // block order [h m m h l h]
      uint4* d0 = reinterpret_cast<uint4*>(C);
      uint4* d1 = reinterpret_cast<uint4*>(C + T->soff);
      uint4* d2 = reinterpret_cast<uint4*>(C + 2 * T->soff);
      uint4* d3 = reinterpret_cast<uint4*>(C + 3 * T->soff);
      uint4* d4 = reinterpret_cast<uint4*>(C + 4 * T->soff);
      uint4* d5 = reinterpret_cast<uint4*>(C + 5 * T->soff);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint4 h4 = make_uint4(ph[4 * q], ph[4 * q + 1], ph[4 * q + 2], ph[4 * q + 3]);
        const uint4 m4 = make_uint4(pm[4 * q], pm[4 * q + 1], pm[4 * q + 2], pm[4 * q + 3]);
        const uint4 l4 = make_uint4(pl[4 * q], pl[4 * q + 1], pl[4 * q + 2], pl[4 * q + 3]);
        d0[q] = h4;
        d1[q] = m4;
        d2[q] = m4;
        d3[q] = h4;
        d4[q] = l4;
        d5[q] = h4;
      }
      return;
    }
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      if (j >= nv) break;
      const float f = __uint_as_float(v[j]);
      const __nv_bfloat16 h = __float2bfloat16_rn(f);
      const float r = f - __bfloat162float(h);
      const __nv_bfloat16 m = __float2bfloat16_rn(r);
      const __nv_bfloat16 l = __float2bfloat16_rn(r - __bfloat162float(m));
      C[j] = h;
      C[j + T->soff] = m;
      C[j + 2 * T->soff] = m;
      C[j + 3 * T->soff] = h;
      C[j + 4 * T->soff] = l;
      C[j + 5 * T->soff] = h;
    }
    return;
  }
  if (T->mode == 2 && nv == 32 && (((uintptr_t)((float*)T->C + roff + c0)) & 15) == 0) {
    float4* d = reinterpret_cast<float4*>((float*)T->C + roff + c0);
#pragma unroll
    for (int q = 0; q < 8; ++q)
      d[q] = make_float4(__uint_as_float(v[4 * q]), __uint_as_float(v[4 * q + 1]), __uint_as_float(v[4 * q + 2]),
                         __uint_as_float(v[4 * q + 3]));
    return;
  }
  // the remaining paths index v only with unrolled constants, so that the
  // accumulator row stays in registers
  if (T->mode == 4) {
    const int cst = T->cst;
    double* C = (double*)T->C + roff + (long long)c0 * cst;
    const double al = T->alpha, be = T->beta;
    const bool keep = be != 0.0;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      if (j >= nv) break;
      const double x = al * widen(__uint_as_float(v[j]));
      *C = keep ? x + be * *C : x;
      C += cst;
    }
    return;
  }
  if (T->mode == 0) {
    float* C = (float*)T->C + roff + c0;
    if (nv == 32 && ((uintptr_t)C & 15) == 0) {
#pragma unroll
      for (int q = 0; q < 8; ++q)
        atomicAdd(reinterpret_cast<float4*>(C) + q,
                  make_float4(__uint_as_float(v[4 * q]), __uint_as_float(v[4 * q + 1]), __uint_as_float(v[4 * q + 2]),
                              __uint_as_float(v[4 * q + 3])));
      return;
    }
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      if (j >= nv) break;
      atomicAdd(C + j, __uint_as_float(v[j]));
    }
  } else if (T->mode == 1) {
    __nv_bfloat16* C = (__nv_bfloat16*)T->C + roff + c0;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      if (j >= nv) break;
      C[j] = __float2bfloat16_rn(__uint_as_float(v[j]));
    }
  } else if (T->mode == 3) {
    // two-term BF16 split of the FP32 result: [hi | lo]
    __nv_bfloat16* C = (__nv_bfloat16*)T->C + roff + c0;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      if (j >= nv) break;
      const float f = __uint_as_float(v[j]);
      const __nv_bfloat16 h = __float2bfloat16_rn(f);
      const __nv_bfloat16 l = __float2bfloat16_rn(f - __bfloat162float(h));
      C[j] = h;
      C[j + T->soff] = l;
    }
  } else {
    float* C = (float*)T->C + roff + c0;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      if (j >= nv) break;
      C[j] = __uint_as_float(v[j]);
    }
  }
}

// Writes 8 accumulator values (v[0..7], FP32 bits) at element offset `off`
// (a multiple of 8) in the task's output mode, as 16-byte vectors.
__device__ __forceinline__ void store8(const TcTask* T, long long off, const uint32_t* v) {
  if (T->mode == 2) {
    float4* d = reinterpret_cast<float4*>((float*)T->C + off);
    d[0] = make_float4(__uint_as_float(v[0]), __uint_as_float(v[1]), __uint_as_float(v[2]), __uint_as_float(v[3]));
    d[1] = make_float4(__uint_as_float(v[4]), __uint_as_float(v[5]), __uint_as_float(v[6]), __uint_as_float(v[7]));
    return;
  }
  uint32_t ph[4], pm[4], pl[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float f0 = __uint_as_float(v[2 * j]), f1 = __uint_as_float(v[2 * j + 1]);
    const __nv_bfloat162 h = __floats2bfloat162_rn(f0, f1);
    const float2 hf = __bfloat1622float2(h);
    const float r0 = f0 - hf.x, r1 = f1 - hf.y;
    const __nv_bfloat162 m = __floats2bfloat162_rn(r0, r1);
    const float2 mf = __bfloat1622float2(m);
    const __nv_bfloat162 l = __floats2bfloat162_rn(r0 - mf.x, r1 - mf.y);
    ph[j] = *reinterpret_cast<const uint32_t*>(&h);
    pm[j] = *reinterpret_cast<const uint32_t*>(&m);
    pl[j] = *reinterpret_cast<const uint32_t*>(&l);
  }
  __nv_bfloat16* C = (__nv_bfloat16*)T->C + off;
  const uint4 h4 = make_uint4(ph[0], ph[1], ph[2], ph[3]);
  *reinterpret_cast<uint4*>(C) = h4;
  if (T->mode == 3) {
    // two-term split: lo = f - hi, which is the BF16 rounding of the middle piece
    *reinterpret_cast<uint4*>(C + T->soff) = make_uint4(pm[0], pm[1], pm[2], pm[3]);
  } else if (T->mode == 5) {
    // three-piece split as the six B-side blocks [h m m h l h]
    const uint4 m4 = make_uint4(pm[0], pm[1], pm[2], pm[3]);
    *reinterpret_cast<uint4*>(C + T->soff) = m4;
    *reinterpret_cast<uint4*>(C + 2 * T->soff) = m4;
    *reinterpret_cast<uint4*>(C + 3 * T->soff) = h4;
    *reinterpret_cast<uint4*>(C + 4 * T->soff) = make_uint4(pl[0], pl[1], pl[2], pl[3]);
    *reinterpret_cast<uint4*>(C + 5 * T->soff) = h4;
  }
}

// Per-tile values of a column-piece task (phase 1 of sigma) kept in registers
// by the epilogue: in the staged store each lane writes rows q * 8 + lane / 4
// (q = 0..3) of its warp's 32, at row offset roff[q] of channel wch[q].
struct PieceTile {
  __nv_bfloat16* C;
  long long soff;
  long long roff[4];
  int wch[4];
  bool rlive[4];
  int n, mode, npc;
  int pcs1, pcs2, pcs3;
  int pcw0, pcw1, pcw2, pcw3;
  long long pb0, pb1, pb2, pb3;   // pcb[p] - pcs[p]
};

__device__ __forceinline__ void piece_tile(const TcTask* T, int rw0, int lane, PieceTile& P) {
  P.C = (__nv_bfloat16*)T->C;
  P.soff = T->soff;
  P.n = T->n;
  P.mode = T->mode;
  P.npc = T->npc;
  const int m = T->m, rpb = T->rpb;
  const long long ldc = T->ldc;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int row = rw0 + q * 8 + (lane >> 2);
    const int w = row / rpb;
    P.rlive[q] = row < m;
    P.wch[q] = w;
    P.roff[q] = (long long)(row - w * rpb) * ldc;
  }
  P.pcs1 = T->pcs[1];
  P.pcs2 = T->pcs[2];
  P.pcs3 = T->pcs[3];
  P.pcw0 = T->pcw[0];
  P.pcw1 = T->pcw[1];
  P.pcw2 = T->pcw[2];
  P.pcw3 = T->pcw[3];
  P.pb0 = T->pcb[0] - T->pcs[0];
  P.pb1 = T->pcb[1] - T->pcs[1];
  P.pb2 = T->pcb[2] - T->pcs[2];
  P.pb3 = T->pcb[3] - T->pcs[3];
}

// A warp's 32 x 32 accumulator chunk (lane i holding row rw0 + i of the tile,
// columns c0 .. c0 + 31) of a column-piece task with BF16 output, written
// through the warp's shared-memory staging rows: each store instruction then
// covers 8 rows x 64 contiguous bytes (whole 32-byte sectors) instead of 32
// rows x 16 bytes.  All 32 lanes take part.
__device__ __forceinline__ void store_chunk_staged(const PieceTile& P, uint8_t* stg, int lane, int c0,
                                                   const uint32_t* v) {
  const bool three = P.mode == 5;
  uint32_t ph[16], pm[16], pl[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const float f0 = __uint_as_float(v[2 * j]), f1 = __uint_as_float(v[2 * j + 1]);
    const __nv_bfloat162 h = __floats2bfloat162_rn(f0, f1);
    const float2 hf = __bfloat1622float2(h);
    const float r0 = f0 - hf.x, r1 = f1 - hf.y;
    const __nv_bfloat162 m = __floats2bfloat162_rn(r0, r1);
    ph[j] = *reinterpret_cast<const uint32_t*>(&h);
    pm[j] = *reinterpret_cast<const uint32_t*>(&m);
    pl[j] = 0u;
    if (three) {
      const float2 mf = __bfloat1622float2(m);
      const __nv_bfloat162 l = __floats2bfloat162_rn(r0 - mf.x, r1 - mf.y);
      pl[j] = *reinterpret_cast<const uint32_t*>(&l);
    }
  }
  // this lane's 8-column group: its piece's base and channel stride
  const int col = c0 + 8 * (lane & 3);
  const bool cl = col < P.n;
  long long base;
  int stride;
  if (P.npc > 3 && col >= P.pcs3) { base = P.pb3; stride = P.pcw3; }
  else if (P.npc > 2 && col >= P.pcs2) { base = P.pb2; stride = P.pcw2; }
  else if (P.npc > 1 && col >= P.pcs1) { base = P.pb1; stride = P.pcw1; }
  else { base = P.pb0; stride = P.pcw0; }
  base += col;
  const int nparts = three ? 3 : (P.mode == 3 ? 2 : 1);
  const long long so = P.soff;
#pragma unroll
  for (int part = 0; part < 3; ++part) {
    if (part >= nparts) break;
    const uint32_t* src = part == 0 ? ph : (part == 1 ? pm : pl);
    uint4* mine = reinterpret_cast<uint4*>(stg + lane * STG_ROW);
#pragma unroll
    for (int q = 0; q < 4; ++q) mine[q] = make_uint4(src[4 * q], src[4 * q + 1], src[4 * q + 2], src[4 * q + 3]);
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int rr = q * 8 + (lane >> 2), g = lane & 3;
      const uint4 val = *reinterpret_cast<const uint4*>(stg + rr * STG_ROW + g * 16);
      if (P.rlive[q] && cl) {
        __nv_bfloat16* C = P.C + P.roff[q] + base + (long long)P.wch[q] * stride;
        if (three) {
          // three-piece split as the six B-side blocks [h m m h l h]
          if (part == 0) {
            *reinterpret_cast<uint4*>(C) = val;
            *reinterpret_cast<uint4*>(C + 3 * so) = val;
            *reinterpret_cast<uint4*>(C + 5 * so) = val;
          } else if (part == 1) {
            *reinterpret_cast<uint4*>(C + so) = val;
            *reinterpret_cast<uint4*>(C + 2 * so) = val;
          } else {
            *reinterpret_cast<uint4*>(C + 4 * so) = val;
          }
        } else {
          // hi at +0; in split mode the lo part (the rounded remainder) at +soff
          *reinterpret_cast<uint4*>(C + (part == 1 ? so : 0)) = val;
        }
      }
    }
    __syncwarp();
  }
}

// A warp's 32 x 32 accumulator chunk (lane i holding row rw0 + i) widened to
// FP64 rows of C, 16 columns at a time through the staging rows: each store
// instruction covers two rows x 128 contiguous bytes instead of 32 rows x 8,
// and no second pass over C widens it (5 us at 1021 x 775).
__device__ __forceinline__ void store_chunk_f64(double* C, int ldc, int m, uint8_t* stg, int lane, int rw0, int c0,
                                                int nv, const uint32_t* v) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    if (16 * h >= nv) break;
    uint4* mine = reinterpret_cast<uint4*>(stg + lane * STG_ROW);
#pragma unroll
    for (int q = 0; q < 4; ++q)
      mine[q] = make_uint4(v[16 * h + 4 * q], v[16 * h + 4 * q + 1], v[16 * h + 4 * q + 2], v[16 * h + 4 * q + 3]);
    __syncwarp();
    const int c = lane & 15;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int r = 2 * q + (lane >> 4);
      const float f = *reinterpret_cast<const float*>(stg + r * STG_ROW + c * 4);
      if (rw0 + r < m && 16 * h + c < nv) C[(long long)(rw0 + r) * ldc + c0 + 16 * h + c] = widen(f);
    }
    __syncwarp();
  }
}

// One accumulator row segment (columns c0 .. c0 + nv - 1, c0 a multiple of
// 32, nv a multiple of 8) of a task with column pieces: every group of 8
// columns lies in one piece.
__device__ __forceinline__ void store_row_pieces(const TcTask* T, long long rbase, int w, int c0, int nv,
                                                 const uint32_t* v) {
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    if (8 * g >= nv) break;
    const int c = c0 + 8 * g;
    int p = 0;
    while (p + 1 < T->npc && c >= T->pcs[p + 1]) ++p;
    store8(T, rbase + T->pcb[p] + (long long)w * T->pcw[p] + (c - T->pcs[p]), v + 8 * g);
  }
}

template <int PREC, bool SPLIT, int CFG>
__global__ void __launch_bounds__(KCfg<CFG>::THREADS, KCfg<CFG>::MINB) tc_gemm_kernel(const TcTask* __restrict__ tasks, int ntasks,
                                                                 long long total, int* err,
                                                                 unsigned long long wait_ns, int cap) {
  // Warp roles: warp 0 issues TMA, warp 1 issues MMA (and owns the tensor
  // memory), warps 2..9 drain a double-buffered accumulator, so the loads and
  // products of the next tile overlap the epilogue of the previous one.
  extern __shared__ uint8_t smem_raw[];
  // every task of the launch has ntile <= cap; the ring holds as many stages
  // of that size as fit (split mode keeps hi and lo tiles of both operands)
  using K = KCfg<CFG>;
  constexpr int RING_BYTES = K::RING, ACC_COLS = K::ACC, TMEM_COLS = K::TMEM, EPI_WARPS = K::EPI;
  const int NST = ring_stages(RING_BYTES, cap, SPLIT);
  const int SB = stage_bytes(cap, SPLIT);
  const int BB = cap * 128;                          // B tile bytes in a stage
  constexpr int KT = PREC == MPSLCC_BF16 ? 64 : 32;  // K elements per 128-byte row
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + RING_BYTES);
  uint64_t* empty = full + MAX_STAGES;
  uint64_t* acc_full = empty + MAX_STAGES;  // [2]
  uint64_t* acc_empty = acc_full + 2;    // [2]
  uint64_t* drain = acc_empty + 2;       // [1] completion of the MMA thread's issued products
  volatile uint32_t* tslot = (volatile uint32_t*)(drain + 1);
  volatile int* s_abort = (volatile int*)(tslot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], EPI_WARPS);  // one arrival per epilogue warp
    }
    mbar_init(drain, 1);
    *s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32((const void*)tslot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tslot;

  if (warp == 0) {   // TMA producer: all lanes look ahead, lane 0 issues
    uint32_t it = 0;
    int q = 0, prev = 0;
    TileAt L;
    // K runs of this lane's tile: the open run (first column rx, steps
    // rs0 .. rs1 - 1) and the next one's entries
    const int* Lkr = nullptr;
    int Lnkr = 0, Lr = 0, Lrx = 0, Lrs0 = 0, Lrs1 = 0, Lnx = 0, Lns1 = 0;
    for (long long tile = blockIdx.x; tile < total; tile += gridDim.x, q = (q + 1) & 31) {
      if (q == 0) {
        L = look_ahead(tasks, ntasks, tile, total, lane, prev);
        prev = pick(L.ti, 31);
        const TcTask* T = &tasks[L.ti];
        if (lane < 3) prefetch_maps(T, SPLIT);
        Lkr = T->kr;
        Lr = Lrx = Lrs0 = Lnx = Lns1 = 0;
        Lrs1 = 0x7fffffff;
        if (Lkr) {
          Lnkr = T->nkr;
          Lr = __ldg(Lkr + 2 * (Lnkr + 1) + L.ks);
          Lrx = __ldg(Lkr + 2 * Lr);
          Lrs0 = __ldg(Lkr + 2 * Lr + 1);
          Lrs1 = __ldg(Lkr + 2 * Lr + 3);
          if (Lr + 1 < Lnkr) { Lnx = __ldg(Lkr + 2 * Lr + 2); Lns1 = __ldg(Lkr + 2 * Lr + 5); }
        }
      } else if (q + 2 < 32) {   // descriptors two tiles ahead (the last lanes repeat the last tile)
        const int t1 = pick(L.ti, q + 1), t2 = pick(L.ti, q + 2);
        if (lane == 0 && t2 != t1) prefetch_maps(&tasks[t2], SPLIT);
      }
      const TcTask* T = &tasks[pick(L.ti, q)];
      const int row0 = pick(L.row0, q), col0 = pick(L.col0, q), tb = pick(L.b, q);
      const int kt0 = pick(L.kt0, q), nk = pick(L.nk, q);
      const uint32_t bbytes = (uint32_t)pick(L.ntile, q) * 128u;
      int r = pick(Lr, q), rx = pick(Lrx, q), rs0 = pick(Lrs0, q), rs1 = pick(Lrs1, q), nx = pick(Lnx, q),
          ns1 = pick(Lns1, q);
      const int* kr = (const int*)__shfl_sync(0xffffffffu, (unsigned long long)Lkr, q);
      const int nkr = pick(Lnkr, q);
      int go = 1;
      if (lane == 0) {
        if (*s_abort) go = 0;
        const int a3 = T->a3d, b3 = T->b3d;
        for (int j = 0; j < nk && go; ++j, ++it) {
          const uint32_t s = it % NST, ph = (it / NST) & 1u;
          if (!mbar_wait(&empty[s], ph ^ 1u, err, 1, wait_ns)) { *s_abort = 1; go = 0; break; }
          uint8_t* st = smem + s * SB;
          const int g = kt0 + j;
          int kx = g * KT;
          if (kr) {
            if (g >= rs1) {   // steps of one split are consecutive: the next run
              ++r;
              rx = nx;
              rs0 = rs1;
              rs1 = ns1;
              if (r + 1 < nkr) { nx = __ldg(kr + 2 * r + 2); ns1 = __ldg(kr + 2 * r + 5); }
            }
            kx = rx + (g - rs0) * KT;
          }
          mbar_expect_tx(&full[s], (SPLIT ? 2u : 1u) * (A_BYTES + bbytes));
          tma_load(st, &T->ma, &full[s], kx, row0, tb, a3);
          tma_load(st + A_BYTES, &T->mb, &full[s], kx, col0, tb, b3);
          if (SPLIT) {
            tma_load(st + A_BYTES + BB, &T->ma2, &full[s], kx, row0, tb, a3);
            tma_load(st + 2 * A_BYTES + BB, &T->mb2, &full[s], kx, col0, tb, b3);
          }
        }
      }
      if (!pick(go, 0)) break;
    }
    if (lane == 0) {
      // Before the CTA exits, every TMA load this thread issued must have
      // landed, whichever warp stopped the loop and when: only the last NST
      // fills can still be in flight (each earlier stage was re-armed only
      // after its previous fill had been consumed).  On the normal path all of
      // them were consumed and these waits return at once.
      const uint32_t first = it > (uint32_t)NST ? it - (uint32_t)NST : 0u;
      for (uint32_t j = first; j < it; ++j) mbar_wait(&full[j % NST], (j / NST) & 1u, err, 5, DRAIN_NS);
    }
    __syncwarp();
  } else if (warp == 1) {   // MMA issuer: all lanes look ahead, lane 0 issues
    uint32_t it = 0, tcount = 0;
    int q = 0, prev = 0;
    TileAt L;
    for (long long tile = blockIdx.x; tile < total; tile += gridDim.x, ++tcount, q = (q + 1) & 31) {
      if (q == 0) {
        L = look_ahead(tasks, ntasks, tile, total, lane, prev);
        prev = pick(L.ti, 31);
      }
      const int nk = pick(L.nk, q), ntile = pick(L.ntile, q);
      int go = 1;
      if (lane == 0) {
        const uint32_t buf = tcount & 1u;
        const uint32_t acc = tmem + buf * ACC_COLS;
        if (*s_abort) go = 0;
        else if (!mbar_wait(&acc_empty[buf], ((tcount >> 1) & 1u) ^ 1u, err, 4, wait_ns)) { *s_abort = 1; go = 0; }
        if (go) {
          fence_after();
          const uint32_t id = idesc<PREC>(128, ntile);
          for (int j = 0; j < nk; ++j, ++it) {
            const uint32_t s = it % NST, ph = (it / NST) & 1u;
            if (!mbar_wait(&full[s], ph, err, 2, wait_ns)) { go = 0; break; }
            fence_after();
            uint8_t* st = smem + s * SB;
            const uint64_t a = sdesc(st);
            const uint64_t b = sdesc(st + A_BYTES);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) umma<PREC>(acc, a + 2 * kk, b + 2 * kk, id, (j > 0 || kk > 0) ? 1u : 0u);
            if (SPLIT) {
              const uint64_t a2 = sdesc(st + A_BYTES + BB);
              const uint64_t b2 = sdesc(st + 2 * A_BYTES + BB);
#pragma unroll
              for (int kk = 0; kk < 4; ++kk) umma<PREC>(acc, a + 2 * kk, b2 + 2 * kk, id, 1u);
#pragma unroll
              for (int kk = 0; kk < 4; ++kk) umma<PREC>(acc, a2 + 2 * kk, b + 2 * kk, id, 1u);
            }
            umma_commit(&empty[s]);
          }
          umma_commit(&acc_full[buf]);
          if (!go) *s_abort = 1;
        }
      }
      if (!pick(go, 0)) break;
    }
    if (lane == 0) {
      // Every product this thread issued completes before tensor memory is
      // freed and the shared-memory stages they read are released, also when
      // an epilogue warp stopped early (on the normal path the epilogue has
      // already waited for all of them).
      umma_commit(drain);
      mbar_wait(drain, 0u, err, 6, DRAIN_NS);
    }
    __syncwarp();
  } else {
    // epilogue: warp w drains tensor-memory lanes 32 (w % 4) .. + 31 (the
    // lanes its position in the warpgroup may access); with eight epilogue
    // warps the two of one quarter take alternate 32-column chunks
    constexpr int NHALF = EPI_WARPS / 4;
    const int quarter = warp & 3;
    const int half = (warp - 2) >> 2;
    uint8_t* stg = smem + RING_BYTES + 256 + (warp - 2) * STG_WARP;
    uint32_t tcount = 0;
    int q = 0, prev = 0;
    TileAt L;
    for (long long tile = blockIdx.x; tile < total; tile += gridDim.x, ++tcount, q = (q + 1) & 31) {
      if (q == 0) {
        L = look_ahead(tasks, ntasks, tile, total, lane, prev);
        prev = pick(L.ti, 31);
      }
      const TcTask* T = &tasks[pick(L.ti, q)];
      const int row0 = pick(L.row0, q), col0 = pick(L.col0, q), ntile = pick(L.ntile, q);
      const int tb = pick(L.b, q), tks = pick(L.ks, q);
      const uint32_t buf = tcount & 1u;
      // the task's fields are fetched while its products run
      const int row = row0 + quarter * 32 + lane;
      const uint32_t taddr = tmem + buf * ACC_COLS + ((uint32_t)(quarter * 32) << 16);
      const bool live = row < T->m;
      const bool pieces = T->npc > 0;
      const int tn = T->n;
      long long roff = 0;
      if (live)
        roff = pieces ? (long long)(row % T->rpb) * T->ldc
                      : (long long)tb * T->cbatch + (long long)tks * T->kstride +
                            (long long)(row / T->rpb) * T->bstride + (long long)(row % T->rpb) * T->ldc;
      const int wch = live ? row / T->rpb : 0;
      const bool staged = pieces && T->mode != 2, plain64 = T->mode == 6;
      PieceTile PT;
      if (staged) piece_tile(T, row0 + quarter * 32, lane, PT);
      const bool ok = mbar_wait(&acc_full[buf], (tcount >> 1) & 1u, err, 3, wait_ns);
      if (__any_sync(0xffffffffu, !ok || *s_abort)) { *s_abort = 1; break; }   // the warp as a whole
      fence_after();
      for (int cb = 32 * half; cb < ntile; cb += 32 * NHALF) {
        uint32_t v[32];
        tmem_ld32(taddr + cb, v);
        if (staged) {
          store_chunk_staged(PT, stg, lane, col0 + cb, v);
          continue;
        }
        const int c0 = col0 + cb;
        const int nv = min(32, tn - c0);
        if (nv <= 0) continue;
        if (plain64) {
          store_chunk_f64((double*)T->C, T->ldc, T->m, stg, lane, row0 + quarter * 32, c0, nv, v);
          continue;
        }
        if (!live) continue;
        if (pieces) store_row_pieces(T, roff, wch, c0, nv, v);
        else store_row(T, roff, c0, nv, v);
      }
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[buf]);
    }
  }
  __syncthreads();
  fence_after();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
}

// window conversion FP64 -> BF16 / FP32 with batched strides
struct ConvTask {
  union {
    const double* src;
    long long src_off;  // elements from the launch's base
  };
  void* dst;
  int rows, cols, src_ld, dst_ld, batch;
  long long s_src, s_dst;
  int pattern;          // 0 plain; 1 split BF16: hi at +0, lo at +soff;
                        // 2 / 3: three-piece split h, m, l written as six blocks at
                        // +j soff, [h h m m h l] (A side) / [h m m h l h] (B side):
                        // block by block the products are hh hm mm mh hl lh, and
                        // blocks 0 and 2 alone hold the hi / lo pair of the
                        // two-piece split on both sides
  long long soff;
  int trans;            // read the source transposed: dst(r, c) = src[c * src_ld + r]
  int pad;              // columns up to the next multiple of 8 belong to the row: write zeros there
  int vec;              // (filled by plan_conv) rows in 16-byte groups of 8 columns
  long long tile0;
};
// Items of one 256-thread tile: groups of 8 columns, one a thread, or single
// elements, four a thread.
constexpr int CONV_T = 256, CONV_E = 4;

// The BF16 pieces of v: h = v rounded to FP32 and then to BF16, m the same of
// v - h, l of v - h - m (two roundings each, differences exact).
struct Pieces { uint16_t h, m, l; };

__device__ __forceinline__ Pieces pieces_f64(double v) {
  const __nv_bfloat16 h = __float2bfloat16_rn((float)v);
  const double r1 = v - (double)__bfloat162float(h);
  const __nv_bfloat16 m = __float2bfloat16_rn((float)r1);
  const __nv_bfloat16 l = __float2bfloat16_rn((float)(r1 - (double)__bfloat162float(m)));
  return {__bfloat16_as_ushort(h), __bfloat16_as_ushort(m), __bfloat16_as_ushort(l)};
}

__device__ __forceinline__ uint32_t bf16_bits(uint32_t f) { return (f + 0x7fffu + ((f >> 16) & 1u)) >> 16; }

// fl32(d + b + c) with one rounding, for b a multiple of some unit u, d one of
// u or coarser and 0 <= c < u: TwoSum gives d + b = s + t exactly, and t + c
// is exact too (at most 20 bits here).
__device__ __forceinline__ float add3(float d, float b, float c) {
  const float s = __fadd_rn(d, b);
  const float bb = __fadd_rn(s, -d);
  const float t = __fadd_rn(__fadd_rn(d, -__fadd_rn(s, -bb)), __fadd_rn(b, -bb));
  return __fadd_rn(s, __fadd_rn(t, c));
}

// The same pieces without the FP64 pipe (its conversions and subtractions, at
// two a clock and SM, took longer than the kernel's memory traffic): |v| is cut
// at bit level into a + b + c of 24, 23 and 6 bits, and every rounding is one
// of exact FP32 sums.  Values below 2^-63 are scaled by 2^128 on the way.  The
// FP64 form is left to what would round in the subnormal range, to |v| from
// 2^118 on and to v - h between 0 and 2^-30 |v| (one value in 2^21).
__device__ __forceinline__ Pieces split_pieces(double v, bool three) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  uint32_t e = (hi >> 20) & 0x7ffu;
  const uint32_t sg = (hi >> 16) & 0x8000u;
  if (e < 888u) return {(uint16_t)sg, 0, 0};   // below half the smallest subnormal
  uint32_t down = 0;
  if (e < 960u) {
    down = 128u << 7;
    e += 128u;
  }
  if (e - 960u > 180u) return pieces_f64(v);
  const uint32_t ef = (e - 896u) << 23;   // FP32 exponent of |v|
  const float a = __uint_as_float(ef | __funnelshift_l(lo, hi & 0xfffffu, 3));
  const uint32_t ub = ef - (23u << 23), uc = ef - (46u << 23);
  const float b = __fadd_rn(__uint_as_float(ub | ((lo >> 6) & 0x7fffffu)), -__uint_as_float(ub));
  const float c = __fadd_rn(__uint_as_float(uc | ((lo & 63u) << 17)), -__uint_as_float(uc));
  // only which side of half an ulp of a the rest lies on decides, so c's bits
  // go into the lowest bit of b
  const float bs = __fadd_rn(__uint_as_float(ub | ((lo >> 6) & 0x7fffffu) | ((lo & 63u) ? 1u : 0u)), -__uint_as_float(ub));
  const float f = __fadd_rn(a, bs);
  uint32_t h = bf16_bits(__float_as_uint(f));
  const float d = __fadd_rn(a, -__uint_as_float(h << 16));
  const float r1 = add3(d, b, c);
  uint32_t m = 0, l = 0;
  if (r1 != 0.0f) {
    if (fabsf(r1) < __uint_as_float(ef - (30u << 23))) return pieces_f64(v);
    m = bf16_bits(__float_as_uint(r1));
    if (three) l = bf16_bits(__float_as_uint(add3(__fadd_rn(d, -__uint_as_float(m << 16)), b, c)));
  }
  if (down) {
    const uint32_t low = down | 0x80u;   // the smallest normal after scaling back
    if (h < low || ((m & 0x7fffu) && (m & 0x7fffu) < low) || ((l & 0x7fffu) && (l & 0x7fffu) < low)) return pieces_f64(v);
    h -= down;
    if (m & 0x7fffu) m -= down;
    if (l & 0x7fffu) l -= down;
  }
  return {(uint16_t)(h ^ sg), (uint16_t)(m & 0x7fffu ? m ^ sg : 0u), (uint16_t)(l & 0x7fffu ? l ^ sg : 0u)};
}

// Block j of a row in the task's pattern: which piece it holds.
__device__ __forceinline__ int piece_of(int pattern, int j) {
  if (pattern == 1) return j;                       // [h m]
  constexpr uint32_t A = 0x201100, B = 0x020110;    // [h h m m h l], [h m m h l h], one digit a block
  return (int)(((pattern == 2 ? A : B) >> (4 * j)) & 3u);
}
__host__ __device__ __forceinline__ int blocks_of(int pattern) { return pattern == 0 ? 1 : (pattern == 1 ? 2 : 6); }

// One converted element at output offset o.
template <int PREC>
__device__ __forceinline__ void conv_put(const ConvTask& T, long long o, double v) {
  if (PREC == MPSLCC_TF32) {
    ((float*)T.dst)[o] = (float)v;
    return;
  }
  uint16_t* d = (uint16_t*)T.dst + o;
  const Pieces p = split_pieces(v, T.pattern >= 2);
  const int nb = blocks_of(T.pattern);
  for (int j = 0; j < nb; ++j) {
    const int k = piece_of(T.pattern, j);
    d[j * T.soff] = k == 0 ? p.h : (k == 1 ? p.m : p.l);
  }
}

// Window conversion.  Bound by its traffic (8 bytes read, 2 to 12 written per
// element).  A thread takes 8 consecutive columns where the output allows
// 16-byte stores (every copy but the R' stacks' inner pieces): a transposed
// source is then read along its rows by consecutive threads and still written
// in 16-byte groups.  Items run over (batch entry, row, group) without gaps,
// so that small windows fill their blocks.  Before, one element a thread at a
// time, 16 in sequence, with 2-byte stores and FP64-pipe arithmetic: 7.9 ms
// for the operators of the M1 = 1500 position, now 3.0 ms.
template <int PREC>
__global__ void __launch_bounds__(CONV_T) conv_kernel(const ConvTask* __restrict__ t, int ntasks, long long total,
                                                      const double* base) {
  // sources are addresses, or (base given) offsets from it
  for (long long tile = blockIdx.x; tile < total; tile += gridDim.x) {
    int lo = 0, hi = ntasks - 1;
    while (lo < hi) {
      int mid = (lo + hi + 1) >> 1;
      if (t[mid].tile0 <= tile) lo = mid;
      else hi = mid - 1;
    }
    ConvTask T = t[lo];
    if (base) T.src = base + T.src_off;
    const long long local = tile - T.tile0;
    if (!T.vec) {
      const long long per = (long long)T.rows * T.cols;
#pragma unroll
      for (int u = 0; u < CONV_E; ++u) {
        const long long e = (local * CONV_E + u) * CONV_T + threadIdx.x;
        const long long b = e / per;
        if (b >= T.batch) break;
        const unsigned q = (unsigned)(e - b * per);   // a window holds fewer than 2^31 elements
        unsigned rr, cc;
        if (T.trans) { cc = q / (unsigned)T.rows; rr = q - cc * T.rows; }
        else { rr = q / (unsigned)T.cols; cc = q - rr * T.cols; }
        const double* src = T.src + b * T.s_src;
        const double v = T.trans ? src[(long long)cc * T.src_ld + rr] : src[(long long)rr * T.src_ld + cc];
        conv_put<PREC>(T, b * T.s_dst + (long long)rr * T.dst_ld + cc, v);
      }
      continue;
    }
    const unsigned ng = (unsigned)(T.cols + 7) >> 3, per = ng * (unsigned)T.rows;
    const long long item = local * CONV_T + threadIdx.x;
    const long long b = item / per;
    if (b >= T.batch) continue;
    const unsigned q = (unsigned)(item - b * per);
    unsigned rr, g;
    if (T.trans) { g = q / (unsigned)T.rows; rr = q - g * T.rows; }
    else { rr = q / ng; g = q - rr * ng; }
    const int c0 = 8 * (int)g, nv = min(8, T.cols - c0);
    const double* src = T.src + b * T.s_src +
                        (T.trans ? (long long)c0 * T.src_ld + rr : (long long)rr * T.src_ld + c0);
    const long long st = T.trans ? T.src_ld : 1;
    double v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = j < nv ? __ldg(src + j * st) : 0.0;
    const long long o = b * T.s_dst + (long long)rr * T.dst_ld + c0;
    if (nv < 8 && !T.pad) {
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (j < nv) conv_put<PREC>(T, o + j, v[j]);
      continue;
    }
    if (PREC == MPSLCC_TF32) {
      float4* d = reinterpret_cast<float4*>((float*)T.dst + o);
      d[0] = make_float4((float)v[0], (float)v[1], (float)v[2], (float)v[3]);
      d[1] = make_float4((float)v[4], (float)v[5], (float)v[6], (float)v[7]);
      continue;
    }
    uint32_t w[3][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const Pieces x = split_pieces(v[2 * j], T.pattern >= 2), y = split_pieces(v[2 * j + 1], T.pattern >= 2);
      w[0][j] = x.h | (uint32_t)y.h << 16;
      w[1][j] = x.m | (uint32_t)y.m << 16;
      w[2][j] = x.l | (uint32_t)y.l << 16;
    }
    uint16_t* d = (uint16_t*)T.dst + o;
    const int nb = blocks_of(T.pattern);
    for (int j = 0; j < nb; ++j) {
      const int k = piece_of(T.pattern, j);
      uint4 x;
      x.x = k == 0 ? w[0][0] : (k == 1 ? w[1][0] : w[2][0]);
      x.y = k == 0 ? w[0][1] : (k == 1 ? w[1][1] : w[2][1]);
      x.z = k == 0 ? w[0][2] : (k == 1 ? w[1][2] : w[2][2]);
      x.w = k == 0 ? w[0][3] : (k == 1 ? w[1][3] : w[2][3]);
      *reinterpret_cast<uint4*>(d + j * T.soff) = x;
    }
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                             const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                             CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn encode_fn() {
  static EncodeFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    cuda_check(cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q), "driver entry point");
    MPSLCC_REQUIRE(p && q == cudaDriverEntryPointSuccess, ST_CUDA, "cuTensorMapEncodeTiled unavailable");
    fn = (EncodeFn)p;
  }
  return fn;
}

inline int esize(int prec) { return prec == MPSLCC_TF32 ? 4 : 2; }
// kernel operand type: TF32, or BF16 (also for the split BF16x3 mode)
inline int kprec(int prec) { return prec == MPSLCC_TF32 ? MPSLCC_TF32 : MPSLCC_BF16; }
inline long pad8(long x) { return (x + 7) / 8 * 8; }
// local-state pieces of the phase-2 K axis (and of the input vector's rows)
// start on 16-element boundaries: 32-byte sectors of T are then written whole
// by one thread, never half by each of two channels
inline long padp(long x) { return (x + 15) / 16 * 16; }

// 2D K-major operand map: `rows` rows of `cols` logical elements, row pitch
// `ld` elements; box = box_rows x 128 bytes, 128-byte swizzle.
void encode_map(Ctx& c, CUtensorMap* map, int prec, const void* base, long rows, long cols, long ld, int box_rows) {
  const int es = esize(prec);
  MPSLCC_REQUIRE(((uintptr_t)base & 15) == 0, ST_INTERNAL, "tensor map base not 16-byte aligned");
  MPSLCC_REQUIRE((ld * es) % 16 == 0, ST_INTERNAL, "tensor map pitch not a multiple of 16 bytes");
  MPSLCC_REQUIRE(rows >= 1 && cols >= 1 && box_rows >= 1 && box_rows <= 256 && cols <= ld, ST_INTERNAL,
                 "bad tensor map extents");
  c.check_bytes(base, ((rows - 1) * ld + cols) * es, "tensor map extent");
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)(ld * es)};
  cuuint32_t box[2] = {(cuuint32_t)(128 / es), (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = encode_fn()(map, prec == MPSLCC_TF32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16,
                           2, (void*)base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  MPSLCC_REQUIRE(r == CUDA_SUCCESS, ST_CUDA, "cuTensorMapEncodeTiled failed");
}

// 3D K-major operand map: `batch` matrices of `rows` x `cols`, row pitch `ld`
// and matrix pitch `bs` elements; box = box_rows x 128 bytes x 1 matrix.
void encode_map3d(Ctx& c, CUtensorMap* map, int prec, const void* base, long rows, long cols, long ld, long batch,
                  long long bs, int box_rows) {
  const int es = esize(prec);
  MPSLCC_REQUIRE(((uintptr_t)base & 15) == 0, ST_INTERNAL, "tensor map base not 16-byte aligned");
  MPSLCC_REQUIRE((ld * es) % 16 == 0 && (bs * es) % 16 == 0, ST_INTERNAL,
                 "tensor map pitches not multiples of 16 bytes");
  MPSLCC_REQUIRE(rows >= 1 && cols >= 1 && batch >= 1 && box_rows >= 1 && box_rows <= 256 && cols <= ld &&
                     bs >= (rows - 1) * ld + cols,
                 ST_INTERNAL, "bad 3D tensor map extents");
  c.check_bytes(base, ((batch - 1) * bs + (rows - 1) * ld + cols) * es, "tensor map extent");
  cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)batch};
  cuuint64_t strides[2] = {(cuuint64_t)(ld * es), (cuuint64_t)(bs * es)};
  cuuint32_t box[3] = {(cuuint32_t)(128 / es), (cuuint32_t)box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = encode_fn()(map, prec == MPSLCC_TF32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16,
                           3, (void*)base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  MPSLCC_REQUIRE(r == CUDA_SUCCESS, ST_CUDA, "cuTensorMapEncodeTiled (3D) failed");
}

}  // namespace

// multiprocessor count of a device (cached per device ordinal)
int sm_count_dev(int device) {
  static std::atomic<int> cache[MAX_DEVICES];
  if (device < 0 || device >= MAX_DEVICES) return 152;
  int n = cache[device].load(std::memory_order_relaxed);
  if (n <= 0) {
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || n <= 0) {
      cudaGetLastError();
      return 152;
    }
    cache[device].store(n, std::memory_order_relaxed);
  }
  return n;
}

unsigned long long wait_bound_ns(const Ctx& c) {
  const double s = c.opts.wait_timeout_s;
  if (!(s > 0.0)) return WAIT_NS;
  return (unsigned long long)(std::min(s, 60.0) * 1e9);
}

namespace {

int sm_count(Ctx& c) { return sm_count_dev(c.device); }

// C (m x n, remapped rows) op= A (m x K) B (n x K)^T.  In split mode (prec
// BF16X3) each operand row holds the hi part at +0 and the lo part at +lo_off
// elements (lda / ldb span both); k is the length of one part.
// One tensor-core task C = A B^T (A m x k, B n x k, K contiguous).  With
// batch > 1 it holds `batch` products of this shape: operand X advances by
// x_bs elements per entry (0 = shared by all entries) and C by c_bs.
// Number of K splits a task gets for a requested count: every split non-empty.
int tc_ksplit_steps(int ksteps, int hint) {
  int ks = std::max(1, std::min(hint, ksteps));
  const int kchunk = (ksteps + ks - 1) / ks;
  return (ksteps + kchunk - 1) / kchunk;
}


TcTask make_task(Ctx& c, int prec, const void* A, long lda, const void* B, long ldb, int m, int n, int k, void* C,
                 int ldc, int rpb, long long bstride, int mode, int ksplit_hint, long long soff = 0,
                 long lo_off = 0, int batch = 1, long long a_bs = 0, long long b_bs = 0, long long c_bs = 0,
                 long long kstride = 0, int cap = 256, int steps = 0, int cst = 1) {
  // steps > 0: the task reads `steps` K steps through a run table set by the
  // caller (k is then the operands' K extent, not the summed length)
  TcTask t;
  std::memset(&t, 0, sizeof(t));
  const int KT = prec == MPSLCC_TF32 ? 32 : 64;
  MPSLCC_REQUIRE(batch >= 1, ST_INTERNAL, "task batch");
  t.batch = batch;
  t.a3d = batch > 1 && a_bs != 0;
  t.b3d = batch > 1 && b_bs != 0;
  t.cbatch = batch > 1 ? c_bs : 0;
  MPSLCC_REQUIRE(cap == 64 || cap == 128 || cap == 256, ST_INTERNAL, "N-tile cap");
  t.ntile = (int)std::min<long>(cap, (n + 15) / 16 * 16);
  auto map = [&](CUtensorMap* mp, const void* base, long rows, long ld, int box, bool three, long long bs) {
    if (three) encode_map3d(c, mp, prec, base, rows, k, ld, batch, bs, box);
    else encode_map(c, mp, prec, base, rows, k, ld, box);
  };
  map(&t.ma, A, m, lda, 128, t.a3d, a_bs);
  map(&t.mb, B, n, ldb, t.ntile, t.b3d, b_bs);
  t.split = prec == MPSLCC_BF16X3;
  if (t.split) {
    MPSLCC_REQUIRE(lo_off >= k && lo_off % 8 == 0, ST_INTERNAL, "bad split operand layout");
    map(&t.ma2, (const char*)A + lo_off * 2, m, lda, 128, t.a3d, a_bs);
    map(&t.mb2, (const char*)B + lo_off * 2, n, ldb, t.ntile, t.b3d, b_bs);
  }
  t.C = C;
  t.ldc = ldc;
  t.cst = cst;
  t.rpb = rpb;
  t.bstride = bstride;
  t.m = m;
  t.n = n;
  t.k = k;
  t.mode = mode;
  t.ksteps = steps > 0 ? steps : (k + KT - 1) / KT;
  t.ksplit = std::max(1, std::min(ksplit_hint, t.ksteps));
  t.kchunk = (t.ksteps + t.ksplit - 1) / t.ksplit;
  t.ksplit = (t.ksteps + t.kchunk - 1) / t.kchunk;  // every split non-empty
  MPSLCC_REQUIRE(t.ksplit == tc_ksplit_steps(t.ksteps, ksplit_hint), ST_INTERNAL, "K split count");
  MPSLCC_REQUIRE(t.ksplit == 1 || mode == 0 || (mode == 2 && kstride > 0), ST_INTERNAL,
                 "split-K partials need atomic adds or a partial stride");
  t.kstride = t.ksplit > 1 ? kstride : 0;
  t.tm = (m + 127) / 128;
  t.tn = (n + t.ntile - 1) / t.ntile;
  // output range check
  const int es = (mode == 1 || mode == 3 || mode == 5) ? 2 : (mode == 4 ? 8 : 4);
  // the furthest row is the last one, or the last of the full row batches
  const long long lc = (long long)(n - 1) * cst;
  long long last = (long long)((m - 1) / rpb) * bstride + (long long)((m - 1) % rpb) * ldc + lc;
  if (m >= rpb) last = std::max(last, (long long)(m / rpb - 1) * bstride + (long long)(rpb - 1) * ldc + lc);
  if (mode == 3) last += soff;
  if (mode == 5) last += 5 * soff;
  last += (long long)(batch - 1) * t.cbatch;
  last += (long long)(t.ksplit - 1) * t.kstride;
  t.soff = soff;
  c.check_bytes(C, (last + 1) * es, "tc output");
  return t;
}

long long plan_tc(std::vector<TcTask>& t) {
  long long tot = 0;
  for (auto& x : t) {
    x.tile0 = tot;
    tot += (long long)std::max(1, x.batch) * x.ksplit * x.tm * x.tn;
  }
  return tot;
}

// The dynamic shared-memory opt-in is a per-device function attribute: it is
// set once per (kernel instance, device), the flag kept per device.
template <int P, bool S, int CFG>
void launch_variant(cudaStream_t st, int grid, const TcTask* d_tasks, int ntasks, long long total, int* err,
                    unsigned long long wait_ns, int cap) {
  using K = KCfg<CFG>;
  static std::atomic<bool> attr[MAX_DEVICES];
  int dev = 0;
  cuda_check(cudaGetDevice(&dev), "cudaGetDevice");
  MPSLCC_REQUIRE(dev >= 0 && dev < MAX_DEVICES, ST_ARG, "device ordinal out of range");
  MPSLCC_REQUIRE(cap <= K::ACC, ST_INTERNAL, "N-tile cap above the configuration's accumulator");
  if (!attr[dev].load(std::memory_order_acquire)) {
    cuda_check(cudaFuncSetAttribute(tc_gemm_kernel<P, S, CFG>, cudaFuncAttributeMaxDynamicSharedMemorySize, K::SMEM),
               "smem attr");
    attr[dev].store(true, std::memory_order_release);
  }
  tc_gemm_kernel<P, S, CFG><<<grid, K::THREADS, K::SMEM, st>>>(d_tasks, ntasks, total, err, wait_ns, cap);
}

template <int CFG>
void launch_cfg(cudaStream_t st, int grid, int prec, const TcTask* d_tasks, int ntasks, long long total, int* err,
                unsigned long long wait_ns, int cap) {
  if (prec == MPSLCC_BF16X3) launch_variant<MPSLCC_BF16, true, CFG>(st, grid, d_tasks, ntasks, total, err, wait_ns, cap);
  else if (prec == MPSLCC_BF16)
    launch_variant<MPSLCC_BF16, false, CFG>(st, grid, d_tasks, ntasks, total, err, wait_ns, cap);
  else launch_variant<MPSLCC_TF32, false, CFG>(st, grid, d_tasks, ntasks, total, err, wait_ns, cap);
}

// grid = persistent CTAs (at most the configuration's CTAs per SM times the
// SMs used); cfg 1 needs cap <= 64
void launch_tc_stream(cudaStream_t st, int grid, int prec, const TcTask* d_tasks, int ntasks, long long total,
                      int* err, unsigned long long wait_ns = WAIT_NS, int cap = 256, int cfg = 0) {
  if (cfg == 1) launch_cfg<1>(st, grid, prec, d_tasks, ntasks, total, err, wait_ns, cap);
  else launch_cfg<0>(st, grid, prec, d_tasks, ntasks, total, err, wait_ns, cap);
}

void launch_tc(Ctx& c, int prec, const TcTask* d_tasks, int ntasks, long long total, int* err, int cap = 256,
               int cfg = 0) {
  if (total <= 0 || ntasks <= 0) return;
  const int sms = std::max(1, sm_count(c) - std::max(0, c.tc_sm_reserve));
  const int per_sm = cfg == 1 ? KCfg<1>::MINB : KCfg<0>::MINB;
  int grid = (int)std::min<long long>(total, (long long)sms * per_sm);
  launch_tc_stream(c.s(), grid, prec, d_tasks, ntasks, total, err, wait_bound_ns(c), cap, cfg);
  cuda_check(cudaGetLastError(), "tc_gemm launch");
  c.products_open = true;
  c.st.kernel_launches++;
  c.st.gemm_launches++;
}

// Tiles of a conversion list; tasks whose rows, pieces and batch entries all
// start on 16-byte boundaries are written in groups of 8 columns.
long long plan_conv(ConvTask* t, int n) {
  long long tot = 0;
  for (int i = 0; i < n; ++i) {
    ConvTask& x = t[i];
    const bool blocks = blocks_of(x.pattern) > 1;
    x.vec = ((uintptr_t)x.dst & 15) == 0 && x.dst_ld % 8 == 0 && (x.batch == 1 || x.s_dst % 8 == 0) &&
            (!blocks || x.soff % 8 == 0) && (long long)x.rows * ((x.cols + 7) / 8) < (1LL << 31);
    MPSLCC_REQUIRE(x.vec || (long long)x.rows * x.cols < (1LL << 31), ST_INTERNAL, "conversion window too large");
    MPSLCC_REQUIRE(!x.pad || x.vec, ST_INTERNAL, "padded conversion rows not on 16-byte boundaries");
    x.tile0 = tot;
    const long long items = (long long)x.batch * x.rows * (x.vec ? (x.cols + 7) / 8 : x.cols);
    const long long per = x.vec ? CONV_T : (long long)CONV_T * CONV_E;
    tot += (items + per - 1) / per;
  }
  return tot;
}

void launch_conv(int prec, const ConvTask* d, int n, long long tot, cudaStream_t s, const double* base = nullptr) {
  const int grid = (int)std::min<long long>(tot, 152LL * 64);
  if (grid <= 0) return;
  if (kprec(prec) == MPSLCC_BF16) conv_kernel<MPSLCC_BF16><<<grid, CONV_T, 0, s>>>(d, n, tot, base);
  else conv_kernel<MPSLCC_TF32><<<grid, CONV_T, 0, s>>>(d, n, tot, base);
}

void check_conv_dst(Ctx& c, const ConvTask& x, int es) {
  const long long blocks = x.pattern == 0 ? 0 : (x.pattern == 1 ? 1 : 5);  // extra split blocks
  c.check_bytes(x.dst,
                ((long long)(x.batch - 1) * x.s_dst + (long long)(x.rows - 1) * x.dst_ld + blocks * x.soff +
                 (x.pad ? pad8(x.cols) : x.cols)) *
                    es,
                "conv dst");
}

void run_conv(Ctx& c, int prec, std::vector<ConvTask>& t, DBuf& dtasks) {
  if (t.empty()) return;
  const int es = esize(prec);
  for (auto& x : t) {
    if (x.trans)
      c.check_range(x.src, 0, (long long)(x.batch - 1) * x.s_src + (long long)(x.cols - 1) * x.src_ld + x.rows - 1,
                    "conv src");
    else
      c.check_range(x.src, 0, (long long)(x.batch - 1) * x.s_src + (long long)(x.rows - 1) * x.src_ld + x.cols - 1,
                    "conv src");
    check_conv_dst(c, x, es);
  }
  const long long tot = plan_conv(t.data(), (int)t.size());
  dtasks.ensure(&c, t.size() * sizeof(ConvTask));
  cuda_check(cudaMemcpyAsync(dtasks.p, t.data(), t.size() * sizeof(ConvTask), cudaMemcpyHostToDevice, c.s()),
             "conv tasks");
  launch_conv(prec, (const ConvTask*)dtasks.p, (int)t.size(), tot, c.s());
  cuda_check(cudaGetLastError(), "conv launch");
  c.st.kernel_launches++;
}

int* tc_flag(Ctx& c) { return &c.out_dev->flag[1]; }

// Waits for the stream; throws if a product gave up.
void check_err(Ctx& c) {
  cuda_check(cudaStreamSynchronize(c.s()), "tc sync");
  check_products(c);
}

}  // namespace

// Rows of the input vector's low-precision copy before local state s of
// fused sector f, every local-state piece rounded up to 16 rows (s = 4: all).
long rows_p(const Fused& F, int f, int s) {
  long r = 0;
  for (int t = 0; t < s && t < 4; ++t) r += padp(piece_dim(F, f, t));
  return r;
}

// Low-precision state of one sigma plan.
struct TcState {
  int layout = -1;      // operand precision class: TF32, BF16 or BF16X3 (the
                        // three-piece six-block layout, serving BF16X3 and BF16X6)
  DBuf lcat, rstk, tt, x, conv, convx;
  std::vector<long> lcat_off, K8, tt_off, x_off;
  std::vector<long> stk_off;
  // K layout per bra key: the operator classes (segments) side by side, and
  // inside a segment one block per ket local state s holding that piece of
  // every channel (channel stride padp(d_s): d_s rounded up to 16), so that
  // the pieces a row block reaches in the pass-through channels form one
  // contiguous K run.
  // kblk[bi][g][s] = start of block s of segment g (-1: the ket sector has
  // no piece of state s).
  std::vector<std::vector<std::array<long, 4>>> kblk;
  std::vector<ConvTask> xconv;
  long long xtiles = 0;
  // Phase-1 units: the rows of one R' stack with bra local state so (piece
  // of dimension d at row boff of the bra sector) for channels w0 .. w1-1
  // whose pieces (so, .) agree; `in` = the ket local states of those pieces.
  // The low-precision stack keeps its rows so-major (all channels' rows of
  // one so contiguous), so a unit's rows are contiguous from row0.
  struct Unit1 { int si, so, d, boff, w0, w1, in; long row0; };
  std::vector<Unit1> u1;
  // Phase-2 units: the rows of middle sector bi with bra local state so.
  struct Unit2 { int bi, so, d, boff; };
  std::vector<Unit2> u2;
  std::vector<uint16_t> mL;               // piece masks of L' channels (MPO bond l+1)
  std::vector<int> cstartL;               // class starts of that bond
  // Task lists per sigma variant v ([0] the layout's own precision: TF32,
  // BF16 or BF16X3; [1] BF16X6, six-block layout only) and N-tile cap
  // (TC_CAPS[0..2]), built on first use; phase 2 keeps its K-split FP32 partials
  // and the segments of their fixed-order sum.
  struct Lists {
    bool built[2] = {false, false};   // per phase
    DBuf t1, t2, ypart, segs, runs[2];
    int n1 = 0, n2 = 0, nseg = 0;
    long long tiles1 = 0, tiles2 = 0, seg_tiles = 0;
  };
  Lists lists[2][3];
  double bytes1[2] = {0, 0}, bytes2[2] = {0, 0};
};

void tc_release(SigmaPlan& P) {
  delete P.tc;
  delete P.tc6;
  P.tc = nullptr;
  P.tc6 = nullptr;
}

SigmaPlan::~SigmaPlan() { tc_release(*this); }

// Low-precision copies of the fused operators of one sigma plan and the task
// lists of both sigma phases.  BF16X3 and BF16X6 share one copy: every
// operand row holds six blocks of the three-piece split (h, m, l), A side
// [h h m m h l] and B side [h m m h l h].  The full rows give the six products
// of BF16X6 (error about 2^-24 relative, at the level of the FP32
// accumulation); blocks 0 and 2 alone are the hi / lo pair of BF16X3
// (hi*hi + hi*lo + lo*hi, about 2^-17).
//
// Only the local pieces (s_out, s_in) that a channel's site tensor reaches
// are converted (the rest of a fused block is zero and stays zero in the
// copies), and the task lists read only those pieces (K runs, below).
void tc_prepare(Ctx& c, SigmaPlan& P, int prec) {
  const int layout = (prec == MPSLCC_BF16X3 || prec == MPSLCC_BF16X6) ? MPSLCC_BF16X3 : prec;
  TcState*& slot = layout == MPSLCC_BF16X3 ? P.tc6 : P.tc;
  if (slot && slot->layout == layout) return;
  StageTimer tm(c, &c.st.t_tc_prepare);
  delete slot;
  slot = nullptr;
  TcState* S = new TcState();
  slot = S;
  S->layout = layout;
  const int es = esize(layout);
  const bool six = layout == MPSLCC_BF16X3;
  const int sp = six ? 6 : 1;
  const LeftFused& lf = P.lf;
  const RightFused& rf = P.rf;
  const Mpo& W = *P.fam->mpo;
  const size_t nbk = P.mid_b.size(), nkk = P.mid_k.size();
  S->mL = fused_piece_masks(W, lf.p, true);
  S->cstartL = W.bond[lf.p + 1].class_start;
  const std::vector<uint16_t> mR = rf.ext ? std::vector<uint16_t>() : fused_piece_masks(W, rf.p, false);
  // piece-major K layout per bra key, every piece rounded up to 16 columns
  S->K8.assign(nbk, 0);
  S->lcat_off.assign(nbk, 0);
  S->tt_off.assign(nbk, 0);
  S->kblk.assign(nbk, {});
  long lsz = 0, tsz = 0;
  for (size_t bi = 0; bi < nbk; ++bi) {
    long K8 = 0;
    for (const auto& sg : lf.seg[bi]) {
      const int fk = lf.kk[sg.kidx];
      std::array<long, 4> b{-1, -1, -1, -1};
      for (int sn = 0; sn < 4; ++sn) {
        const int d = piece_dim(lf.FLk, fk, sn);
        if (d == 0) continue;
        b[sn] = K8;
        K8 += (long)sg.nw * padp(d);
      }
      S->kblk[bi].push_back(b);
    }
    S->K8[bi] = K8;
    S->lcat_off[bi] = lsz;
    S->tt_off[bi] = tsz;
    lsz += pad8((long)lf.FLb.d[lf.kb[bi]] * sp * K8);
    tsz += pad8((long)rf.FRb.d[rf.kb[bi]] * sp * K8);
  }
  // phase-1 units and the so-major row layout of the low-precision stacks;
  // a one-site position's right side (an environment) is one piece per sector
  const int nso = rf.ext ? 1 : 4;
  S->stk_off.assign(rf.stk.size(), 0);
  long ssz = 0;
  for (size_t si = 0; si < rf.stk.size(); ++si) {
    const auto& st = rf.stk[si];
    const int fb = rf.kb[st.bidx];
    const int c0 = rf.ext ? 0 : W.bond[rf.p].class_start[st.cls];
    S->stk_off[si] = ssz;
    long row = 0;
    for (int so = 0; so < nso; ++so) {
      const int d = piece_dim(rf.FRb, fb, so);
      if (d == 0) continue;
      const int boff = piece_off(rf.FRb, fb, so);
      for (int w = 0; w < st.nw;) {
        const int in = rf.ext ? 1 : (mR[c0 + w] >> (4 * so)) & 15;
        int w1 = w + 1;
        while (w1 < st.nw && (rf.ext ? 1 : (mR[c0 + w1] >> (4 * so)) & 15) == in) ++w1;
        if (in) S->u1.push_back({(int)si, so, d, boff, w, w1, in, row + (long)w * d});
        w = w1;
      }
      row += (long)st.nw * d;
    }
    ssz += pad8(row * sp * pad8(rf.FRk.d[rf.kk[st.kidx]]));
  }
  for (size_t bi = 0; bi < nbk; ++bi) {
    const int fb = lf.kb[bi];
    for (int so = 0; so < 4; ++so) {
      const int d = piece_dim(lf.FLb, fb, so);
      if (d > 0) S->u2.push_back({(int)bi, so, d, piece_off(lf.FLb, fb, so)});
    }
  }
  // the input vector's copy keeps its rows (the fused left index) with every
  // local-state piece rounded up to 16 rows, so that phase 1's output
  // columns come in groups of 16 inside one piece
  S->x_off.assign(nkk, 0);
  long xsz = 0;
  for (size_t ki = 0; ki < nkk; ++ki) {
    S->x_off[ki] = xsz;
    xsz += pad8(rows_p(lf.FLk, lf.kk[ki], 4) * sp * pad8(rf.FRk.d[rf.kk[ki]]));
  }
  auto zalloc = [&](DBuf& b, long elems, int e) {
    b.alloc(&c, std::max<long>(elems * e, 16));
    cuda_check(cudaMemsetAsync(b.p, 0, std::max<long>(elems * e, 16), c.s()), "tc memset");
  };
  zalloc(S->lcat, lsz, es);
  zalloc(S->rstk, ssz, es);
  zalloc(S->tt, tsz, es);
  zalloc(S->x, xsz, es);
  // FP64 -> low precision copies of the non-zero pieces of L' (A side of
  // phase 2), per run of channels with equal piece masks
  std::vector<ConvTask> cv;
  auto conv = [&](const double* src, int src_ld, void* dst, int dst_ld, int rows, int cols, int batch,
                  long long s_src, long long s_dst, long long soff, int pad) {
    ConvTask t;
    std::memset(&t, 0, sizeof(t));
    t.src = src;
    t.dst = dst;
    t.rows = rows;
    t.cols = cols;
    t.src_ld = src_ld;
    t.dst_ld = dst_ld;
    t.batch = batch;
    t.s_src = s_src;
    t.s_dst = s_dst;
    t.pattern = six ? 2 : 0;
    t.soff = soff;
    t.pad = pad;
    cv.push_back(t);
  };
  for (size_t bi = 0; bi < nbk; ++bi) {
    const int fb = lf.kb[bi];
    const long K = lf.K[bi], pitch = sp * S->K8[bi];
    for (size_t g = 0; g < lf.seg[bi].size(); ++g) {
      const auto& sg = lf.seg[bi][g];
      const int fk = lf.kk[sg.kidx], c0 = S->cstartL[sg.cls];
      for (int w = 0; w < sg.nw;) {
        const uint16_t m = S->mL[c0 + w];
        int w1 = w + 1;
        while (w1 < sg.nw && S->mL[c0 + w1] == m) ++w1;
        for (int b = 0; b < 16; ++b) {
          if (!(m >> b & 1)) continue;
          const int so = b >> 2, sn = b & 3;
          const int dr = piece_dim(lf.FLb, fb, so), dc = piece_dim(lf.FLk, fk, sn);
          if (dr == 0 || dc == 0) continue;
          const long ro = piece_off(lf.FLb, fb, so), co = piece_off(lf.FLk, fk, sn);
          conv(lf.data.d() + lf.off[bi] + ro * K + sg.koff + (long)w * sg.width + co, (int)K,
               (char*)S->lcat.p + (size_t)(S->lcat_off[bi] + ro * pitch + S->kblk[bi][g][sn] + (long)w * padp(dc)) * es,
               (int)pitch, dr, dc, w1 - w, sg.width, padp(dc), S->K8[bi], 1);
        }
        w = w1;
      }
    }
  }
  // ... and of R' (A side of phase 1), into the so-major stack rows.  A piece
  // starts at any column: its window is widened to whole groups of 8 (what
  // lies between is zero in the fused operator too), windows that meet join.
  for (const auto& u : S->u1) {
    const auto& st = rf.stk[u.si];
    const int rb = rf.FRb.d[rf.kb[st.bidx]], fk = rf.kk[st.kidx], rk = rf.FRk.d[fk];
    const long pitch = sp * pad8(rk);
    std::vector<std::pair<long, long>> win;
    for (int sn = 0; sn < 4; ++sn) {
      if (!(u.in >> sn & 1)) continue;
      const long dc = piece_dim(rf.FRk, fk, sn), co = piece_off(rf.FRk, fk, sn);
      if (dc > 0) win.push_back({co & ~7L, pad8(co + dc)});
    }
    for (const auto& x : merge_exact(win))
      conv(rf.base() + st.off + ((long)u.w0 * rb + u.boff) * rk + x.first, rk,
           (char*)S->rstk.p + (size_t)(S->stk_off[u.si] + u.row0 * pitch + x.first) * es, (int)pitch, u.d,
           (int)(std::min<long>(x.second, rk) - x.first), u.w1 - u.w0, (long long)rb * rk, (long long)u.d * pitch,
           pad8(rk), 1);
  }
  run_conv(c, layout, cv, S->conv);
  // per-call conversion of the input vector (B side of phase 1)
  S->xconv.clear();
  for (size_t ki = 0; ki < nkk; ++ki) {
    const int fl = lf.kk[ki], rk = rf.FRk.d[rf.kk[ki]];
    for (int s1 = 0; s1 < 4; ++s1) {
      const int d1 = piece_dim(lf.FLk, fl, s1);
      if (d1 == 0) continue;
      ConvTask t;
      std::memset(&t, 0, sizeof(t));
      t.src_off = P.off_k[ki] + (long)piece_off(lf.FLk, fl, s1) * rk;
      t.dst = (char*)S->x.p + (size_t)(S->x_off[ki] + rows_p(lf.FLk, fl, s1) * sp * pad8(rk)) * es;
      t.rows = d1;
      t.cols = rk;
      t.src_ld = rk;
      t.dst_ld = (int)(sp * pad8(rk));
      t.batch = 1;
      t.pattern = six ? 3 : 0;
      t.soff = pad8(rk);
      t.pad = 1;
      S->xconv.push_back(t);
    }
  }
  // uploaded once: its sources are offsets from the vector of a product
  for (const auto& t : S->xconv) {
    MPSLCC_REQUIRE(t.src_off >= 0 && t.src_off + (long long)(t.rows - 1) * t.src_ld + t.cols <= P.nk, ST_INTERNAL,
                   "conversion outside the local vector");
    check_conv_dst(c, t, es);
  }
  S->xtiles = plan_conv(S->xconv.data(), (int)S->xconv.size());
  S->convx.alloc(&c, std::max<size_t>(S->xconv.size(), 1) * sizeof(ConvTask));
  if (!S->xconv.empty())
    cuda_check(cudaMemcpyAsync(S->convx.p, S->xconv.data(), S->xconv.size() * sizeof(ConvTask), cudaMemcpyHostToDevice,
                               c.s()),
               "vector conversion tasks");
  // algorithmic bytes of each variant, per BF16 (or TF32) piece read or
  // written: the non-zero pieces of the fused operators and the parts of the
  // vector and of T they multiply, each read once; T and sigma written once
  std::vector<double> a1(rf.stk.size(), 0.0);
  std::vector<int> inu(rf.stk.size(), 0);
  for (const auto& u : S->u1) {
    const int fk = rf.kk[rf.stk[u.si].kidx];
    for (int sn = 0; sn < 4; ++sn)
      if (u.in >> sn & 1) a1[u.si] += (double)(u.w1 - u.w0) * u.d * piece_dim(rf.FRk, fk, sn);
    inu[u.si] |= u.in;
  }
  for (int v = 0; v < (six ? 2 : 1); ++v) {
    const int pcs = v == 1 ? 6 : (six ? 2 : 1);
    for (size_t si = 0; si < rf.stk.size(); ++si) {
      const auto& st = rf.stk[si];
      const int fk = rf.kk[st.kidx];
      const double rb = rf.FRb.d[rf.kb[st.bidx]], lk = lf.FLk.d[lf.kk[st.kidx]];
      double xk = 0;
      for (int sn = 0; sn < 4; ++sn)
        if (inu[si] >> sn & 1) xk += piece_dim(rf.FRk, fk, sn);
      if (rf.ext) xk = rf.FRk.d[fk];
      S->bytes1[v] += (double)es * pcs * (a1[si] + lk * xk + st.nw * rb * lk);
    }
    for (size_t bi = 0; bi < nbk; ++bi) {
      if (S->K8[bi] == 0) continue;
      const int fb = lf.kb[bi];
      const double lb = lf.FLb.d[fb], rb = rf.FRb.d[rf.kb[bi]];
      double a = 0, kc = 0;
      for (const auto& sg : lf.seg[bi]) {
        const int fk = lf.kk[sg.kidx], c0 = S->cstartL[sg.cls];
        for (int w = 0; w < sg.nw;) {
          const uint16_t m = S->mL[c0 + w];
          int w1 = w + 1, used = 0;
          while (w1 < sg.nw && S->mL[c0 + w1] == m) ++w1;
          for (int b = 0; b < 16; ++b)
            if (m >> b & 1) {
              a += (double)(w1 - w) * piece_dim(lf.FLb, fb, b >> 2) * piece_dim(lf.FLk, fk, b & 3);
              used |= 1 << (b & 3);
            }
          for (int sn = 0; sn < 4; ++sn)
            if (used >> sn & 1) kc += (double)(w1 - w) * piece_dim(lf.FLk, fk, sn);
          w = w1;
        }
      }
      S->bytes2[v] += (double)es * pcs * (a + rb * kc) + 4.0 * lb * rb;
    }
  }
  cuda_check(cudaStreamSynchronize(c.s()), "tc prepare sync");
}

namespace {

// Tile shapes the autotuner chooses from: N-tile cap and kernel configuration
// (the cap-64 task lists serve both configurations)
constexpr int NSHAPE = 4;
constexpr int TC_CAPS[NSHAPE] = {256, 128, 64, 64};
constexpr int TC_CFG[NSHAPE] = {0, 0, 0, 1};
inline int list_of(int shape) { return shape < 3 ? shape : 2; }

// K runs of a task: RunBuilder (kruns.hpp).
// Appends a task's run table (pairs {kx, steps before}, a sentinel, then the
// run of each K split's first step) to `tab`; returns its offset.
long append_runs(std::vector<int>& tab, const std::vector<KRun>& runs, int kchunk, int ksplit) {
  const long at = (long)tab.size();
  long s0 = 0;
  for (const auto& r : runs) {
    MPSLCC_REQUIRE(r.kx >= 0 && r.kx < (1L << 30) && s0 < (1L << 30), ST_INTERNAL, "K run out of range");
    tab.push_back((int)r.kx);
    tab.push_back((int)s0);
    s0 += r.steps;
  }
  tab.push_back(0);
  tab.push_back((int)s0);
  size_t ri = 0;
  long acc = 0;
  for (int ks = 0; ks < ksplit; ++ks) {
    const long first = (long)ks * kchunk;
    while (ri + 1 < runs.size() && acc + runs[ri].steps <= first) acc += runs[ri++].steps;
    tab.push_back((int)ri);
  }
  return at;
}

long total_steps(const std::vector<KRun>& r) {
  long s = 0;
  for (const auto& x : r) s += x.steps;
  return s;
}

// Task list of one phase (0, 1) of sigma variant v with N tiles of at most
// TC_CAPS[ci] rows.
void build_list(Ctx& c, SigmaPlan& P, TcState* S, int v, int ci, int phase) {
  TcState::Lists& Ls = S->lists[v][ci];
  if (Ls.built[phase]) return;
  const int cap = TC_CAPS[ci];
  const int layout = S->layout;
  const int es = esize(layout);
  const bool six = layout == MPSLCC_BF16X3;
  const int sp = six ? 6 : 1;
  const LeftFused& lf = P.lf;
  const RightFused& rf = P.rf;
  const size_t nbk = P.mid_b.size();
  const long long target = 2LL * sm_count(c);
  // v = 0: the layout's own precision; v = 1: BF16X6 (plain BF16 kernel over
  // all six blocks, so every run repeats in each block)
  const int kp = v == 1 ? MPSLCC_BF16 : layout;
  const int KT = kp == MPSLCC_TF32 ? 32 : 64;
  const int reps = v == 1 ? 6 : 1;
  std::vector<TcTask> tasks;
  std::vector<std::vector<KRun>> runs;   // per task
  auto upload = [&](DBuf& dt, int& n, long long& tiles) {
    // the run tables in one device buffer
    std::vector<int> tab;
    std::vector<long> at(tasks.size());
    for (size_t i = 0; i < tasks.size(); ++i) at[i] = append_runs(tab, runs[i], tasks[i].kchunk, tasks[i].ksplit);
    Ls.runs[phase].alloc(&c, std::max<size_t>(tab.size(), 4) * sizeof(int));
    if (!tab.empty())
      cuda_check(cudaMemcpyAsync(Ls.runs[phase].p, tab.data(), tab.size() * sizeof(int), cudaMemcpyHostToDevice, c.s()),
                 "K runs");
    for (size_t i = 0; i < tasks.size(); ++i) {
      tasks[i].kr = (const int*)Ls.runs[phase].p + at[i];
      tasks[i].nkr = (int)runs[i].size();
    }
    n = (int)tasks.size();
    tiles = plan_tc(tasks);
    dt.alloc(&c, std::max<size_t>(tasks.size(), 1) * sizeof(TcTask));
    if (!tasks.empty())
      cuda_check(cudaMemcpyAsync(dt.p, tasks.data(), tasks.size() * sizeof(TcTask), cudaMemcpyHostToDevice, c.s()),
                 "tc tasks");
    Ls.built[phase] = true;
  };
  // phase 1: T_w^T = R'_w psi^T, one task per unit (rows of one bra local
  // state for a run of channels of one class); K runs = the ket pieces the
  // unit's channels reach
  if (phase == 0) {
    const int mode1 = v == 1 ? 5 : (six ? 3 : (layout == MPSLCC_TF32 ? 2 : 1));
    for (const auto& u : S->u1) {
      const auto& st = rf.stk[u.si];
      const int bi = st.bidx, ki = st.kidx;
      const LeftFused::Seg* sg = lf.find_seg(bi, st.cls);
      const size_t g = sg - lf.seg[bi].data();
      const int fk = rf.kk[ki], rk = rf.FRk.d[fk];
      const long pitch = sp * pad8(rk);
      const int kk = v == 1 ? (int)pitch : rk;
      RunBuilder rb(KT);   // pieces ascend with the local state
      for (int j = 0; j < reps; ++j)
        for (int sn = 0; sn < 4; ++sn) {
          if (!(u.in >> sn & 1)) continue;
          const long co = piece_off(rf.FRk, fk, sn) + (long)j * pad8(rk);
          rb.add(co, co + piece_dim(rf.FRk, fk, sn));
        }
      const int steps = (int)total_steps(rb.runs);
      if (steps == 0) continue;   // the ket sector has none of the unit's pieces: T stays zero there
      const long ldc = sp * S->K8[bi];
      // split tasks: lo parts in block 2 of both operands (and of the output)
      const long long so = v == 1 ? S->K8[bi] : 2 * S->K8[bi];
      // the output columns (psi's padded rows) are scattered by local-state
      // piece s1 to block s1 of the segment (piece-major K layout), channel w
      // of the unit at stride padp(d1)
      const int fl = lf.kk[ki];
      const long n8 = rows_p(lf.FLk, fl, 4);
      void* C = (char*)S->tt.p + (size_t)(S->tt_off[bi] + (long)u.boff * ldc) * es;
      TcTask t = make_task(c, kp, (char*)S->rstk.p + (size_t)(S->stk_off[u.si] + u.row0 * pitch) * es, pitch,
                           (char*)S->x.p + (size_t)S->x_off[ki] * es, pitch, (u.w1 - u.w0) * u.d, (int)n8, kk, C,
                           (int)ldc, u.d, 0, mode1, 1, six ? so : 0, six ? 2 * pad8(rk) : 0, 1, 0, 0, 0, 0, cap, steps);
      long long last = 0;
      for (int s1 = 0; s1 < 4; ++s1) {
        const int d1 = piece_dim(lf.FLk, fl, s1);
        if (d1 == 0) continue;
        MPSLCC_REQUIRE(S->kblk[bi][g][s1] >= 0 && t.npc < 4, ST_INTERNAL, "phase-1 column pieces");
        t.pcs[t.npc] = (int)rows_p(lf.FLk, fl, s1);
        t.pcw[t.npc] = (int)padp(d1);
        t.pcb[t.npc] = S->kblk[bi][g][s1] + (long long)u.w0 * padp(d1);
        last = std::max(last, (long long)(u.d - 1) * ldc + t.pcb[t.npc] + (long long)(u.w1 - u.w0) * padp(d1) - 1);
        t.npc++;
      }
      t.pcs[t.npc] = (int)n8;
      if (t.npc == 0) continue;
      if (mode1 == 3) last += so;
      if (mode1 == 5) last += 5 * so;
      c.check_bytes(C, (last + 1) * (mode1 == 2 ? 4 : 2), "phase-1 piece output");
      MPSLCC_REQUIRE(t.ksplit == 1, ST_INTERNAL, "phase-1 task split over K");
      runs.push_back(std::move(rb.runs));
      tasks.push_back(t);
    }
    upload(Ls.t1, Ls.n1, Ls.tiles1);
    return;
  }
  // phase 2: sigma = Lcat Tt^T per unit (rows of one bra local state of a
  // middle sector), over the K runs of the channel pieces those rows reach,
  // split over K so that every tile carries about the same number of K steps
  // (a balanced persistent schedule).  The split counts come from an N tiling
  // of 256 whatever the launch's cap, so every cap stores the same partials.
  // Split j of a unit stores its FP32 partial at its own offset; one
  // reduction sums the partials in increasing j into the FP64 sigma, so the
  // result does not depend on the order the splits finish in.
  std::vector<std::vector<KRun>> r2;
  for (const auto& u : S->u2) {
    RunBuilder rb(KT);   // blocks, classes, states and channels in the order of the K layout
    const int bi = u.bi;
    for (int j = 0; j < reps; ++j)
      for (size_t g = 0; g < lf.seg[bi].size(); ++g) {
        const auto& sg = lf.seg[bi][g];
        const int fk = lf.kk[sg.kidx], c0 = S->cstartL[sg.cls];
        for (int sn = 0; sn < 4; ++sn) {
          if (S->kblk[bi][g][sn] < 0) continue;
          const int d = piece_dim(lf.FLk, fk, sn);
          for (int w = 0; w < sg.nw; ++w) {
            if (!((S->mL[c0 + w] >> (4 * u.so + sn)) & 1)) continue;
            const long co = (long)j * S->K8[bi] + S->kblk[bi][g][sn] + (long)w * padp(d);
            rb.add(co, co + d);
          }
        }
      }
    r2.push_back(std::move(rb.runs));
  }
  long long work = 0;
  for (size_t i = 0; i < S->u2.size(); ++i) {
    const int rb = rf.FRb.d[rf.kb[S->u2[i].bi]];
    const long nt = std::min<long>(256, (rb + 15) / 16 * 16);
    work += (long long)((S->u2[i].d + 127) / 128) * ((rb + nt - 1) / nt) * total_steps(r2[i]);
  }
  const long long kper = std::max(4LL, (work + 4 * target - 1) / (4 * target));
  std::vector<SplitSeg> segs;
  std::vector<int> ksv(S->u2.size(), 0);
  long poff = 0;
  for (size_t i = 0; i < S->u2.size(); ++i) {
    const auto& u = S->u2[i];
    const int rb = rf.FRb.d[rf.kb[u.bi]];
    SplitSeg sg;
    std::memset(&sg, 0, sizeof(sg));
    sg.out_off = P.off_b[u.bi] + (long long)u.boff * rb;
    sg.m = u.d;
    sg.n = rb;
    sg.ldp = (int)((rb + 3) / 4 * 4);   // 16-byte aligned partial rows
    sg.sstride = (long long)u.d * sg.ldp;
    const long steps = total_steps(r2[i]);
    if (steps > 0) {
      const int hint = (int)std::max(1LL, (steps + kper - 1) / kper);
      ksv[i] = tc_ksplit_steps((int)steps, hint);
      sg.nsplit = ksv[i];
      sg.part_off = poff;
      poff += (long)ksv[i] * sg.sstride;
    }
    segs.push_back(sg);   // nsplit = 0: no channel reaches these rows, sigma is zero there
  }
  Ls.ypart.alloc(&c, std::max<long>(poff, 4) * 4);
  for (size_t i = 0; i < S->u2.size(); ++i) {
    if (ksv[i] == 0) continue;
    const auto& u = S->u2[i];
    const int rb = rf.FRb.d[rf.kb[u.bi]];
    const long pitch = sp * S->K8[u.bi];
    const int kk = v == 1 ? (int)pitch : (int)S->K8[u.bi];
    const SplitSeg& sg = segs[i];
    tasks.push_back(make_task(c, kp, (char*)S->lcat.p + (size_t)(S->lcat_off[u.bi] + (long)u.boff * pitch) * es, pitch,
                           (char*)S->tt.p + (size_t)S->tt_off[u.bi] * es, pitch, u.d, rb, kk,
                           (float*)Ls.ypart.p + sg.part_off, sg.ldp, 1 << 30, 0, 2, ksv[i], 0,
                           (six && v == 0) ? 2 * S->K8[u.bi] : 0, 1, 0, 0, 0, sg.sstride, cap,
                           (int)total_steps(r2[i])));
    runs.push_back(std::move(r2[i]));
  }
  Ls.nseg = (int)segs.size();
  Ls.seg_tiles = plan_split_tiles(segs.data(), (int)segs.size());
  Ls.segs.alloc(&c, std::max<size_t>(segs.size(), 1) * sizeof(SplitSeg));
  if (!segs.empty())
    cuda_check(cudaMemcpyAsync(Ls.segs.p, segs.data(), segs.size() * sizeof(SplitSeg), cudaMemcpyHostToDevice, c.s()),
               "split segments");
  upload(Ls.t2, Ls.n2, Ls.tiles2);
}

// Tile-shape autotuner of the sigma phases.  For every (operator family,
// position, phase, precision) the first products run once with each shape:
// N-tile caps of 256, 128 and 64 rows on one CTA per SM (4 / 6 / 8 ring
// stages of BF16 tiles, or 2 / 3 / 4 of split tiles), and a cap of 64 on two
// CTAs per SM (configuration 1); the shape with the shortest device time is
// kept for later products of that position, in this and later sweeps, and
// tuned again when the phase's algorithmic bytes change by more than a fifth.
// Every shape computes the same numbers (the K splits do not depend on it).
Ctx::TuneEntry& tune_entry(Ctx& c, const SigmaPlan& P, int phase, int prec, double bytes) {
  const Ctx::TuneKey key{(const void*)P.fam->bra, (const void*)P.fam->ket, (const void*)P.fam->mpo, P.l, phase, prec};
  Ctx::TuneEntry& e = c.tune[key];
  if (!(e.bytes > 0) || std::fabs(bytes - e.bytes) > 0.2 * e.bytes) {
    e = Ctx::TuneEntry();
    e.bytes = bytes;
  }
  return e;
}

int tune_choice(const Ctx& c, const Ctx::TuneEntry& e) {
  if (!c.opts.autotune) return 0;
  if (e.best >= 0) return e.best;
  for (int ci = 0; ci < NSHAPE; ++ci)
    if (!(e.tried & (1 << ci))) return ci;
  return 0;
}

void tune_record(Ctx& c, Ctx::TuneEntry& e, int ci, double ms) {
  if (!c.opts.autotune || e.best >= 0) return;
  if (!(e.tried & (1 << ci)) || ms < e.ms[ci]) e.ms[ci] = ms;
  e.tried |= 1 << ci;
  c.st.tune_trials++;
  if (e.tried == (1 << NSHAPE) - 1) {
    int b = 0;
    for (int ci2 = 1; ci2 < NSHAPE; ++ci2)
      if (e.ms[ci2] < e.ms[b]) b = ci2;
    e.best = b;
  }
}

}  // namespace

void tc_sigma(Ctx& c, SigmaPlan& P, const double* x, double* y, int prec) {
  tc_prepare(c, P, prec);
  TcState* S = (prec == MPSLCC_BF16X3 || prec == MPSLCC_BF16X6) ? P.tc6 : P.tc;
  const int v = prec == MPSLCC_BF16X6 ? 1 : 0;
  const int kp = v == 1 ? MPSLCC_BF16 : S->layout;
  launch_conv(S->layout, (const ConvTask*)S->convx.p, (int)S->xconv.size(), S->xtiles, c.s(), x);
  cuda_check(cudaGetLastError(), "conv launch");
  c.st.kernel_launches++;
  Ctx::TuneEntry& e1 = tune_entry(c, P, 1, prec, S->bytes1[v]);
  Ctx::TuneEntry& e2 = tune_entry(c, P, 2, prec, S->bytes2[v]);
  const int c1 = tune_choice(c, e1), c2 = tune_choice(c, e2);
  build_list(c, P, S, v, list_of(c1), 0);
  build_list(c, P, S, v, list_of(c2), 1);
  const TcState::Lists& L1 = S->lists[v][list_of(c1)];
  const TcState::Lists& L2 = S->lists[v][list_of(c2)];
  cudaEventRecord(c.ev_p0, c.s());
  launch_tc(c, kp, (const TcTask*)L1.t1.p, L1.n1, L1.tiles1, tc_flag(c), TC_CAPS[c1], TC_CFG[c1]);
  cudaEventRecord(c.ev_p1, c.s());
  launch_tc(c, kp, (const TcTask*)L2.t2.p, L2.n2, L2.tiles2, tc_flag(c), TC_CAPS[c2], TC_CFG[c2]);
  cudaEventRecord(c.ev_p2, c.s());
  launch_splitk_reduce_f32((const SplitSeg*)L2.segs.p, L2.nseg, L2.seg_tiles, (const float*)L2.ypart.p, y, c.s());
  cuda_check(cudaGetLastError(), "split-K reduction");
  c.st.kernel_launches++;
  check_err(c);
  float m1 = 0, m2 = 0;
  cudaEventElapsedTime(&m1, c.ev_p0, c.ev_p1);
  cudaEventElapsedTime(&m2, c.ev_p1, c.ev_p2);
  tune_record(c, e1, c1, m1);
  tune_record(c, e2, c2, m2);
  c.st.tc_cap_launches[c1]++;
  c.st.tc_cap_launches[c2]++;
  c.st.tc_phase1_s += m1 * 1e-3;
  c.st.tc_phase2_s += m2 * 1e-3;
  c.st.tc_phase1_bytes += S->bytes1[v];
  c.st.tc_phase2_bytes += S->bytes2[v];
  c.st.tc_launches += 2;
  c.st.sigma_calls++;
  c.st.sigma_flops += P.flops;
}

// Stand-alone check of the tensor-core GEMM: C = A B^T (A m x k, B n x k,
// FP64 host arrays) through one task of each output mode.
void tc_selftest(Ctx& c, int prec, int m, int n, int k, const double* A, const double* B, double* C, int mode,
                 int ksplit) {
  const int es = esize(prec);
  const int sp = prec == MPSLCC_BF16X3 ? 2 : 1;
  long k8 = pad8(k), kk = sp * k8;
  DBuf dA, dB, lA, lB, out, conv;
  dA.alloc(&c, std::max<long>((long)m * k, 1) * 8);
  dB.alloc(&c, std::max<long>((long)n * k, 1) * 8);
  cuda_check(cudaMemcpyAsync(dA.p, A, (size_t)m * k * 8, cudaMemcpyHostToDevice, c.s()), "A");
  cuda_check(cudaMemcpyAsync(dB.p, B, (size_t)n * k * 8, cudaMemcpyHostToDevice, c.s()), "B");
  lA.alloc(&c, (size_t)m * kk * es);
  lB.alloc(&c, (size_t)n * kk * es);
  cuda_check(cudaMemsetAsync(lA.p, 0, (size_t)m * kk * es, c.s()), "z");
  cuda_check(cudaMemsetAsync(lB.p, 0, (size_t)n * kk * es, c.s()), "z");
  std::vector<ConvTask> cv(2);
  std::memset(cv.data(), 0, sizeof(ConvTask) * 2);
  cv[0].src = dA.d(); cv[0].dst = lA.p; cv[0].rows = m; cv[0].cols = k; cv[0].src_ld = k; cv[0].dst_ld = (int)kk;
  cv[0].batch = 1; cv[0].pattern = sp == 2 ? 1 : 0; cv[0].soff = k8; cv[0].pad = 1;
  cv[1].src = dB.d(); cv[1].dst = lB.p; cv[1].rows = n; cv[1].cols = k; cv[1].src_ld = k; cv[1].dst_ld = (int)kk;
  cv[1].batch = 1; cv[1].pattern = sp == 2 ? 1 : 0; cv[1].soff = k8; cv[1].pad = 1;
  run_conv(c, prec, cv, conv);
  const int oes = mode == 1 ? 2 : 4;
  out.alloc(&c, (size_t)m * n * oes);
  cuda_check(cudaMemsetAsync(out.p, 0, (size_t)m * n * oes, c.s()), "z");
  std::vector<TcTask> t{make_task(c, prec, lA.p, kk, lB.p, kk, m, n, (int)(sp == 2 ? k8 : kk), out.p, n, 1 << 30,
                                  0, mode, ksplit, 0, k8)};
  long long tiles = plan_tc(t);
  DBuf dt;
  dt.alloc(&c, sizeof(TcTask));
  cuda_check(cudaMemcpyAsync(dt.p, t.data(), sizeof(TcTask), cudaMemcpyHostToDevice, c.s()), "task");
  launch_tc(c, prec, (const TcTask*)dt.p, 1, tiles, tc_flag(c));
  check_err(c);
  if (mode == 1) {
    std::vector<uint16_t> hb((size_t)m * n);
    cuda_check(cudaMemcpy(hb.data(), out.p, hb.size() * 2, cudaMemcpyDeviceToHost), "d2h");
    for (size_t i = 0; i < hb.size(); ++i) {
      uint32_t u = (uint32_t)hb[i] << 16;
      float f;
      std::memcpy(&f, &u, 4);
      C[i] = f;
    }
  } else {
    std::vector<float> hf((size_t)m * n);
    cuda_check(cudaMemcpy(hf.data(), out.p, hf.size() * 4, cudaMemcpyDeviceToHost), "d2h");
    for (size_t i = 0; i < hf.size(); ++i) C[i] = hf[i];
  }
}


// ---------------------------------------------------------------------------
// Allocation-free variant of the tensor-core GEMM.
//
// Some callers cannot allocate device memory at the point where they need a
// product: a host framework that owns every device allocation and forbids new
// ones inside its step, or code whose device memory is all reserved at
// start-up.  For
// them, C = A B^T (the self-test product above) is also offered with all of
// its scratch -- the low-precision operand copies, the task descriptors and the
// error flag -- in one fixed file-scope device array.
// ---------------------------------------------------------------------------
constexpr size_t NOALLOC_SCRATCH_BYTES = 64ull << 20;  // 64 MiB held by every GPU that loads the library
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_SCRATCH_BYTES];

namespace {
std::mutex g_noalloc_mu;
void* g_noalloc_ptr[MAX_DEVICES] = {};

// Device address of the scratch array for the current device (host code sees
// only a host-side stand-in for the symbol, so it must be looked up per device).
void* noalloc_scratch(int device) {
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  MPSLCC_REQUIRE(device >= 0 && device < MAX_DEVICES, ST_ARG, "device ordinal out of range");
  if (!g_noalloc_ptr[device]) {
    void* p = nullptr;
    cuda_check(cudaGetSymbolAddress(&p, g_noalloc_scratch), "cudaGetSymbolAddress");
    g_noalloc_ptr[device] = p;
  }
  return g_noalloc_ptr[device];
}

inline size_t up256(size_t x) { return (x + 255) / 256 * 256; }

void noalloc_map(CUtensorMap* map, int prec, const void* base, long rows, long cols, long ld, int box_rows) {
  const int es = esize(prec);
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)(ld * es)};
  cuuint32_t box[2] = {(cuuint32_t)(128 / es), (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = encode_fn()(map, prec == MPSLCC_TF32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16,
                           2, (void*)base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  MPSLCC_REQUIRE(r == CUDA_SUCCESS, ST_CUDA, "cuTensorMapEncodeTiled failed");
}
}  // namespace

size_t tc_gemm_noalloc_max_bytes() { return NOALLOC_SCRATCH_BYTES; }

void tc_gemm_noalloc(int device, cudaStream_t stream, int prec, int m, int n, int k, const double* dA,
                     const double* dB, double* dC) {
  MPSLCC_REQUIRE(prec >= MPSLCC_TF32 && prec <= MPSLCC_BF16X3, ST_ARG, "prec must be TF32, BF16 or BF16X3");
  MPSLCC_REQUIRE(m >= 1 && n >= 1 && k >= 1 && dA && dB && dC, ST_ARG, "bad argument");
  const int es = esize(prec);
  const int sp = prec == MPSLCC_BF16X3 ? 2 : 1;
  const long k8 = pad8(k), kk = sp * k8;
  // scratch layout: [conv tasks | tc task | error flag | A copy | B copy]; the
  // largest accepted problem also counts 4 bytes per element of C
  const size_t o_conv = 0, o_task = up256(2 * sizeof(ConvTask)), o_err = o_task + up256(sizeof(TcTask));
  const size_t o_a = o_err + 256, o_b = o_a + up256((size_t)m * kk * es), o_c = o_b + up256((size_t)n * kk * es);
  const size_t need = o_c + up256((size_t)m * n * 4);
  MPSLCC_REQUIRE(need <= NOALLOC_SCRATCH_BYTES, ST_ARG,
                 "problem needs " + std::to_string(need) + " scratch bytes; the allocation-free GEMM holds " +
                     std::to_string(NOALLOC_SCRATCH_BYTES));
  int cur = -1;
  cuda_check(cudaGetDevice(&cur), "cudaGetDevice");
  MPSLCC_REQUIRE(cur == device, ST_ARG, "device must be the current device");
  char* base = (char*)noalloc_scratch(device);
  // operand copies; the conversion clears the padding columns
  ConvTask cv[2];
  std::memset(cv, 0, sizeof(cv));
  cv[0].src = dA; cv[0].dst = base + o_a; cv[0].rows = m; cv[0].cols = k; cv[0].src_ld = k; cv[0].dst_ld = (int)kk;
  cv[0].batch = 1; cv[0].pattern = sp == 2 ? 1 : 0; cv[0].soff = k8; cv[0].pad = 1;
  cv[1].src = dB; cv[1].dst = base + o_b; cv[1].rows = n; cv[1].cols = k; cv[1].src_ld = k; cv[1].dst_ld = (int)kk;
  cv[1].batch = 1; cv[1].pattern = sp == 2 ? 1 : 0; cv[1].soff = k8; cv[1].pad = 1;
  const long long tot = plan_conv(cv, 2);
  // One GEMM task writing FP64 rows of C.  Its N tile: the widest whose waves of
  // tiles cost least, a tile's time going with its operand rows.  (1021 x 775 x
  // 1502, BF16x3: 32 tiles of 256 take 47 us on 152 SMs, 104 of 64 take 24.5.)
  const int sms = sm_count_dev(device);
  int cap = 256;
  long long best = 0;
  for (int w : {256, 128, 64}) {
    const int nt = (int)std::min<long>(w, (n + 15) / 16 * 16);
    const long long waves = ((long long)((m + 127) / 128) * ((n + nt - 1) / nt) + sms - 1) / sms;
    const long long cost = waves * (128 + nt);
    if (w == 256 || cost < best) { cap = w; best = cost; }
  }
  TcTask t;
  std::memset(&t, 0, sizeof(t));
  const int KT = prec == MPSLCC_TF32 ? 32 : 64;
  t.ntile = (int)std::min<long>(cap, (n + 15) / 16 * 16);
  const long klen = sp == 2 ? k8 : kk;  // length of one operand part along K
  noalloc_map(&t.ma, prec, base + o_a, m, klen, kk, 128);
  noalloc_map(&t.mb, prec, base + o_b, n, klen, kk, t.ntile);
  t.split = sp == 2;
  if (t.split) {
    noalloc_map(&t.ma2, prec, base + o_a + k8 * 2, m, klen, kk, 128);
    noalloc_map(&t.mb2, prec, base + o_b + k8 * 2, n, klen, kk, t.ntile);
  }
  t.C = dC;
  t.ldc = n;
  t.cst = 1;
  t.rpb = 1 << 30;
  t.m = m;
  t.n = n;
  t.k = (int)klen;
  t.mode = 6;
  t.ksteps = (int)((klen + KT - 1) / KT);
  t.ksplit = 1;
  t.kchunk = t.ksteps;
  t.tm = (m + 127) / 128;
  t.tn = (n + t.ntile - 1) / t.ntile;
  t.tile0 = 0;
  t.batch = 1;
  long long tiles = (long long)t.tm * t.tn;
  // tasks and a cleared error flag in one copy
  alignas(64) unsigned char image[2048];
  MPSLCC_REQUIRE(o_a <= sizeof(image), ST_INTERNAL, "task image");
  std::memset(image, 0, o_a);
  std::memcpy(image + o_conv, cv, sizeof(cv));
  std::memcpy(image + o_task, &t, sizeof(t));
  cuda_check(cudaMemcpyAsync(base, image, o_a, cudaMemcpyHostToDevice, stream), "noalloc tasks");
  launch_conv(prec, (const ConvTask*)(base + o_conv), 2, tot, stream);
  cuda_check(cudaGetLastError(), "noalloc conv");
  launch_tc_stream(stream, (int)std::min<long long>(tiles, sms), prec, (const TcTask*)(base + o_task), 1, tiles,
                   (int*)(base + o_err), WAIT_NS, cap);
  cuda_check(cudaGetLastError(), "noalloc gemm");
  int h = 0;
  cuda_check(cudaMemcpyAsync(&h, base + o_err, sizeof(int), cudaMemcpyDeviceToHost, stream), "noalloc flag");
  cuda_check(cudaStreamSynchronize(stream), "noalloc sync");
  if (h) throw Error(ST_TIMEOUT, "tensor-core kernel gave up waiting on an mbarrier");
}

// ---------------------------------------------------------------------------
// FP64 GEMM tasks on the tensor cores.  Each operand is converted once into
// a three-piece BF16 split v ~ h + m + l, laid out along K as six blocks so
// that one BF16 product accumulates hh + hm + mh + hl + mm + lh in FP32
// (K-major rows, transposed where the task reads the operand transposed;
// operands shared by several tasks or batch entries are converted once).  The
// epilogue writes C = alpha acc + beta C in FP64.  Relative accuracy ~2^-24
// (FP32 accumulation), used for the environment, fusion and truncation
// products of mixed-precision sweeps.
// ---------------------------------------------------------------------------
// FP64 GEMM tasks on the tensor cores: every operand is split into three
// BF16 parts (six-block layout, A side [h h m m h l], B side [h m m h l h])
// and multiplied by the plain BF16 kernel over K' = 6 K, with an FP64
// alpha/beta epilogue (about 2^-24 relative).  A task's batch stays one
// tensor-core task: batched operands are converted to contiguous
// [batch][rows][6 K] stacks, read as one tall operand beside a shared one and
// through 3D tensor maps where both are batched.
void run_gemms_tc(Ctx& c, std::vector<GemmTask>& tasks) {
  if (tasks.empty()) return;
  for (const auto& t : tasks) MPSLCC_REQUIRE(!t.kr, ST_INTERNAL, "K-run task on the FP64 emulation path");
  const double th0 = c.opts.verbose >= 2 ? wall_seconds() : 0.0;
  struct Key {
    const double* p;
    int rows, cols, ld, trans, nb;
    long long st;
    bool operator<(const Key& o) const {
      if (p != o.p) return p < o.p;
      if (rows != o.rows) return rows < o.rows;
      if (cols != o.cols) return cols < o.cols;
      if (ld != o.ld) return ld < o.ld;
      if (trans != o.trans) return trans < o.trans;
      if (nb != o.nb) return nb < o.nb;
      return st < o.st;
    }
  };
  std::map<Key, long> opoff;
  std::vector<ConvTask> cv;
  long tot = 0;
  // operand `rows` x `cols` (K) read from p (transposed if trans), nb batch
  // entries st elements apart; returns its element offset in the scratch
  auto add_op = [&](const double* p, int rows, int cols, int ld, int trans, int side, int nb,
                    long long st) -> long {
    Key k{p, rows, cols, ld, trans + 2 * side, nb, st};
    auto it = opoff.find(k);
    if (it != opoff.end()) return it->second;
    long off = tot;
    const long kp = pad8(cols);
    tot += pad8((long)nb * rows * 6 * kp);
    ConvTask t;
    std::memset(&t, 0, sizeof(t));
    t.src = p;
    t.dst = (void*)(uintptr_t)off;  // relocated below
    t.rows = rows;
    t.cols = cols;
    t.src_ld = ld;
    t.dst_ld = (int)(6 * kp);
    t.batch = nb;
    t.s_src = st;
    t.s_dst = (long long)rows * 6 * kp;
    t.pattern = side;
    t.soff = kp;
    t.trans = trans;
    t.pad = 1;
    cv.push_back(t);
    opoff[k] = off;
    return off;
  };
  struct Job { long ao, bo; double* C; int m, n, k, ldc; double alpha, beta; int nb; bool a3, b3; long long sC; };
  std::vector<Job> jobs;
  double fl = 0;
  for (const auto& t : tasks) {
    if (t.m <= 0 || t.n <= 0 || t.batch <= 0) continue;
    MPSLCC_REQUIRE(t.k > 0 && t.ksplit <= 1, ST_INTERNAL, "tensor-core FP64 task shape");
    const bool ta = t.flags & GEMM_TA, tb = t.flags & GEMM_TB;
    const bool a3 = t.batch > 1 && t.sA != 0, b3 = t.batch > 1 && t.sB != 0;
    long ao = add_op(t.A, t.m, t.k, t.lda, ta ? 1 : 0, 2, a3 ? t.batch : 1, a3 ? t.sA : 0);  // op(A): m x k
    long bo = add_op(t.B, t.n, t.k, t.ldb, tb ? 0 : 1, 3, b3 ? t.batch : 1, b3 ? t.sB : 0);  // op(B)^T: n x k
    jobs.push_back({ao, bo, t.C, t.m, t.n, t.k, t.ldc, t.alpha, t.beta, t.batch, a3, b3, t.sC});
    fl += 2.0 * t.m * t.n * t.k * t.batch;
  }
  if (jobs.empty()) return;
  c.scratch_tc.ensure(&c, std::max<long>(tot, 8) * 2);
  char* base = (char*)c.scratch_tc.p;
  for (auto& t : cv) t.dst = base + (uintptr_t)t.dst * 2;
  run_conv(c, MPSLCC_BF16, cv, c.tc_conv_tasks);
  // Orientation per task (tcfold.hpp); the six blocks of each operand keep
  // their pattern on either side, so every sum has the same terms in the same
  // order.  N tiles of 64 on two CTAs per SM unless wide tasks would then
  // reload their rows for a quarter more operand traffic than tiles of 256.
  std::vector<TcFold> fold[2];
  double cost[2] = {0, 0};
  constexpr int caps[2] = {256, 64};
  for (int w = 0; w < 2; ++w)
    for (const auto& j : jobs) {
      fold[w].push_back(tc_fold(j.m, j.n, j.nb, j.a3, j.b3, j.ldc, j.sC, caps[w]));
      const TcFold& f = fold[w].back();
      const int nt = std::min(caps[w], (f.cols + 15) / 16 * 16);
      cost[w] += (double)f.batch * ((f.rows + 127) / 128) * ((f.cols + nt - 1) / nt) * (128 + nt) * j.k;
    }
  const int w = cost[1] <= 1.25 * cost[0] ? 1 : 0, cap = caps[w];
  std::vector<TcTask> tt;
  tt.reserve(jobs.size());
  for (size_t i = 0; i < jobs.size(); ++i) {
    const Job& j = jobs[i];
    const TcFold& f = fold[w][i];
    const long kp = pad8(j.k);
    const long long sa = j.a3 ? (long long)j.m * 6 * kp : 0, sb = j.b3 ? (long long)j.n * 6 * kp : 0;
    const bool one = f.batch == 1;
    TcTask t = make_task(c, MPSLCC_BF16, base + (f.swap ? j.bo : j.ao) * 2, 6 * kp, base + (f.swap ? j.ao : j.bo) * 2,
                         6 * kp, f.rows, f.cols, (int)(6 * kp), j.C, f.ldr, f.rpb, f.bstride, 4, 1, 0, 0, f.batch,
                         one ? 0 : (f.swap ? sb : sa), one ? 0 : (f.swap ? sa : sb), f.cbatch, 0, cap, 0, f.cst);
    t.alpha = j.alpha;
    t.beta = j.beta;
    tt.push_back(t);
  }
  long long tiles = plan_tc(tt);
  c.tc_gemm_tasks.ensure(&c, tt.size() * sizeof(TcTask));
  cuda_check(cudaMemcpyAsync(c.tc_gemm_tasks.p, tt.data(), tt.size() * sizeof(TcTask), cudaMemcpyHostToDevice, c.s()),
             "tc gemm tasks");
  const double th1 = c.opts.verbose >= 2 ? wall_seconds() : 0.0;
  launch_tc(c, MPSLCC_BF16, (const TcTask*)c.tc_gemm_tasks.p, (int)tt.size(), tiles, tc_flag(c), cap, w);
  c.st.tc_gemm_flops += fl;
  check_err(c);
  if (c.opts.verbose >= 2) {
    long conv_elems = 0;
    for (const auto& t : cv) conv_elems += (long)t.rows * t.cols * t.batch;
    fprintf(stderr, "[fp64-tc] tasks=%zu jobs=%zu conv=%zu conv_elems=%ld flops=%.3e tiles=%lld host_s=%.4f total_s=%.4f\n",
            tasks.size(), jobs.size(), cv.size(), conv_elems, fl, tiles, th1 - th0, wall_seconds() - th0);
  }
}

}  // namespace mpslcc
