// FP64 device kernels: strided window copies and the BLAS-1 / reduction
// kernels of the iterative solvers.
#include "kernels.hpp"
#include "widen.cuh"

#include <cuda_bf16.h>
#include <algorithm>

namespace mpslcc {

namespace {
constexpr int COPY_CHUNK = 2048;

template <class T>
__device__ __forceinline__ int find_task(const T* t, int n, long long tile) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (t[mid].tile0 <= tile) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

__global__ void copy_f64_kernel(const CopyTask* __restrict__ tasks, int ntasks, long long total) {
  for (long long tile = blockIdx.x; tile < total; tile += gridDim.x) {
    const CopyTask T = tasks[find_task(tasks, ntasks, tile)];
    const long long local = tile - T.tile0;
    const long long nel = (long long)T.rows * T.cols;
    const long long per_batch = (nel + COPY_CHUNK - 1) / COPY_CHUNK;
    const int b = (int)(local / per_batch);
    const long long chunk = local - (long long)b * per_batch;
    const double* src = T.src + (long long)b * T.s_src;
    double* dst = T.dst + (long long)b * T.s_dst;
    const long long e1 = min(nel, (chunk + 1) * COPY_CHUNK);
    for (long long e = chunk * COPY_CHUNK + threadIdx.x; e < e1; e += blockDim.x) {
      const int r = (int)(e / T.cols), c = (int)(e - (long long)r * T.cols);
      const double v = T.alpha * src[(long long)r * T.src_ld + c];
      double* d = dst + (long long)r * T.dst_ld + c;
      *d = T.accumulate ? *d + v : v;
    }
  }
}

// One output per thread and chunk: the serial chain is the sum over splits
// (up to some hundreds), so outputs are what fills the chip.  With 16 outputs
// a thread (4096 a block) a sigma of 1e5 entries ran on 32 blocks: 112 us.
constexpr int SPLIT_CHUNK = 256;

template <class T>
__global__ void __launch_bounds__(SPLIT_CHUNK) splitk_reduce_kernel(const SplitSeg* __restrict__ segs, int nseg,
                                                                    long long total, const T* __restrict__ part,
                                                                    double* __restrict__ out) {
  for (long long tile = blockIdx.x; tile < total; tile += gridDim.x) {
    const SplitSeg* S = segs + find_task(segs, nseg, tile);
    const int n = S->n, ns = S->nsplit;
    const long long nel = (long long)S->m * n, st = S->sstride;
    const long long e = (tile - S->tile0) * SPLIT_CHUNK + threadIdx.x;
    if (e >= nel) continue;
    const int r = (int)(e / n), c = (int)(e - (long long)r * n);
    const T* p = part + S->part_off + (long long)r * S->ldp + c;
    double acc = 0.0;
    int j = 0;
    for (; j + 8 <= ns; j += 8) {
      T x[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) x[q] = __ldg(p + (j + q) * st);
#pragma unroll
      for (int q = 0; q < 8; ++q) acc += widen(x[q]);
    }
    for (; j < ns; ++j) acc += widen(__ldg(p + j * st));
    out[S->out_off + e] = acc;
  }
}

constexpr int RED_BLOCKS = 512, RED_T = 256;

__device__ __forceinline__ double block_sum(double v) {
  __shared__ double sh[RED_T / 32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) sh[w] = v;
  __syncthreads();
  v = (threadIdx.x < (blockDim.x >> 5)) ? sh[threadIdx.x] : 0.0;
  if (w == 0)
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  __syncthreads();
  return v;
}

// Ends a reduction over RED_BLOCKS blocks of RED_T threads.  Every block stores
// its partial sums; the block that finishes last (a ticket counter) adds the
// partials in block order, so the value does not depend on timing.  Short
// vectors launch only the blocks that hold elements; the others' partials are
// the zeros they would have stored.
__device__ __forceinline__ void finish_dots(double s1, double s2, bool two, double* __restrict__ part,
                                            unsigned int* ticket, double* __restrict__ out) {
  s1 = block_sum(s1);
  if (two) s2 = block_sum(s2);
  __shared__ unsigned int tk;
  if (threadIdx.x == 0) {
    part[blockIdx.x] = s1;
    if (two) part[RED_BLOCKS + blockIdx.x] = s2;
    __threadfence();
    tk = atomicAdd(ticket, 1u);
  }
  __syncthreads();
  if (tk != gridDim.x - 1) return;
  __threadfence();
  const volatile double* vp = part;
  double a = 0.0, b = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += RED_T) {
    a += vp[i];
    if (two) b += vp[RED_BLOCKS + i];
  }
  a = block_sum(a);
  if (two) b = block_sum(b);
  if (threadIdx.x == 0) {
    out[0] = a;
    if (two) out[1] = b;
    *ticket = 0u;
  }
}

// The vector steps of the local solvers are bound by their launches and the
// waits between them (2.4 to 11 us each at up to 2e5 elements, five launches
// and two copies a CG iteration), so each is one pass that ends in the dots it
// needs (a six-site program of 1300 local products: 128 -> 110 ms); element i goes to thread i mod (RED_BLOCKS RED_T) in
// ascending order whatever the pass, so every dot keeps its value.
#define RED_LOOP(i, n) \
  for (long i = blockIdx.x * (long)RED_T + threadIdx.x; i < n; i += (long)RED_BLOCKS * RED_T)

// Dots of one or two vector pairs.
__global__ void dot_fused(const double* __restrict__ x1, const double* __restrict__ y1,
                          const double* __restrict__ x2, const double* __restrict__ y2, long n,
                          double* __restrict__ part, unsigned int* ticket, double* __restrict__ out) {
  const bool two = x2 != nullptr;
  double s1 = 0.0, s2 = 0.0;
  RED_LOOP(i, n) {
    s1 = fma(x1[i], y1[i], s1);
    if (two) s2 = fma(x2[i], y2[i], s2);
  }
  finish_dots(s1, s2, two, part, ticket, out);
}

// y -= shift q, then p . y
__global__ void shift_dot_kernel(long n, double shift, const double* __restrict__ q, double* __restrict__ y,
                                 const double* __restrict__ p, double* __restrict__ part, unsigned int* ticket,
                                 double* __restrict__ out) {
  double s = 0.0;
  RED_LOOP(i, n) {
    const double v = fma(-shift, q[i], y[i]);
    y[i] = v;
    s = fma(p[i], v, s);
  }
  finish_dots(s, 0.0, false, part, ticket, out);
}

__device__ __forceinline__ double precond_den(double d, double shift, double fl, int absval) {
  double den = d - shift;
  if (absval) den = fmax(fabs(den), fl);
  else if (fabs(den) < fl) den = (den < 0.0) ? -fl : fl;
  return den;
}

// One CG update: x += alpha p, r -= alpha ap, z = r / max(|d - shift|, fl),
// then r . z and r . r
__global__ void cg_update_kernel(long n, double alpha, const double* __restrict__ p, const double* __restrict__ ap,
                                 double* __restrict__ x, double* __restrict__ r, const double* __restrict__ d,
                                 double shift, double fl, double* __restrict__ z, double* __restrict__ part,
                                 unsigned int* ticket, double* __restrict__ out) {
  double s1 = 0.0, s2 = 0.0;
  RED_LOOP(i, n) {
    x[i] = fma(alpha, p[i], x[i]);
    const double ri = fma(-alpha, ap[i], r[i]);
    const double zi = ri / precond_den(d[i], shift, fl, 1);
    r[i] = ri;
    z[i] = zi;
    s1 = fma(ri, zi, s1);
    s2 = fma(ri, ri, s2);
  }
  finish_dots(s1, s2, true, part, ticket, out);
}

struct LincombArgs { double c[LINCOMB_ARGS]; };

// Ritz vector xs = sum_j c_j V_j and residual r = sum_j c_j AV_j - theta xs, then r . r
__global__ void ritz_kernel(long n, int m, const double* __restrict__ V, const double* __restrict__ AV, long ld,
                            const __grid_constant__ LincombArgs coef, double theta, double* __restrict__ xs,
                            double* __restrict__ r, double* __restrict__ part, unsigned int* ticket,
                            double* __restrict__ out) {
  double s = 0.0;
  RED_LOOP(i, n) {
    double x = 0.0, a = 0.0;
    for (int j = 0; j < m; ++j) {
      x = fma(coef.c[j], V[j * ld + i], x);
      a = fma(coef.c[j], AV[j * ld + i], a);
    }
    a = fma(-theta, x, a);
    xs[i] = x;
    r[i] = a;
    s = fma(a, a, s);
  }
  finish_dots(s, 0.0, false, part, ticket, out);
}

// t -= sum_j c_j V_j with the coefficients on the device
__global__ void gs_kernel(long n, int m, const double* __restrict__ V, long ld, const double* __restrict__ c,
                          double* __restrict__ t) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int j = 0; j < m; ++j) s = fma(-c[j], V[j * ld + i], s);
    t[i] += s;
  }
}

// y += sgn * (*a) x with the coefficient read on the device (no host round trip)
__global__ void axpy_dev_kernel(long n, const double* __restrict__ a, double sgn, const double* __restrict__ x,
                                double* __restrict__ y) {
  const double cf = sgn * *a;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    y[i] = fma(cf, x[i], y[i]);
}

// proj[j] = <V_j, x>: MD_BLOCKS blocks per vector, the last one of each vector
// (a ticket per vector) adds its partials.
constexpr int MD_BLOCKS = 64;
__global__ void multidot_kernel(const double* __restrict__ V, long ld, const double* __restrict__ x, long n,
                                double* __restrict__ part, unsigned int* ticket, double* __restrict__ out) {
  const double* v = V + blockIdx.y * ld;
  double s = 0.0;
  for (long i = blockIdx.x * (long)RED_T + threadIdx.x; i < n; i += (long)MD_BLOCKS * RED_T) s = fma(v[i], x[i], s);
  s = block_sum(s);
  __shared__ unsigned int tk;
  if (threadIdx.x == 0) {
    part[blockIdx.y * MD_BLOCKS + blockIdx.x] = s;
    __threadfence();
    tk = atomicAdd(ticket + blockIdx.y, 1u);
  }
  __syncthreads();
  if (tk != gridDim.x - 1) return;
  __threadfence();
  const volatile double* vp = part + blockIdx.y * MD_BLOCKS;
  double a = threadIdx.x < gridDim.x ? 0.0 + vp[threadIdx.x] : 0.0;
  a = block_sum(a);
  if (threadIdx.x == 0) {
    out[blockIdx.y] = a;
    ticket[blockIdx.y] = 0u;
  }
}

__global__ void axpby_kernel(long n, double a, const double* x, double b, double* y,
                             int mode) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    if (mode == 0) y[i] = fma(a, x[i], y[i]);
    else if (mode == 1) y[i] = a * x[i] + b * y[i];
    else if (mode == 2) y[i] = a * x[i];
    else y[i] = a;
  }
}

__global__ void precond_kernel(long n, const double* __restrict__ x, const double* __restrict__ d, double shift,
                               double fl, double* __restrict__ y, int absval) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    y[i] = x[i] / precond_den(d[i], shift, fl, absval);
  }
}

__global__ void lincomb_kernel(long n, int m, const double* __restrict__ V, long ld,
                               const double* __restrict__ coef, double* __restrict__ out) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int j = 0; j < m; ++j) s = fma(coef[j], V[j * ld + i], s);
    out[i] = s;
  }
}

__global__ void lincomb_args_kernel(long n, int m, const double* __restrict__ V, long ld,
                                    const __grid_constant__ LincombArgs coef, double* __restrict__ out) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int j = 0; j < m; ++j) s = fma(coef.c[j], V[j * ld + i], s);
    out[i] = s;
  }
}

__global__ void gather_kernel(const GatherTask* __restrict__ t, int max_elems) {
  const GatherTask T = t[blockIdx.y];
  const long nel = (long)T.nw * T.n;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < nel; e += (long)gridDim.x * blockDim.x) {
    const int w = (int)(e / T.n), r = (int)(e - (long)w * T.n);
    T.dst[e] = T.src[w * T.sw + r * T.sr];
  }
}

__global__ void take_eigvecs_kernel(const double* __restrict__ V, int n, int m, int right,
                                    double* __restrict__ out) {
  const long nel = (long)n * m;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < nel; e += (long)gridDim.x * blockDim.x) {
    if (!right) {
      const int r = (int)(e / m), j = (int)(e - (long)r * m);
      out[e] = V[r + (long)(n - 1 - j) * n];
    } else {
      const int j = (int)(e / n), c = (int)(e - (long)j * n);
      out[e] = V[c + (long)(n - 1 - j) * n];
    }
  }
}

// x[i] += amp * (u_i - 1/2), u_i uniform from the splitmix64 hash of (seed, i)
__global__ void noise_kernel(long n, double amp, unsigned long long seed, double* __restrict__ x) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    unsigned long long z = seed + (unsigned long long)(i + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    const double u = (double)(z >> 11) * (1.0 / 9007199254740992.0);
    x[i] += amp * (u - 0.5);
  }
}

__global__ void f64_to_bf16_kernel(long n, const double* __restrict__ x, __nv_bfloat16* __restrict__ y) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    y[i] = __float2bfloat16_rn((float)x[i]);
}
__global__ void f64_to_f32_kernel(long n, const double* __restrict__ x, float* __restrict__ y) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    y[i] = (float)x[i];
}
inline int red_grid(long n, int blocks) {
  return (int)std::max(1L, std::min((n + RED_T - 1) / RED_T, (long)blocks));
}
inline int elem_grid(long n) {
  long g = (n + 255) / 256;
  return (int)std::max(1L, std::min(g, 152L * 16));
}
}  // namespace

long long plan_split_tiles(SplitSeg* s, int n) {
  long long tot = 0;
  for (int i = 0; i < n; ++i) {
    s[i].tile0 = tot;
    tot += ((long long)s[i].m * s[i].n + SPLIT_CHUNK - 1) / SPLIT_CHUNK;
  }
  return tot;
}

void launch_splitk_reduce_f32(const SplitSeg* d_segs, int nseg, long long total, const float* part, double* out,
                              cudaStream_t s) {
  if (total <= 0 || nseg <= 0) return;
  int grid = (int)std::min<long long>(total, 152LL * 64);
  splitk_reduce_kernel<float><<<grid, SPLIT_CHUNK, 0, s>>>(d_segs, nseg, total, part, out);
}

void launch_splitk_reduce_f64(const SplitSeg* d_segs, int nseg, long long total, const double* part, double* out,
                              cudaStream_t s) {
  if (total <= 0 || nseg <= 0) return;
  int grid = (int)std::min<long long>(total, 152LL * 64);
  splitk_reduce_kernel<double><<<grid, SPLIT_CHUNK, 0, s>>>(d_segs, nseg, total, part, out);
}

long long plan_copy_tiles(CopyTask* t, int n) {
  long long tot = 0;
  for (int i = 0; i < n; ++i) {
    t[i].tile0 = tot;
    long long nel = (long long)t[i].rows * t[i].cols;
    tot += (long long)t[i].batch * ((nel + COPY_CHUNK - 1) / COPY_CHUNK);
  }
  return tot;
}

void launch_copy_f64(const CopyTask* d_tasks, int ntasks, long long total, cudaStream_t s) {
  if (total <= 0 || ntasks <= 0) return;
  int grid = (int)std::min<long long>(total, 152LL * 16);
  copy_f64_kernel<<<grid, 256, 0, s>>>(d_tasks, ntasks, total);
}

void launch_dot_fused(const double* x1, const double* y1, const double* x2, const double* y2, long n, double* d_out,
                      double* d_part, unsigned int* d_ticket, cudaStream_t s) {
  dot_fused<<<red_grid(n, RED_BLOCKS), RED_T, 0, s>>>(x1, y1, x2, y2, n, d_part, d_ticket, d_out);
}

void launch_shift_dot(long n, double shift, const double* q, double* y, const double* p, const Reduction& R,
                      cudaStream_t s) {
  shift_dot_kernel<<<red_grid(n, RED_BLOCKS), RED_T, 0, s>>>(n, shift, q, y, p, R.part, R.ticket, R.out);
}

void launch_cg_update(long n, double alpha, const double* p, const double* ap, double* x, double* r, const double* d,
                      double shift, double fl, double* z, const Reduction& R, cudaStream_t s) {
  cg_update_kernel<<<red_grid(n, RED_BLOCKS), RED_T, 0, s>>>(n, alpha, p, ap, x, r, d, shift, fl, z, R.part, R.ticket,
                                                             R.out);
}

void launch_ritz(long n, int m, const double* V, const double* AV, long ld, const double* coef, double theta,
                 double* xs, double* r, const Reduction& R, cudaStream_t s) {
  LincombArgs a;
  for (int j = 0; j < LINCOMB_ARGS; ++j) a.c[j] = j < m ? coef[j] : 0.0;
  ritz_kernel<<<red_grid(n, RED_BLOCKS), RED_T, 0, s>>>(n, m, V, AV, ld, a, theta, xs, r, R.part, R.ticket, R.out);
}

void launch_gs(long n, int m, const double* V, long ld, const double* d_coef, double* t, cudaStream_t s) {
  gs_kernel<<<elem_grid(n), 256, 0, s>>>(n, m, V, ld, d_coef, t);
}

void launch_axpy_dev(long n, const double* d_a, double sgn, const double* x, double* y, cudaStream_t s) {
  axpy_dev_kernel<<<elem_grid(n), 256, 0, s>>>(n, d_a, sgn, x, y);
}

void launch_multidot(long n, int m, const double* V, long ld, const double* x, double* d_out, double* d_part,
                     unsigned int* d_tickets, cudaStream_t s) {
  for (int j = 0; j < m; j += MD_TICKETS)
    multidot_kernel<<<dim3(red_grid(n, MD_BLOCKS), std::min(m - j, MD_TICKETS)), RED_T, 0, s>>>(
        V + j * ld, ld, x, n, d_part + (long)j * MD_BLOCKS, d_tickets, d_out + j);
}

void launch_axpy(long n, double a, const double* x, double* y, cudaStream_t s) {
  axpby_kernel<<<elem_grid(n), 256, 0, s>>>(n, a, x, 0.0, y, 0);
}
void launch_axpby(long n, double a, const double* x, double b, double* y, cudaStream_t s) {
  axpby_kernel<<<elem_grid(n), 256, 0, s>>>(n, a, x, b, y, 1);
}
void launch_scale(long n, double a, const double* x, double* y, cudaStream_t s) {
  axpby_kernel<<<elem_grid(n), 256, 0, s>>>(n, a, x, 0.0, y, 2);
}
void launch_fill(long n, double v, double* x, cudaStream_t s) {
  axpby_kernel<<<elem_grid(n), 256, 0, s>>>(n, v, nullptr, 0.0, x, 3);
}
void launch_precond(long n, const double* x, const double* d, double shift, double fl, double* y, int absval,
                    cudaStream_t s) {
  precond_kernel<<<elem_grid(n), 256, 0, s>>>(n, x, d, shift, fl, y, absval);
}
void launch_lincomb(long n, int m, const double* V, long ld, const double* coef, double* out, cudaStream_t s) {
  lincomb_kernel<<<elem_grid(n), 256, 0, s>>>(n, m, V, ld, coef, out);
}
void launch_lincomb_args(long n, int m, const double* V, long ld, const double* coef, double* out, cudaStream_t s) {
  LincombArgs a;
  for (int j = 0; j < LINCOMB_ARGS; ++j) a.c[j] = j < m ? coef[j] : 0.0;
  lincomb_args_kernel<<<elem_grid(n), 256, 0, s>>>(n, m, V, ld, a, out);
}
void launch_gather(const GatherTask* d_tasks, int ntasks, int max_elems, cudaStream_t s) {
  if (ntasks <= 0) return;
  int gx = std::max(1, std::min((max_elems + 255) / 256, 64));
  gather_kernel<<<dim3(gx, ntasks), 256, 0, s>>>(d_tasks, max_elems);
}
void launch_take_eigvecs(const double* V, int n, int m, int right, double* out, cudaStream_t s) {
  take_eigvecs_kernel<<<elem_grid((long)n * m), 256, 0, s>>>(V, n, m, right, out);
}
void launch_noise(long n, double amp, unsigned long long seed, double* x, cudaStream_t s) {
  noise_kernel<<<elem_grid(n), 256, 0, s>>>(n, amp, seed, x);
}
void launch_f64_to_bf16(long n, const double* x, uint16_t* y, cudaStream_t s) {
  f64_to_bf16_kernel<<<elem_grid(n), 256, 0, s>>>(n, x, reinterpret_cast<__nv_bfloat16*>(y));
}
void launch_f64_to_f32(long n, const double* x, float* y, cudaStream_t s) {
  f64_to_f32_kernel<<<elem_grid(n), 256, 0, s>>>(n, x, y);
}

}  // namespace mpslcc
