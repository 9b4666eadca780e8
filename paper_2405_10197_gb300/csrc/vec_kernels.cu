// Davidson-Liu building blocks on long vectors (step a7), for FP64 vectors and
// for the FP32 vectors of the reduced-precision phase.  Each kernel streams its
// operands once; reductions go through per-block partial sums (FP64) and a second
// pass, so results do not depend on atomic ordering.  FP32 kernels accumulate in
// FP32 within a warp and in FP64 across warps and blocks.
#include <type_traits>

#include "forte_internal.h"

namespace forte {

constexpr int VK_THREADS = 256;
constexpr int VK_EPT = 16;  // elements per thread per block
constexpr long long VK_CHUNK = (long long)VK_THREADS * VK_EPT;
constexpr int VK_MAXV = 64;  // vectors handled by one multidot / update launch

static inline unsigned vk_blocks(long long n) { return (unsigned)((n + VK_CHUNK - 1) / VK_CHUNK); }

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block-wide sum; every thread returns the total.  red must hold 32 doubles.
__device__ __forceinline__ double block_sum(double v, double *red) {
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  double t = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : 0.0;
  if (w == 0) t = warp_sum(t);
  if (threadIdx.x == 0) red[0] = t;
  __syncthreads();
  return red[0];
}

// Block-wide sum of per-thread values of type T: warp sums in T, the sum over
// warps in FP64 (one warp); every thread returns the total.  red holds 32 doubles.
template <typename T>
__device__ __forceinline__ double block_sum_t(T v, double *red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = (double)v;
  __syncthreads();
  double t = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : 0.0;
  if (w == 0) t = warp_sum(t);
  if (threadIdx.x == 0) red[0] = t;
  __syncthreads();
  return red[0];
}

// Second pass of a reduction, fused into the kernel that writes the partials: every
// block publishes its partials part[block][0..m) and counts itself in; the last block
// to arrive sums part[b][c] over b (strided by thread, then block_sum: the order of
// a separate 256-thread pass) into out[c] and resets the counter for the next
// launch on the stream.  No block waits for another.
__device__ __forceinline__ bool last_block(unsigned *counter) {
  __shared__ bool s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(counter, 1u) == gridDim.x - 1;
  __syncthreads();
  if (s_last) __threadfence();
  return s_last;
}
__device__ __forceinline__ void last_block_sums(const double *part, int m, double *__restrict__ out,
                                                unsigned *counter, double *red) {
  if (!last_block(counter)) return;
  const int nblk = (int)gridDim.x;
  for (int c = 0; c < m; ++c) {
    double s = 0.0;
    for (int b = threadIdx.x; b < nblk; b += blockDim.x) s += __ldcg(part + (long long)b * m + c);
    s = block_sum(s, red);
    if (threadIdx.x == 0) out[c] = s;
  }
  if (threadIdx.x == 0) *counter = 0u;
}
// The same with a group of g lanes (a power of two, m groups if they fit) per column: the
// FP64 pipe issues a warp's addition in 16 clocks, so a block-wide sum per column, most of
// whose lanes add zeros, takes longer than the rest of a short kernel.
__device__ __forceinline__ void last_block_lanes(const double *part, int m, double *__restrict__ out,
                                                 unsigned *counter) {
  if (!last_block(counter)) return;
  const int nblk = (int)gridDim.x;
  int g = 32;
  while (g > 4 && m * g > (int)blockDim.x) g >>= 1;
  const int groups = blockDim.x / g, lane = threadIdx.x % g;
  for (int c0 = 0; c0 < m; c0 += groups) {
    const int c = c0 + threadIdx.x / g;
    double s = 0.0;
    if (c < m) {
#pragma unroll 4
      for (int b = lane; b < nblk; b += g) s += __ldcg(part + (long long)b * m + c);
    }
    for (int o = g >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (c < m && lane == 0) out[c] = s;
  }
  if (threadIdx.x == 0) *counter = 0u;
}

// part[block][i] = sum over the block's chunk of V_i . x   (i < nv)
template <typename T>
__global__ void __launch_bounds__(VK_THREADS) k_multidot(const T *__restrict__ V, int nv, long long ld,
                                                         const T *__restrict__ x, long long n,
                                                         double *__restrict__ part, double *__restrict__ out,
                                                         unsigned *counter) {
  __shared__ double red[32];
  const long long base = (long long)blockIdx.x * VK_CHUNK + threadIdx.x;
  T xr[VK_EPT];
#pragma unroll
  for (int k = 0; k < VK_EPT; ++k) {
    long long j = base + (long long)k * VK_THREADS;
    xr[k] = (j < n) ? x[j] : T(0);
  }
  for (int i = 0; i < nv; ++i) {
    const T *v = V + (long long)i * ld;
    T a = 0;
#pragma unroll
    for (int k = 0; k < VK_EPT; ++k) {
      long long j = base + (long long)k * VK_THREADS;
      if (j < n) a += v[j] * xr[k];
    }
    const double at = block_sum_t<T>(a, red);
    if (threadIdx.x == 0) part[(long long)blockIdx.x * nv + i] = at;
  }
  last_block_sums(part, nv, out, counter, red);
}

// out_{c0+c} = sum_i coef[i*ncomb + c0 + c] V_i  for c < NC.  NC is a template
// parameter: the FP64 pipe of this GPU is narrow enough that issuing
// predicated-off multiply-adds for unused outputs would dominate the kernel.
template <int NC, typename T>
__global__ void __launch_bounds__(VK_THREADS) k_combine(const T *__restrict__ V, int nv, long long ld,
                                                        const double *__restrict__ coef, int ncomb, int c0,
                                                        T *__restrict__ out, long long ldo, long long n) {
  __shared__ T sc[VK_MAXV * NC];
  for (int i = threadIdx.x; i < nv * NC; i += blockDim.x) sc[i] = (T)coef[(i / NC) * ncomb + c0 + i % NC];
  __syncthreads();
  for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n;
       j += (long long)gridDim.x * blockDim.x) {
    T acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] = 0;
#pragma unroll 4
    for (int i = 0; i < nv; ++i) {
      const T v = V[(long long)i * ld + j];
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[c] += sc[i * NC + c] * v;
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) out[(long long)(c0 + c) * ldo + j] = acc[c];
  }
}

// r = sum_i u_i S_i - theta sum_i u_i B_i ;  t = r / (theta - hdiag) (guarded);
// part[block] = sum r^2 over the block's chunk.
template <typename T>
__global__ void __launch_bounds__(VK_THREADS) k_residual_precond(
    const T *__restrict__ B, const T *__restrict__ S, int k, long long ld,
    const double *__restrict__ u, double theta, const double *__restrict__ hd, double guard,
    T *__restrict__ t, long long n, double *__restrict__ part, double *__restrict__ out, unsigned *counter) {
  __shared__ double red[32];
  __shared__ T su[VK_MAXV];
  for (int i = threadIdx.x; i < k; i += blockDim.x) su[i] = (T)u[i];
  __syncthreads();
  const long long base = (long long)blockIdx.x * VK_CHUNK + threadIdx.x;
  const T th = (T)theta;
  T rr = 0;
#pragma unroll 4
  for (int e = 0; e < VK_EPT; ++e) {
    long long j = base + (long long)e * VK_THREADS;
    if (j >= n) break;
    T hx = 0, x = 0;
    for (int i = 0; i < k; ++i) {
      hx += su[i] * S[(long long)i * ld + j];
      x += su[i] * B[(long long)i * ld + j];
    }
    const T r = hx - th * x;
    rr += r * r;
    double den = theta - hd[j];
    if (fabs(den) < guard) den = (den >= 0.0) ? guard : -guard;
    t[j] = r / (T)den;
  }
  const double rt = block_sum_t<T>(rr, red);
  if (threadIdx.x == 0) part[blockIdx.x] = rt;
  last_block_sums(part, 1, out, counter, red);
}

// t_out = t_in - sum_i c_i B_i ; part[block][i] = B_i . t_out (i < k), part[block][k] = |t_out|^2.
// Without DOTS the B_i . t_out are not formed (a second read of every B_i) and part
// holds zeros there.  c == nullptr: no update (t_out = t_in; the B_i are read once,
// for the dots).
template <typename T, bool DOTS>
__global__ void __launch_bounds__(VK_THREADS) k_orth_update(const T *__restrict__ Bm, int k,
                                                            long long ld, const double *__restrict__ c,
                                                            const T *t_in, T *t_out, long long n,
                                                            double *__restrict__ part, double *__restrict__ out,
                                                            unsigned *counter) {
  __shared__ double red[32];
  __shared__ T sc[VK_MAXV];
  const int ku = c ? k : 0;  // vectors to subtract
  for (int i = threadIdx.x; i < ku; i += blockDim.x) sc[i] = (T)c[i];
  __syncthreads();
  const long long base = (long long)blockIdx.x * VK_CHUNK + threadIdx.x;
  T tr[VK_EPT];
#pragma unroll
  for (int e = 0; e < VK_EPT; ++e) {
    long long j = base + (long long)e * VK_THREADS;
    tr[e] = (j < n) ? t_in[j] : T(0);
  }
  for (int i = 0; i < ku; ++i) {
    const T *b = Bm + (long long)i * ld;
#pragma unroll
    for (int e = 0; e < VK_EPT; ++e) {
      long long j = base + (long long)e * VK_THREADS;
      if (j < n) tr[e] -= sc[i] * b[j];
    }
  }
  T nn = 0;
#pragma unroll
  for (int e = 0; e < VK_EPT; ++e) {
    long long j = base + (long long)e * VK_THREADS;
    if (j < n) {
      t_out[j] = tr[e];
      nn += tr[e] * tr[e];
    }
  }
  if (DOTS) {
    for (int i = 0; i < k; ++i) {
      const T *b = Bm + (long long)i * ld;
      T a = 0;
#pragma unroll
      for (int e = 0; e < VK_EPT; ++e) {
        long long j = base + (long long)e * VK_THREADS;
        if (j < n) a += b[j] * tr[e];
      }
      const double at = block_sum_t<T>(a, red);
      if (threadIdx.x == 0) part[(long long)blockIdx.x * (k + 1) + i] = at;
    }
  } else {
    for (int i = threadIdx.x; i < k; i += blockDim.x) part[(long long)blockIdx.x * (k + 1) + i] = 0.0;
  }
  const double nt = block_sum_t<T>(nn, red);
  if (threadIdx.x == 0) part[(long long)blockIdx.x * (k + 1) + k] = nt;
  last_block_sums(part, k + 1, out, counter, red);
}

// y = a x + b y
__global__ void k_axpby(double a, const double *__restrict__ x, double b, double *__restrict__ y, long long n) {
  for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n;
       j += (long long)gridDim.x * blockDim.x)
    y[j] = a * x[j] + b * y[j];
}

// rinv = 1 / |theta - hdiag| with the magnitude clamped below at guard: the FP64
// divisions of the diagonal preconditioner, done once per correction solve (the FP64
// pipe of this GPU makes a division per element and application the bound otherwise)
__global__ void k_precond_inv(const double *__restrict__ hd, double theta, double guard, double *__restrict__ rinv,
                              long long n) {
  for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (long long)gridDim.x * blockDim.x) {
    double den = fabs(theta - hd[j]);
    if (den < guard) den = guard;
    rinv[j] = 1.0 / den;
  }
}

template <typename T>
__global__ void k_scale(T *__restrict__ x, const T *__restrict__ src, double alpha, long long n) {
  const T al = (T)alpha;
  for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n;
       j += (long long)gridDim.x * blockDim.x)
    x[j] = al * src[j];
}

template <typename TI, typename TO>
__global__ void k_convert(const TI *__restrict__ x, TO *__restrict__ y, long long n) {
  for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n;
       j += (long long)gridDim.x * blockDim.x)
    y[j] = (TO)x[j];
}

// Block minimum of (value, index) over entries not in excl[0..nex); lexicographic.
__global__ void k_argmin(const double *__restrict__ x, long long n, const long long *__restrict__ excl,
                         int nex, double *__restrict__ bval, long long *__restrict__ bidx) {
  __shared__ double sv[VK_THREADS];
  __shared__ long long si[VK_THREADS];
  double best = INFINITY;
  long long bi = -1;
  for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n;
       j += (long long)gridDim.x * blockDim.x) {
    double v = x[j];
    bool skip = false;
    for (int e = 0; e < nex; ++e) skip |= (excl[e] == j);
    if (skip) continue;
    if (bi < 0 || v < best || (v == best && j < bi)) { best = v; bi = j; }
  }
  sv[threadIdx.x] = best;
  si[threadIdx.x] = bi;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      double v2 = sv[threadIdx.x + s];
      long long i2 = si[threadIdx.x + s];
      double v1 = sv[threadIdx.x];
      long long i1 = si[threadIdx.x];
      bool take = (i2 >= 0) && (i1 < 0 || v2 < v1 || (v2 == v1 && i2 < i1));
      if (take) { sv[threadIdx.x] = v2; si[threadIdx.x] = i2; }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) { bval[blockIdx.x] = sv[0]; bidx[blockIdx.x] = si[0]; }
}

__global__ void k_nonfinite(const double *__restrict__ x, long long n, int *flag) {
  for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n;
       j += (long long)gridDim.x * blockDim.x)
    if (!isfinite(x[j])) *flag = 1;
}

// ------------------------------------------------------------------ short vectors
// Up to VS_MAX_N elements the kernels above and below leave most SMs idle (a block takes
// 4096 or 2048 elements), and the FP64 work of a block is then the time: 5 blocks of a
// 4900-element residual pass took 31 us.  Here a block of 64 threads takes 128 elements,
// one chunk, so that the vectors spread over the SMs; the per-thread sums of a column
// meet in shared memory, where 4 threads add one column (64 values), instead of a
// five-step warp reduction per column.  Elements are loaded singly, so any count and
// alignment will do.  FP64 vectors only: the FP32 ones of the reduced-precision phase keep
// the kernels above and below, whose order of sums its rounding follows.  One GB300,
// CAS(8,8) FP64 solve (133 iterations): residual pass 31 -> 14 us, 11-vector dots 22 ->
// 9 us, whole solve 18.9 -> 14.0 ms.
constexpr int VS_T = 64;
constexpr int VS_E = 2;
constexpr long long VS_CHUNK = VS_T * VS_E;
constexpr int VS_COLS = 16;  // columns reduced at a time
constexpr long long VS_MAX_N = VS_CHUNK * 608;

struct VsRed {
  double v[VS_COLS][VS_T + 1];
};
// Publish the block's sums of columns c0 .. c0 + nc (r.v filled by every thread).
__device__ __forceinline__ void vs_columns(VsRed &r, int c0, int nc, int m, double *part) {
  __syncthreads();
  const int c = threadIdx.x >> 2, q = threadIdx.x & 3;
  double a = 0.0, b = 0.0;
  if (c < nc) {
#pragma unroll
    for (int k = 0; k < VS_T / 4; k += 2) {
      a += r.v[c][q + 4 * k];
      b += r.v[c][q + 4 * k + 4];
    }
  }
  a += b;
  a += __shfl_xor_sync(0xffffffffu, a, 1);
  a += __shfl_xor_sync(0xffffffffu, a, 2);
  if (c < nc && q == 0) part[(long long)blockIdx.x * m + c0 + c] = a;
  __syncthreads();
}

// part[block][col0 + i] = sum over the chunk of V_i . x, i < nv (m columns in all).
__device__ __forceinline__ void vs_dots(VsRed &r, const double *__restrict__ V, int nv, long long ld, const double (&x)[VS_E],
                                        long long j0, long long n, int col0, int m, double *part) {
  for (int i0 = 0; i0 < nv; i0 += VS_COLS) {
    const int nc = min(VS_COLS, nv - i0);
#pragma unroll 4
    for (int i = 0; i < nc; ++i) {
      const double *v = V + (long long)(i0 + i) * ld;
      double a = 0;
#pragma unroll
      for (int e = 0; e < VS_E; ++e)
        if (j0 + e * VS_T < n) a += v[j0 + e * VS_T] * x[e];
      r.v[i][threadIdx.x] = a;
    }
    vs_columns(r, col0 + i0, nc, m, part);
  }
}

__global__ void __launch_bounds__(VS_T) k_multidot_s(const double *__restrict__ V, int nv, long long ld,
                                                     const double *__restrict__ x, long long n, double *__restrict__ part,
                                                     double *__restrict__ out, unsigned *counter) {
  __shared__ VsRed r;
  const long long j0 = (long long)blockIdx.x * VS_CHUNK + threadIdx.x;
  double xr[VS_E];
#pragma unroll
  for (int e = 0; e < VS_E; ++e) xr[e] = j0 + e * VS_T < n ? x[j0 + e * VS_T] : 0.0;
  vs_dots(r, V, nv, ld, xr, j0, n, 0, nv, part);
  last_block_lanes(part, nv, out, counter);
}

// As k_orth_update_p: t_out = scale (t_in - B c), out = [B^T t_out (zeros unless DOTS), |t_out|^2].
template <bool DOTS>
__global__ void __launch_bounds__(VS_T) k_orth_update_s(const double *__restrict__ B, int k, long long ld,
                                                        const double *__restrict__ c, const double *t_in, double *t_out,
                                                        long long n, double scale, double *__restrict__ part,
                                                        double *__restrict__ out, unsigned *counter) {
  __shared__ VsRed r;
  __shared__ double sc[VK_MAXV];
  const int ku = c ? k : 0;
  for (int i = threadIdx.x; i < ku; i += VS_T) sc[i] = c[i];
  __syncthreads();
  const long long j0 = (long long)blockIdx.x * VS_CHUNK + threadIdx.x;
  double t[VS_E], nn = 0;
#pragma unroll
  for (int e = 0; e < VS_E; ++e) t[e] = j0 + e * VS_T < n ? t_in[j0 + e * VS_T] : 0.0;
#pragma unroll 4
  for (int i = 0; i < ku; ++i)
#pragma unroll
    for (int e = 0; e < VS_E; ++e)
      if (j0 + e * VS_T < n) t[e] -= sc[i] * B[(long long)i * ld + j0 + e * VS_T];
#pragma unroll
  for (int e = 0; e < VS_E; ++e)
    if (j0 + e * VS_T < n) {
      if (scale != 1.0) t[e] *= scale;
      t_out[j0 + e * VS_T] = t[e];
      nn += t[e] * t[e];
    }
  r.v[0][threadIdx.x] = nn;
  vs_columns(r, k, 1, k + 1, part);
  if (DOTS) {
    vs_dots(r, B, k, ld, t, j0, n, 0, k + 1, part);
  } else {
    for (int i = threadIdx.x; i < k; i += VS_T) part[(long long)blockIdx.x * (k + 1) + i] = 0.0;
  }
  last_block_lanes(part, k + 1, out, counter);
}

// As k_residual_precond_p: t = r / (theta - H_II), out = [|r|^2 (, B^T t, |t|^2)].
template <bool DOTS>
__global__ void __launch_bounds__(VS_T) k_residual_precond_s(const double *__restrict__ B, const double *__restrict__ S, int k,
                                                             long long ld, const double *__restrict__ u, double theta,
                                                             const double *__restrict__ hd, double guard,
                                                             double *__restrict__ t, long long n, double *__restrict__ part,
                                                             double *__restrict__ out, unsigned *counter) {
  __shared__ VsRed r;
  __shared__ double su[VK_MAXV];
  const int m = DOTS ? k + 2 : 1;
  for (int i = threadIdx.x; i < k; i += VS_T) su[i] = u[i];
  __syncthreads();
  const long long j0 = (long long)blockIdx.x * VS_CHUNK + threadIdx.x;
  double hx[VS_E], xv[VS_E], rr = 0, tt = 0;
#pragma unroll
  for (int e = 0; e < VS_E; ++e) hx[e] = xv[e] = 0;
#pragma unroll 4
  for (int i = 0; i < k; ++i)
#pragma unroll
    for (int e = 0; e < VS_E; ++e)
      if (j0 + e * VS_T < n) {
        hx[e] += su[i] * S[(long long)i * ld + j0 + e * VS_T];
        xv[e] += su[i] * B[(long long)i * ld + j0 + e * VS_T];
      }
#pragma unroll
  for (int e = 0; e < VS_E; ++e)
    if (j0 + e * VS_T < n) {
      const double res = hx[e] - theta * xv[e];
      rr += res * res;
      double den = theta - hd[j0 + e * VS_T];
      if (fabs(den) < guard) den = (den >= 0.0) ? guard : -guard;
      hx[e] = res / den;  // hx now holds t
      tt += hx[e] * hx[e];
      t[j0 + e * VS_T] = hx[e];
    }
  r.v[0][threadIdx.x] = rr;
  vs_columns(r, 0, 1, m, part);
  if (DOTS) {
    r.v[0][threadIdx.x] = tt;
    vs_columns(r, k + 1, 1, m, part);
    vs_dots(r, B, k, ld, hx, j0, n, 1, m, part);
  }
  last_block_lanes(part, m, out, counter);
}

// ------------------------------------------------------------------ packet kernels
// The kernels below move every operand in 16-byte packets (float4 / double2), run a
// persistent grid (4 resident blocks of 256 threads per SM) over chunks of
// VK_THREADS x VP_PER packets, keep per-warp partial sums in shared memory across the
// chunks of a block (no block barrier per chunk, one reduction per block instead of
// one per 4096 elements), and finish with the fused last-block pass.  They need the
// element count and the leading dimension to be multiples of the packet and 16-byte
// aligned bases; the element kernels above serve every other case.  Per element they
// do the arithmetic of the element kernels in the same order; only the order of the
// partial sums differs (fixed for a given grid, so results are reproducible).
template <typename T>
struct Pk;
template <>
struct Pk<float> {
  using V = float4;
  static constexpr int P = 4;
};
template <>
struct Pk<double> {
  using V = double2;
  static constexpr int P = 2;
};

constexpr int VP_PER = 4;                   // packets per thread per chunk
constexpr int VP_CH = VK_THREADS * VP_PER;  // packets per chunk
constexpr int VP_WARPS = VK_THREADS / 32;
constexpr int VP_BPS = 4;                   // resident blocks per SM (64 registers a thread)

template <typename T>
__device__ __forceinline__ void pk_ld(const T *p, long long q, T (&x)[Pk<T>::P]) {
  const typename Pk<T>::V v = reinterpret_cast<const typename Pk<T>::V *>(p)[q];
  if constexpr (Pk<T>::P == 4) {
    x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
  } else {
    x[0] = v.x; x[1] = v.y;
  }
}
template <typename T>
__device__ __forceinline__ void pk_st(T *p, long long q, const T (&x)[Pk<T>::P]) {
  typename Pk<T>::V v;
  if constexpr (Pk<T>::P == 4) {
    v.x = x[0]; v.y = x[1]; v.z = x[2]; v.w = x[3];
  } else {
    v.x = x[0]; v.y = x[1];
  }
  reinterpret_cast<typename Pk<T>::V *>(p)[q] = v;
}
// the P FP64 diagonal entries of packet q (hd is FP64 for either vector type)
template <int P>
__device__ __forceinline__ void hd_ld(const double *hd, long long q, double (&h)[P]) {
  const double2 a = reinterpret_cast<const double2 *>(hd)[q * (P / 2)];
  h[0] = a.x;
  h[1] = a.y;
  if constexpr (P == 4) {
    const double2 b = reinterpret_cast<const double2 *>(hd)[q * 2 + 1];
    h[2] = b.x;
    h[3] = b.y;
  }
}

// Lane 0 adds the warp's sum of v (summed in T across the warp) to acc[warp].
template <typename T>
__device__ __forceinline__ void warp_add(T v, double *acc) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) acc[threadIdx.x >> 5] += (double)v;
}

// part[block][i] = sum over warps of sw[i][warp], i < m (warps in a fixed order).
__device__ __forceinline__ void block_partials(const double *sw, int m, double *part) {
  __syncthreads();
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < VP_WARPS; ++w) s += sw[i * VP_WARPS + w];
    part[(long long)blockIdx.x * m + i] = s;
  }
}

// out[i] = V_i . x (i < nv); np = packets per vector.
template <typename T>
__global__ void __launch_bounds__(VK_THREADS, VP_BPS) k_multidot_p(const T *__restrict__ V, int nv, long long ld,
                                                           const T *__restrict__ x, long long np,
                                                           double *__restrict__ part, double *__restrict__ out,
                                                           unsigned *counter) {
  constexpr int P = Pk<T>::P;
  __shared__ double red[32];
  __shared__ double sw[VK_MAXV * VP_WARPS];
  for (int i = threadIdx.x; i < nv * VP_WARPS; i += blockDim.x) sw[i] = 0.0;
  __syncthreads();
  const long long nch = (np + VP_CH - 1) / VP_CH;
  for (long long ch = blockIdx.x; ch < nch; ch += gridDim.x) {
    const long long q0 = ch * VP_CH + threadIdx.x;
    T xr[VP_PER][P];
#pragma unroll
    for (int e = 0; e < VP_PER; ++e) {
      const long long q = q0 + (long long)e * VK_THREADS;
      if (q < np) {
        pk_ld(x, q, xr[e]);
      } else {
#pragma unroll
        for (int p = 0; p < P; ++p) xr[e][p] = T(0);
      }
    }
    for (int i = 0; i < nv; ++i) {
      const T *v = V + (long long)i * ld;
      T a = 0;
#pragma unroll
      for (int e = 0; e < VP_PER; ++e) {
        const long long q = q0 + (long long)e * VK_THREADS;
        if (q < np) {
          T vv[P];
          pk_ld(v, q, vv);
#pragma unroll
          for (int p = 0; p < P; ++p) a += vv[p] * xr[e][p];
        }
      }
      warp_add(a, sw + i * VP_WARPS);
    }
  }
  block_partials(sw, nv, part);
  last_block_sums(part, nv, out, counter, red);
}

// The same for nv <= KMAX: loop over the vectors unrolled, partial sums of the
// block's chunks in registers, one warp reduction per vector and block.
template <typename T, int KMAX>
__global__ void __launch_bounds__(VK_THREADS, VP_BPS) k_multidot_u(const T *__restrict__ V, int nv, long long ld,
                                                                   const T *__restrict__ x, long long np,
                                                                   double *__restrict__ part,
                                                                   double *__restrict__ out, unsigned *counter) {
  constexpr int P = Pk<T>::P;
  __shared__ double red[32];
  __shared__ double sw[KMAX * VP_WARPS];
  for (int i = threadIdx.x; i < nv * VP_WARPS; i += blockDim.x) sw[i] = 0.0;
  __syncthreads();
  T acc[KMAX];
#pragma unroll
  for (int i = 0; i < KMAX; ++i) acc[i] = T(0);
  const long long nch = (np + VP_CH - 1) / VP_CH;
  for (long long ch = blockIdx.x; ch < nch; ch += gridDim.x) {
    const long long q0 = ch * VP_CH + threadIdx.x;
    T xr[VP_PER][P];
#pragma unroll
    for (int e = 0; e < VP_PER; ++e) {
      const long long q = q0 + (long long)e * VK_THREADS;
      if (q < np) {
        pk_ld(x, q, xr[e]);
      } else {
#pragma unroll
        for (int p = 0; p < P; ++p) xr[e][p] = T(0);
      }
    }
#pragma unroll
    for (int i = 0; i < KMAX; ++i) {
      if (i < nv) {
        const T *v = V + (long long)i * ld;
#pragma unroll
        for (int e = 0; e < VP_PER; ++e) {
          const long long q = q0 + (long long)e * VK_THREADS;
          if (q < np) {
            T vv[P];
            pk_ld(v, q, vv);
#pragma unroll
            for (int p = 0; p < P; ++p) acc[i] += vv[p] * xr[e][p];
          }
        }
      }
    }
  }
#pragma unroll
  for (int i = 0; i < KMAX; ++i)
    if (i < nv) warp_add(acc[i], sw + i * VP_WARPS);
  block_partials(sw, nv, part);
  last_block_sums(part, nv, out, counter, red);
}

// t_out = scale (t_in - sum_i c_i B_i); out = [B_i . t_out (i < k, zeros unless DOTS),
// |t_out|^2].  c == nullptr: no update.  t_in may alias t_out.
template <typename T, bool DOTS>
__global__ void __launch_bounds__(VK_THREADS, VP_BPS) k_orth_update_p(const T *__restrict__ Bm, int k, long long ld,
                                                              const double *__restrict__ c, const T *t_in,
                                                              T *t_out, long long np, double scale,
                                                              double *__restrict__ part, double *__restrict__ out,
                                                              unsigned *counter) {
  constexpr int P = Pk<T>::P;
  __shared__ double red[32];
  __shared__ double sw[(VK_MAXV + 1) * VP_WARPS];
  __shared__ T sc[VK_MAXV];
  const int ku = c ? k : 0;
  for (int i = threadIdx.x; i < ku; i += blockDim.x) sc[i] = (T)c[i];
  for (int i = threadIdx.x; i < (k + 1) * VP_WARPS; i += blockDim.x) sw[i] = 0.0;
  __syncthreads();
  const T s = (T)scale;
  const bool scaled = scale != 1.0;  // FP64 multiplies cost FP64-pipe slots: skip the identity
  const long long nch = (np + VP_CH - 1) / VP_CH;
  for (long long ch = blockIdx.x; ch < nch; ch += gridDim.x) {
    const long long q0 = ch * VP_CH + threadIdx.x;
    T tr[VP_PER][P];
#pragma unroll
    for (int e = 0; e < VP_PER; ++e) {
      const long long q = q0 + (long long)e * VK_THREADS;
      if (q < np) {
        pk_ld(t_in, q, tr[e]);
      } else {
#pragma unroll
        for (int p = 0; p < P; ++p) tr[e][p] = T(0);
      }
    }
    for (int i = 0; i < ku; ++i) {
      const T *b = Bm + (long long)i * ld;
      const T ci = sc[i];
#pragma unroll
      for (int e = 0; e < VP_PER; ++e) {
        const long long q = q0 + (long long)e * VK_THREADS;
        if (q < np) {
          T bv[P];
          pk_ld(b, q, bv);
#pragma unroll
          for (int p = 0; p < P; ++p) tr[e][p] -= ci * bv[p];
        }
      }
    }
    T nn = 0;
#pragma unroll
    for (int e = 0; e < VP_PER; ++e) {
      const long long q = q0 + (long long)e * VK_THREADS;
      if (q < np) {
#pragma unroll
        for (int p = 0; p < P; ++p) {
          if (scaled) tr[e][p] *= s;
          nn += tr[e][p] * tr[e][p];
        }
        pk_st(t_out, q, tr[e]);
      }
    }
    warp_add(nn, sw + k * VP_WARPS);
    if (DOTS) {
      for (int i = 0; i < k; ++i) {
        const T *b = Bm + (long long)i * ld;
        T a = 0;
#pragma unroll
        for (int e = 0; e < VP_PER; ++e) {
          const long long q = q0 + (long long)e * VK_THREADS;
          if (q < np) {
            T bv[P];
            pk_ld(b, q, bv);
#pragma unroll
            for (int p = 0; p < P; ++p) a += bv[p] * tr[e][p];
          }
        }
        warp_add(a, sw + i * VP_WARPS);
      }
    }
  }
  block_partials(sw, k + 1, part);
  last_block_sums(part, k + 1, out, counter, red);
}

// The same for k <= KMAX: loops over the basis unrolled, partial sums in registers.
template <typename T, bool DOTS, int KMAX>
__global__ void __launch_bounds__(VK_THREADS, VP_BPS) k_orth_update_u(const T *__restrict__ Bm, int k, long long ld,
                                                                      const double *__restrict__ c, const T *t_in,
                                                                      T *t_out, long long np, double scale,
                                                                      double *__restrict__ part,
                                                                      double *__restrict__ out, unsigned *counter) {
  constexpr int P = Pk<T>::P;
  __shared__ double red[32];
  __shared__ double sw[(KMAX + 1) * VP_WARPS];
  __shared__ T sc[KMAX];
  const int ku = c ? k : 0;
  for (int i = threadIdx.x; i < ku; i += blockDim.x) sc[i] = (T)c[i];
  for (int i = threadIdx.x; i < (k + 1) * VP_WARPS; i += blockDim.x) sw[i] = 0.0;
  __syncthreads();
  const T s = (T)scale;
  const bool scaled = scale != 1.0;
  T nn = 0, acc[KMAX];
#pragma unroll
  for (int i = 0; i < KMAX; ++i) acc[i] = T(0);
  const long long nch = (np + VP_CH - 1) / VP_CH;
  for (long long ch = blockIdx.x; ch < nch; ch += gridDim.x) {
    const long long q0 = ch * VP_CH + threadIdx.x;
    T tr[VP_PER][P];
#pragma unroll
    for (int e = 0; e < VP_PER; ++e) {
      const long long q = q0 + (long long)e * VK_THREADS;
      if (q < np) {
        pk_ld(t_in, q, tr[e]);
      } else {
#pragma unroll
        for (int p = 0; p < P; ++p) tr[e][p] = T(0);
      }
    }
#pragma unroll
    for (int i = 0; i < KMAX; ++i) {
      if (i < ku) {
        const T *b = Bm + (long long)i * ld;
        const T ci = sc[i];
#pragma unroll
        for (int e = 0; e < VP_PER; ++e) {
          const long long q = q0 + (long long)e * VK_THREADS;
          if (q < np) {
            T bv[P];
            pk_ld(b, q, bv);
#pragma unroll
            for (int p = 0; p < P; ++p) tr[e][p] -= ci * bv[p];
          }
        }
      }
    }
#pragma unroll
    for (int e = 0; e < VP_PER; ++e) {
      const long long q = q0 + (long long)e * VK_THREADS;
      if (q < np) {
#pragma unroll
        for (int p = 0; p < P; ++p) {
          if (scaled) tr[e][p] *= s;
          nn += tr[e][p] * tr[e][p];
        }
        pk_st(t_out, q, tr[e]);
      }
    }
    if (DOTS) {
#pragma unroll
      for (int i = 0; i < KMAX; ++i) {
        if (i < k) {
          const T *b = Bm + (long long)i * ld;
#pragma unroll
          for (int e = 0; e < VP_PER; ++e) {
            const long long q = q0 + (long long)e * VK_THREADS;
            if (q < np) {
              T bv[P];
              pk_ld(b, q, bv);
#pragma unroll
              for (int p = 0; p < P; ++p) acc[i] += bv[p] * tr[e][p];
            }
          }
        }
      }
    }
  }
  warp_add(nn, sw + k * VP_WARPS);
  if (DOTS) {
#pragma unroll
    for (int i = 0; i < KMAX; ++i)
      if (i < k) warp_add(acc[i], sw + i * VP_WARPS);
  }
  block_partials(sw, k + 1, part);
  last_block_sums(part, k + 1, out, counter, red);
}

// r = sum_i u_i S_i - theta sum_i u_i B_i ;  t = r / (theta - hdiag) (guarded).
// out[0] = |r|^2; with DOTS also out[1 + i] = B_i . t (i < k) and out[1 + k] = |t|^2,
// which the Gram-Schmidt step of the new direction needs (B is read here anyway).
// PER packets per thread per chunk: the dots re-read the chunk's B_i right after
// forming t, and a small chunk keeps the 2k vectors of all resident chunks (~70 MB
// at PER = 2) within L2, so the re-read does not reach DRAM.
template <typename T, bool DOTS, int PER>
__global__ void __launch_bounds__(VK_THREADS, VP_BPS) k_residual_precond_p(
    const T *__restrict__ B, const T *__restrict__ S, int k, long long ld, const double *__restrict__ u,
    double theta, const double *__restrict__ hd, double guard, T *__restrict__ t, long long np,
    double *__restrict__ part, double *__restrict__ out, unsigned *counter) {
  constexpr int P = Pk<T>::P;
  __shared__ double red[32];
  __shared__ double sw[(VK_MAXV + 2) * VP_WARPS];
  __shared__ T su[VK_MAXV];
  const int m = DOTS ? k + 2 : 1;
  for (int i = threadIdx.x; i < k; i += blockDim.x) su[i] = (T)u[i];
  for (int i = threadIdx.x; i < m * VP_WARPS; i += blockDim.x) sw[i] = 0.0;
  __syncthreads();
  const T th = (T)theta;
  const long long nch = (np + (VK_THREADS * PER) - 1) / (VK_THREADS * PER);
  for (long long ch = blockIdx.x; ch < nch; ch += gridDim.x) {
    const long long q0 = ch * (VK_THREADS * PER) + threadIdx.x;
    T hx[PER][P], xv[PER][P];
#pragma unroll
    for (int e = 0; e < PER; ++e)
#pragma unroll
      for (int p = 0; p < P; ++p) hx[e][p] = xv[e][p] = T(0);
    for (int i = 0; i < k; ++i) {
      const T ui = su[i];
      const T *sp = S + (long long)i * ld, *bp = B + (long long)i * ld;
#pragma unroll
      for (int e = 0; e < PER; ++e) {
        const long long q = q0 + (long long)e * VK_THREADS;
        if (q < np) {
          T sv[P], bv[P];
          pk_ld(sp, q, sv);
          pk_ld(bp, q, bv);
#pragma unroll
          for (int p = 0; p < P; ++p) {
            hx[e][p] += ui * sv[p];
            xv[e][p] += ui * bv[p];
          }
        }
      }
    }
    T rr = 0, tt = 0;
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      const long long q = q0 + (long long)e * VK_THREADS;
      if (q < np) {
        double h[P];
        hd_ld<P>(hd, q, h);
#pragma unroll
        for (int p = 0; p < P; ++p) {
          const T r = hx[e][p] - th * xv[e][p];
          rr += r * r;
          double den = theta - h[p];
          if (fabs(den) < guard) den = (den >= 0.0) ? guard : -guard;
          hx[e][p] = r / (T)den;  // hx now holds t
          tt += hx[e][p] * hx[e][p];
        }
        pk_st(t, q, hx[e]);
      }
    }
    warp_add(rr, sw);
    if (DOTS) {
      warp_add(tt, sw + (k + 1) * VP_WARPS);
      for (int i = 0; i < k; ++i) {
        const T *bp = B + (long long)i * ld;
        T a = 0;
#pragma unroll
        for (int e = 0; e < PER; ++e) {
          const long long q = q0 + (long long)e * VK_THREADS;
          if (q < np) {
            T bv[P];
            pk_ld(bp, q, bv);
#pragma unroll
            for (int p = 0; p < P; ++p) a += bv[p] * hx[e][p];
          }
        }
        warp_add(a, sw + (1 + i) * VP_WARPS);
      }
    }
  }
  block_partials(sw, m, part);
  last_block_sums(part, m, out, counter, red);
}

// The same for k <= KMAX with the loops over the basis unrolled (the loads of all k
// vectors of a chunk can be in flight together) and the partial sums of the block's
// chunks kept in registers, reduced over the warp once per block.
template <typename T, bool DOTS, int PER, int KMAX>
__global__ void __launch_bounds__(VK_THREADS, VP_BPS) k_residual_precond_u(
    const T *__restrict__ B, const T *__restrict__ S, int k, long long ld, const double *__restrict__ u,
    double theta, const double *__restrict__ hd, double guard, T *__restrict__ t, long long np,
    double *__restrict__ part, double *__restrict__ out, unsigned *counter) {
  constexpr int P = Pk<T>::P;
  __shared__ double red[32];
  __shared__ double sw[(KMAX + 2) * VP_WARPS];
  __shared__ T su[KMAX];
  const int m = DOTS ? k + 2 : 1;
  for (int i = threadIdx.x; i < k; i += blockDim.x) su[i] = (T)u[i];
  for (int i = threadIdx.x; i < m * VP_WARPS; i += blockDim.x) sw[i] = 0.0;
  __syncthreads();
  const T th = (T)theta;
  T rr = 0, tt = 0, acc[KMAX];
#pragma unroll
  for (int i = 0; i < KMAX; ++i) acc[i] = T(0);
  const long long nch = (np + (VK_THREADS * PER) - 1) / (VK_THREADS * PER);
  for (long long ch = blockIdx.x; ch < nch; ch += gridDim.x) {
    const long long q0 = ch * (VK_THREADS * PER) + threadIdx.x;
    T hx[PER][P], xv[PER][P];
#pragma unroll
    for (int e = 0; e < PER; ++e)
#pragma unroll
      for (int p = 0; p < P; ++p) hx[e][p] = xv[e][p] = T(0);
#pragma unroll
    for (int i = 0; i < KMAX; ++i) {
      if (i < k) {
        const T ui = su[i];
        const T *sp = S + (long long)i * ld, *bp = B + (long long)i * ld;
#pragma unroll
        for (int e = 0; e < PER; ++e) {
          const long long q = q0 + (long long)e * VK_THREADS;
          if (q < np) {
            T sv[P], bv[P];
            pk_ld(sp, q, sv);
            pk_ld(bp, q, bv);
#pragma unroll
            for (int p = 0; p < P; ++p) {
              hx[e][p] += ui * sv[p];
              xv[e][p] += ui * bv[p];
            }
          }
        }
      }
    }
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      const long long q = q0 + (long long)e * VK_THREADS;
      if (q < np) {
        double h[P];
        hd_ld<P>(hd, q, h);
#pragma unroll
        for (int p = 0; p < P; ++p) {
          const T r = hx[e][p] - th * xv[e][p];
          rr += r * r;
          double den = theta - h[p];
          if (fabs(den) < guard) den = (den >= 0.0) ? guard : -guard;
          hx[e][p] = r / (T)den;  // hx now holds t
          tt += hx[e][p] * hx[e][p];
        }
        pk_st(t, q, hx[e]);
      } else {
#pragma unroll
        for (int p = 0; p < P; ++p) hx[e][p] = T(0);
      }
    }
    if (DOTS) {
#pragma unroll
      for (int i = 0; i < KMAX; ++i) {
        if (i < k) {
          const T *bp = B + (long long)i * ld;
#pragma unroll
          for (int e = 0; e < PER; ++e) {
            const long long q = q0 + (long long)e * VK_THREADS;
            if (q < np) {
              T bv[P];
              pk_ld(bp, q, bv);
#pragma unroll
              for (int p = 0; p < P; ++p) acc[i] += bv[p] * hx[e][p];
            }
          }
        }
      }
    }
  }
  warp_add(rr, sw);
  if (DOTS) {
    warp_add(tt, sw + (k + 1) * VP_WARPS);
#pragma unroll
    for (int i = 0; i < KMAX; ++i)
      if (i < k) warp_add(acc[i], sw + (1 + i) * VP_WARPS);
  }
  block_partials(sw, m, part);
  last_block_sums(part, m, out, counter, red);
}

// y = a x + b y and x = alpha src over packets (grid-stride).  With a or b equal to 1
// the update is one fused multiply-add per element (the FP64 pipe is the bound of
// these kernels on this GPU, not HBM).
__global__ void k_axpby_p(double a, const double *__restrict__ x, double b, double *__restrict__ y, long long np) {
  const int form = b == 1.0 ? 1 : (a == 1.0 ? 2 : 0);
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < np; q += (long long)gridDim.x * blockDim.x) {
    double xv[2], yv[2];
    pk_ld(x, q, xv);
    pk_ld((const double *)y, q, yv);
#pragma unroll
    for (int p = 0; p < 2; ++p)
      yv[p] = form == 1 ? fma(a, xv[p], yv[p]) : form == 2 ? fma(b, yv[p], xv[p]) : a * xv[p] + b * yv[p];
    pk_st(y, q, yv);
  }
}
template <typename T>
__global__ void k_scale_p(T *x, const T *src, double alpha, long long np) {
  constexpr int P = Pk<T>::P;
  const T al = (T)alpha;
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < np; q += (long long)gridDim.x * blockDim.x) {
    T v[P];
    pk_ld(src, q, v);
#pragma unroll
    for (int p = 0; p < P; ++p) v[p] = al * v[p];
    pk_st(x, q, v);
  }
}

// ------------------------------------------------------------------ correction solve
// One step of the preconditioned conjugate gradients on P (H - theta) P t = -r of the
// Jacobi-Davidson refinement (P projects out V_0 .. V_nk-1) in four passes, FP64:
//   shift    q -= theta p,                 out = V^T q
//   project  q -= V c,                     out = p . q
//   step     x += alpha p, r -= alpha q, z = r * rinv,   out = [r . z, r . r, V^T z]
//   turn     p = (z - V d) + beta p
// 21 vector reads and writes at nk = 1, where a kernel per operation with two
// Gram-Schmidt passes per projection took 36 and twelve launches.  One pass is enough
// here: it leaves 2^-53 of the vector, and the solve is stopped at a 50th of its start.
// VEC: elements a thread takes at a time (2: 16-byte loads, for even counts).  Sums: per
// thread, then a warp adds a column of the block's threads from shared memory, then
// last_block_lanes.  One GB300, CAS(14,14), one root: 0.70 -> 0.36 ms an inner iteration.
constexpr int JD_T = 256;
constexpr int JD_COLS = 8;  // columns reduced at a time

template <int VEC>
struct JdV {
  double v[VEC];
};
template <int VEC>
__device__ __forceinline__ JdV<VEC> jd_ld(const double *p, long long i) {
  JdV<VEC> r;
  if constexpr (VEC == 2) {
    const double2 t = reinterpret_cast<const double2 *>(p)[i];
    r.v[0] = t.x;
    r.v[1] = t.y;
  } else {
    r.v[0] = p[i];
  }
  return r;
}
template <int VEC>
__device__ __forceinline__ void jd_st(double *p, long long i, const JdV<VEC> &x) {
  if constexpr (VEC == 2)
    reinterpret_cast<double2 *>(p)[i] = make_double2(x.v[0], x.v[1]);
  else
    p[i] = x.v[0];
}

// part[block][c] = sum of the block's acc[c], c < m <= M; then the last block's totals.
template <int M>
__device__ __forceinline__ void jd_reduce(const double (&acc)[M], int m, double *part, double *out, unsigned *counter) {
  __shared__ double red[JD_COLS][JD_T + 1];
  const int lane = threadIdx.x & 31, warps = blockDim.x >> 5;
#pragma unroll
  for (int c0 = 0; c0 < M; c0 += JD_COLS) {
    if (c0 < m) {
      __syncthreads();
#pragma unroll
      for (int c = 0; c < JD_COLS; ++c)
        if (c0 + c < M) red[c][threadIdx.x] = acc[c0 + c < M ? c0 + c : 0];
      __syncthreads();
      for (int c = threadIdx.x >> 5; c < JD_COLS && c0 + c < m; c += warps) {
        double t = 0.0;
        for (int k = lane; k < (int)blockDim.x; k += 32) t += red[c][k];
        t = warp_sum(t);
        if (lane == 0) part[(long long)blockIdx.x * m + c0 + c] = t;
      }
    }
  }
  last_block_lanes(part, m, out, counter);
}

template <int VEC, int KM>
__global__ void __launch_bounds__(JD_T) k_jd_shift(double *__restrict__ q, const double *__restrict__ p, double theta,
                                                   const double *__restrict__ V, int nk, long long ld, long long n,
                                                   double *__restrict__ part, double *__restrict__ out,
                                                   unsigned *counter) {
  double acc[KM];
#pragma unroll
  for (int k = 0; k < KM; ++k) acc[k] = 0.0;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    JdV<VEC> y = jd_ld<VEC>(q, i);
    const JdV<VEC> x = jd_ld<VEC>(p, i);
#pragma unroll
    for (int e = 0; e < VEC; ++e) y.v[e] = fma(-theta, x.v[e], y.v[e]);
    jd_st<VEC>(q, i, y);
#pragma unroll
    for (int k = 0; k < KM; ++k)
      if (k < nk) {
        const JdV<VEC> b = jd_ld<VEC>(V + (long long)k * ld, i);
#pragma unroll
        for (int e = 0; e < VEC; ++e) acc[k] = fma(b.v[e], y.v[e], acc[k]);
      }
  }
  jd_reduce(acc, nk, part, out, counter);
}

template <int VEC, int KM>
__global__ void __launch_bounds__(JD_T) k_jd_project(double *__restrict__ q, const double *__restrict__ p,
                                                     const double *__restrict__ V, int nk, long long ld,
                                                     const double *__restrict__ c, long long n,
                                                     double *__restrict__ part, double *__restrict__ out,
                                                     unsigned *counter) {
  double ck[KM], acc[1] = {0.0};
#pragma unroll
  for (int k = 0; k < KM; ++k) ck[k] = k < nk ? c[k] : 0.0;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    JdV<VEC> y = jd_ld<VEC>(q, i);
    const JdV<VEC> x = jd_ld<VEC>(p, i);
#pragma unroll
    for (int k = 0; k < KM; ++k)
      if (k < nk) {
        const JdV<VEC> b = jd_ld<VEC>(V + (long long)k * ld, i);
#pragma unroll
        for (int e = 0; e < VEC; ++e) y.v[e] = fma(-ck[k], b.v[e], y.v[e]);
      }
    jd_st<VEC>(q, i, y);
#pragma unroll
    for (int e = 0; e < VEC; ++e) acc[0] = fma(x.v[e], y.v[e], acc[0]);
  }
  jd_reduce(acc, 1, part, out, counter);
}

template <int VEC, int KM>
__global__ void __launch_bounds__(JD_T) k_jd_step(double alpha, const double *__restrict__ p, const double *__restrict__ q,
                                                  double *__restrict__ x, double *__restrict__ r,
                                                  const double *__restrict__ rinv, double *__restrict__ z,
                                                  const double *__restrict__ V, int nk, long long ld, long long n,
                                                  double *__restrict__ part, double *__restrict__ out,
                                                  unsigned *counter) {
  double acc[KM + 2];
#pragma unroll
  for (int k = 0; k < KM + 2; ++k) acc[k] = 0.0;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const JdV<VEC> pv = jd_ld<VEC>(p, i), qv = jd_ld<VEC>(q, i), iv = jd_ld<VEC>(rinv, i);
    JdV<VEC> xv = jd_ld<VEC>(x, i), rv = jd_ld<VEC>(r, i), zv;
#pragma unroll
    for (int e = 0; e < VEC; ++e) {
      xv.v[e] = fma(alpha, pv.v[e], xv.v[e]);
      rv.v[e] = fma(-alpha, qv.v[e], rv.v[e]);
      zv.v[e] = rv.v[e] * iv.v[e];
      acc[0] = fma(rv.v[e], zv.v[e], acc[0]);
      acc[1] = fma(rv.v[e], rv.v[e], acc[1]);
    }
    jd_st<VEC>(x, i, xv);
    jd_st<VEC>(r, i, rv);
    jd_st<VEC>(z, i, zv);
#pragma unroll
    for (int k = 0; k < KM; ++k)
      if (k < nk) {
        const JdV<VEC> b = jd_ld<VEC>(V + (long long)k * ld, i);
#pragma unroll
        for (int e = 0; e < VEC; ++e) acc[2 + k] = fma(b.v[e], zv.v[e], acc[2 + k]);
      }
  }
  jd_reduce(acc, nk + 2, part, out, counter);
}

template <int VEC, int KM>
__global__ void __launch_bounds__(JD_T) k_jd_turn(double *__restrict__ p, const double *__restrict__ z, double beta,
                                                  const double *__restrict__ V, int nk, long long ld,
                                                  const double *__restrict__ d, long long n) {
  double dk[KM];
#pragma unroll
  for (int k = 0; k < KM; ++k) dk[k] = k < nk ? d[k] : 0.0;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    JdV<VEC> y = jd_ld<VEC>(z, i);
    const JdV<VEC> x = jd_ld<VEC>(p, i);
#pragma unroll
    for (int k = 0; k < KM; ++k)
      if (k < nk) {
        const JdV<VEC> b = jd_ld<VEC>(V + (long long)k * ld, i);
#pragma unroll
        for (int e = 0; e < VEC; ++e) y.v[e] = fma(-dk[k], b.v[e], y.v[e]);
      }
#pragma unroll
    for (int e = 0; e < VEC; ++e) y.v[e] = fma(beta, x.v[e], y.v[e]);
    jd_st<VEC>(p, i, y);
  }
}

// ------------------------------------------------------------------ host wrappers

// Partials of the reductions in the context's small scratch, and the arrival counter
// of the fused second pass (zeroed once; every reduction leaves it at zero).
static int part_buffer(forte_ctx *ctx, size_t doubles, double **p, unsigned **counter) {
  int rc = ctx->sc_small.ensure(sizeof(double) * (doubles + 64));
  if (rc) return rc;
  *p = (double *)ctx->sc_small.ptr;
  if (!ctx->d_vk_count) {
    FORTE_CUDA_TRY(dev_alloc(&ctx->d_vk_count, sizeof(unsigned)));
    FORTE_CUDA_TRY(cudaMemsetAsync(ctx->d_vk_count, 0, sizeof(unsigned), ctx->stream));
  }
  *counter = ctx->d_vk_count;
  return FORTE_OK;
}

// Packet kernels apply when the count and the leading dimension are multiples of the
// packet (16 bytes) and every vector base is 16-byte aligned.
template <typename T>
static bool vp_ok(long long n, long long ld, std::initializer_list<const void *> ptrs) {
  constexpr long long P = Pk<T>::P;
  if (n % P != 0 || ld % P != 0) return false;
  for (const void *q : ptrs)
    if (q && ((uintptr_t)q & 15u) != 0) return false;
  return true;
}
static unsigned vs_blocks(long long n) { return (unsigned)std::max<long long>(1, (n + VS_CHUNK - 1) / VS_CHUNK); }
// persistent grid: VP_BPS resident blocks of VK_THREADS per SM, at least one block
static unsigned vp_grid(const forte_ctx *ctx, long long np) {
  int nsm = 0;
  if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device) != cudaSuccess || nsm <= 0) {
    cudaGetLastError();
    nsm = 152;
  }
  const long long nch = (np + VP_CH - 1) / VP_CH;
  return (unsigned)std::max<long long>(1, std::min<long long>(nch, (long long)VP_BPS * nsm));
}

template <typename T>
static int vk_multidot_t(forte_ctx *ctx, const T *V, int nv, long long ld, const T *x, long long n, double *out) {
  if (nv <= 0) return FORTE_OK;
  if (nv > VK_MAXV) { set_error("multidot: too many vectors (%d)", nv); return FORTE_ERR_ARG; }
  const bool vs = sizeof(T) == 8 && n <= VS_MAX_N, pk = vp_ok<T>(n, ld, {V, x});
  const unsigned nb = vs ? vs_blocks(n) : pk ? vp_grid(ctx, n / Pk<T>::P) : vk_blocks(n);
  double *part;
  unsigned *cnt;
  int rc = part_buffer(ctx, (size_t)nb * nv, &part, &cnt);
  if (rc) return rc;
  FORTE_PROF(ctx, "multidot");
  if (vs) {
    if constexpr (sizeof(T) == 8) k_multidot_s<<<nb, VS_T, 0, ctx->stream>>>(V, nv, ld, x, n, part, out, cnt);
  } else if (pk && nv <= 4)
    k_multidot_u<T, 4><<<nb, VK_THREADS, 0, ctx->stream>>>(V, nv, ld, x, n / Pk<T>::P, part, out, cnt);
  else if (pk && nv <= 8)
    k_multidot_u<T, 8><<<nb, VK_THREADS, 0, ctx->stream>>>(V, nv, ld, x, n / Pk<T>::P, part, out, cnt);
  else if (pk && nv <= 16)
    k_multidot_u<T, 16><<<nb, VK_THREADS, 0, ctx->stream>>>(V, nv, ld, x, n / Pk<T>::P, part, out, cnt);
  else if (pk)
    k_multidot_p<T><<<nb, VK_THREADS, 0, ctx->stream>>>(V, nv, ld, x, n / Pk<T>::P, part, out, cnt);
  else
    k_multidot<T><<<nb, VK_THREADS, 0, ctx->stream>>>(V, nv, ld, x, n, part, out, cnt);
  FORTE_LAUNCH_CHECK();
  return FORTE_OK;
}

template <typename T>
static int vk_combine_t(forte_ctx *ctx, const T *V, int nv, long long ld, const double *coef, int ncomb, T *out,
                        long long ldo, long long n) {
  if (nv > VK_MAXV || ncomb > 64) { set_error("combine: too many vectors"); return FORTE_ERR_ARG; }
  unsigned nb = (unsigned)std::min<long long>((n + 255) / 256, 152LL * 16);
  // outputs in groups of 8, 4, 2, 1 (each group streams V once)
  for (int c0 = 0; c0 < ncomb;) {
    const int left = ncomb - c0, g = left >= 8 ? 8 : left >= 4 ? 4 : left >= 2 ? 2 : 1;
    FORTE_PROF(ctx, "combine");
    if (g == 8)
      k_combine<8, T><<<nb, VK_THREADS, 0, ctx->stream>>>(V, nv, ld, coef, ncomb, c0, out, ldo, n);
    else if (g == 4)
      k_combine<4, T><<<nb, VK_THREADS, 0, ctx->stream>>>(V, nv, ld, coef, ncomb, c0, out, ldo, n);
    else if (g == 2)
      k_combine<2, T><<<nb, VK_THREADS, 0, ctx->stream>>>(V, nv, ld, coef, ncomb, c0, out, ldo, n);
    else
      k_combine<1, T><<<nb, VK_THREADS, 0, ctx->stream>>>(V, nv, ld, coef, ncomb, c0, out, ldo, n);
    FORTE_LAUNCH_CHECK();
    c0 += g;
  }
  return FORTE_OK;
}

template <typename T>
static int vk_residual_precond_t(forte_ctx *ctx, const T *B, const T *S, int k, long long ld, const double *u,
                                 double theta, double guard, T *t, double *rnorm2, long long n, double *dots) {
  if (k > VK_MAXV) { set_error("residual: subspace too large (%d)", k); return FORTE_ERR_ARG; }
  const bool vs = sizeof(T) == 8 && n <= VS_MAX_N, pk = vp_ok<T>(n, ld, {B, S, t, ctx->d_hdiag});
  if (dots && !pk && !vs) return -1;  // no fused dots: the caller forms them with vk_orth_update
  const unsigned nb = vs ? vs_blocks(n) : pk ? vp_grid(ctx, 2 * (n / Pk<T>::P)) : vk_blocks(n);  // chunks of half the packets
  const int m = dots ? k + 2 : 1;
  double *part;
  unsigned *cnt;
  int rc = part_buffer(ctx, (size_t)nb * m, &part, &cnt);
  if (rc) return rc;
  FORTE_PROF(ctx, "residual_precond");
  const long long npk = n / Pk<T>::P;
  const double *hd = ctx->d_hdiag;
#define FORTE_RESID_U(KM)                                                                                            \
  do {                                                                                                               \
    if (dots)                                                                                                        \
      k_residual_precond_u<T, true, 2, KM><<<nb, VK_THREADS, 0, ctx->stream>>>(B, S, k, ld, u, theta, hd, guard, t,  \
                                                                               npk, part, dots, cnt);                \
    else                                                                                                             \
      k_residual_precond_u<T, false, 2, KM><<<nb, VK_THREADS, 0, ctx->stream>>>(B, S, k, ld, u, theta, hd, guard, t, \
                                                                                npk, part, rnorm2, cnt);             \
  } while (0)
  if (vs) {
    if constexpr (sizeof(T) == 8) {
      if (dots)
        k_residual_precond_s<true><<<nb, VS_T, 0, ctx->stream>>>(B, S, k, ld, u, theta, hd, guard, t, n, part, dots, cnt);
      else
        k_residual_precond_s<false><<<nb, VS_T, 0, ctx->stream>>>(B, S, k, ld, u, theta, hd, guard, t, n, part, rnorm2, cnt);
    }
  } else if (pk && k <= 4)
    FORTE_RESID_U(4);
  else if (pk && k <= 8)
    FORTE_RESID_U(8);
  else if (pk && k <= 16 && sizeof(T) == 4)  // FP64 accumulators for 16 vectors would spill
    FORTE_RESID_U(16);
#undef FORTE_RESID_U
  else if (pk && dots)
    k_residual_precond_p<T, true, 2><<<nb, VK_THREADS, 0, ctx->stream>>>(B, S, k, ld, u, theta, hd, guard, t, npk,
                                                                         part, dots, cnt);
  else if (pk)
    k_residual_precond_p<T, false, 2><<<nb, VK_THREADS, 0, ctx->stream>>>(B, S, k, ld, u, theta, hd, guard, t, npk,
                                                                          part, rnorm2, cnt);
  else
    k_residual_precond<T><<<nb, VK_THREADS, 0, ctx->stream>>>(B, S, k, ld, u, theta, ctx->d_hdiag, guard, t, n,
                                                              part, rnorm2, cnt);
  FORTE_LAUNCH_CHECK();
  return FORTE_OK;
}

// d[i] *= s (i < k), d[k] *= s^2: dots and squared norm of a vector scaled by s
__global__ void k_rescale_dots(double *d, int k, double s) {
  for (int i = threadIdx.x; i <= k; i += blockDim.x) d[i] *= (i < k) ? s : s * s;
}
static int vk_rescale_dots(forte_ctx *ctx, double *d, int k, double s) {
  FORTE_PROF(ctx, "rescale_dots");
  k_rescale_dots<<<1, 64, 0, ctx->stream>>>(d, k, s);
  FORTE_LAUNCH_CHECK();
  return FORTE_OK;
}

template <typename T>
static int vk_orth_update_t(forte_ctx *ctx, const T *B, int k, long long ld, const double *c, const T *t_in,
                            T *t_out, double *dots_out, long long n, bool dots, double scale) {
  if (k + 1 > VK_MAXV) { set_error("orth: subspace too large (%d)", k); return FORTE_ERR_ARG; }
  const bool vs = sizeof(T) == 8 && n <= VS_MAX_N, pk = vp_ok<T>(n, ld, {B, t_in, t_out});
  const unsigned nb = vs ? vs_blocks(n) : pk ? vp_grid(ctx, n / Pk<T>::P) : vk_blocks(n);
  double *part;
  unsigned *cnt;
  int rc = part_buffer(ctx, (size_t)nb * (k + 1), &part, &cnt);
  if (rc) return rc;
  if (!pk && !vs && scale != 1.0) {  // element path: the scale is a separate pass
    if ((rc = vk_orth_update_t(ctx, B, k, ld, c, t_in, t_out, dots_out, n, dots, 1.0))) return rc;
    if ((rc = vk_scale(ctx, t_out, t_out, scale, n))) return rc;
    // |t_out|^2 and the dots scale with scale^2 and scale
    return vk_rescale_dots(ctx, dots_out, k, scale);
  }
  FORTE_PROF(ctx, "orth_update");
  const long long npk = n / Pk<T>::P;
#define FORTE_ORTH_U(KM)                                                                                    \
  do {                                                                                                      \
    if (dots)                                                                                               \
      k_orth_update_u<T, true, KM><<<nb, VK_THREADS, 0, ctx->stream>>>(B, k, ld, c, t_in, t_out, npk, scale, \
                                                                       part, dots_out, cnt);                \
    else                                                                                                    \
      k_orth_update_u<T, false, KM><<<nb, VK_THREADS, 0, ctx->stream>>>(B, k, ld, c, t_in, t_out, npk,      \
                                                                        scale, part, dots_out, cnt);        \
  } while (0)
  if (vs) {
    if constexpr (sizeof(T) == 8) {
      if (dots)
        k_orth_update_s<true><<<nb, VS_T, 0, ctx->stream>>>(B, k, ld, c, t_in, t_out, n, scale, part, dots_out, cnt);
      else
        k_orth_update_s<false><<<nb, VS_T, 0, ctx->stream>>>(B, k, ld, c, t_in, t_out, n, scale, part, dots_out, cnt);
    }
  } else if (pk && k <= 4)
    FORTE_ORTH_U(4);
  else if (pk && k <= 8)
    FORTE_ORTH_U(8);
  else if (pk && k <= 16 && sizeof(T) == 4)
    FORTE_ORTH_U(16);
#undef FORTE_ORTH_U
  else if (pk && dots)
    k_orth_update_p<T, true><<<nb, VK_THREADS, 0, ctx->stream>>>(B, k, ld, c, t_in, t_out, n / Pk<T>::P, scale,
                                                                 part, dots_out, cnt);
  else if (pk)
    k_orth_update_p<T, false><<<nb, VK_THREADS, 0, ctx->stream>>>(B, k, ld, c, t_in, t_out, n / Pk<T>::P, scale,
                                                                  part, dots_out, cnt);
  else if (dots)
    k_orth_update<T, true><<<nb, VK_THREADS, 0, ctx->stream>>>(B, k, ld, c, t_in, t_out, n, part, dots_out, cnt);
  else
    k_orth_update<T, false><<<nb, VK_THREADS, 0, ctx->stream>>>(B, k, ld, c, t_in, t_out, n, part, dots_out, cnt);
  FORTE_LAUNCH_CHECK();
  return FORTE_OK;
}

template <typename T>
static int vk_scale_t(forte_ctx *ctx, T *x, const T *src, double alpha, long long n) {
  FORTE_PROF(ctx, "scale");
  if (vp_ok<T>(n, n, {x, src})) {
    const long long np = n / Pk<T>::P;
    k_scale_p<T><<<(unsigned)std::min<long long>((np + 255) / 256, 152LL * 16), 256, 0, ctx->stream>>>(x, src, alpha,
                                                                                                       np);
  } else {
    k_scale<T><<<(unsigned)std::min<long long>((n + 255) / 256, 152LL * 16), 256, 0, ctx->stream>>>(x, src, alpha, n);
  }
  FORTE_LAUNCH_CHECK();
  return FORTE_OK;
}

int vk_multidot(forte_ctx *ctx, const double *V, int nv, long long ld, const double *x, long long n, double *out) {
  return vk_multidot_t(ctx, V, nv, ld, x, n, out);
}
int vk_multidot(forte_ctx *ctx, const float *V, int nv, long long ld, const float *x, long long n, double *out) {
  return vk_multidot_t(ctx, V, nv, ld, x, n, out);
}
int vk_combine(forte_ctx *ctx, const double *V, int nv, long long ld, const double *coef, int ncomb, double *out,
               long long ldo, long long n) {
  return vk_combine_t(ctx, V, nv, ld, coef, ncomb, out, ldo, n);
}
int vk_combine(forte_ctx *ctx, const float *V, int nv, long long ld, const double *coef, int ncomb, float *out,
               long long ldo, long long n) {
  return vk_combine_t(ctx, V, nv, ld, coef, ncomb, out, ldo, n);
}
int vk_residual_precond(forte_ctx *ctx, const double *B, const double *S, int k, long long ld, const double *u,
                        double theta, double guard, double *t, double *rnorm2, long long n, double *dots) {
  return vk_residual_precond_t(ctx, B, S, k, ld, u, theta, guard, t, rnorm2, n, dots);
}
int vk_residual_precond(forte_ctx *ctx, const float *B, const float *S, int k, long long ld, const double *u,
                        double theta, double guard, float *t, double *rnorm2, long long n, double *dots) {
  return vk_residual_precond_t(ctx, B, S, k, ld, u, theta, guard, t, rnorm2, n, dots);
}
int vk_orth_update(forte_ctx *ctx, const double *B, int k, long long ld, const double *c, const double *t_in,
                   double *t_out, double *dots_out, long long n, bool dots, double scale) {
  return vk_orth_update_t(ctx, B, k, ld, c, t_in, t_out, dots_out, n, dots, scale);
}
int vk_orth_update(forte_ctx *ctx, const float *B, int k, long long ld, const double *c, const float *t_in,
                   float *t_out, double *dots_out, long long n, bool dots, double scale) {
  return vk_orth_update_t(ctx, B, k, ld, c, t_in, t_out, dots_out, n, dots, scale);
}
int vk_scale(forte_ctx *ctx, double *x, const double *src, double alpha, long long n) {
  return vk_scale_t(ctx, x, src, alpha, n);
}
int vk_scale(forte_ctx *ctx, float *x, const float *src, double alpha, long long n) {
  return vk_scale_t(ctx, x, src, alpha, n);
}
template <typename TI, typename TO>
static int vk_convert_t(forte_ctx *ctx, const TI *x, TO *y, long long n) {
  unsigned nb = (unsigned)std::min<long long>((n + 255) / 256, 152LL * 16);
  FORTE_PROF(ctx, "convert");
  k_convert<TI, TO><<<nb, 256, 0, ctx->stream>>>(x, y, n);
  FORTE_LAUNCH_CHECK();
  return FORTE_OK;
}
int vk_convert(forte_ctx *ctx, const double *x, float *y, long long n) { return vk_convert_t(ctx, x, y, n); }
int vk_convert(forte_ctx *ctx, const float *x, double *y, long long n) { return vk_convert_t(ctx, x, y, n); }

int vk_axpby(forte_ctx *ctx, double a, const double *x, double b, double *y, long long n) {
  FORTE_PROF(ctx, "axpby");
  if (vp_ok<double>(n, n, {x, y})) {
    const long long np = n / 2;
    k_axpby_p<<<(unsigned)std::min<long long>((np + 255) / 256, 152LL * 16), 256, 0, ctx->stream>>>(a, x, b, y, np);
  } else {
    k_axpby<<<(unsigned)std::min<long long>((n + 255) / 256, 152LL * 16), 256, 0, ctx->stream>>>(a, x, b, y, n);
  }
  FORTE_LAUNCH_CHECK();
  return FORTE_OK;
}

// Launch shape of the correction-solve kernels: packets when the count, the leading
// dimension and the bases allow 16-byte loads.
struct JdShape {
  bool vec;
  long long n;  // packets or elements
  unsigned nb, nt;
};
static JdShape jd_shape(const forte_ctx *ctx, long long n, long long ld, std::initializer_list<const void *> ptrs) {
  JdShape s;
  s.vec = vp_ok<double>(n, ld, ptrs);
  s.n = s.vec ? n / 2 : n;
  s.nt = n <= VS_MAX_N ? 64 : JD_T;  // short vectors: more, smaller blocks
  int nsm = 0;
  if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device) != cudaSuccess || nsm <= 0) {
    cudaGetLastError();
    nsm = 152;
  }
  s.nb = (unsigned)std::max<long long>(1, std::min<long long>((s.n + s.nt - 1) / s.nt, 4LL * nsm));
  return s;
}
// one launch of kernel<VEC, KM>, KM the smallest of 1, 2, 4, 8, 32 that holds nk
#define FORTE_JD(kernel, ...)                                                                       \
  do {                                                                                              \
    auto go = [&](auto km) {                                                                        \
      constexpr int KM = decltype(km)::value;                                                       \
      if (sh.vec)                                                                                   \
        kernel<2, KM><<<sh.nb, sh.nt, 0, ctx->stream>>>(__VA_ARGS__);                               \
      else                                                                                          \
        kernel<1, KM><<<sh.nb, sh.nt, 0, ctx->stream>>>(__VA_ARGS__);                               \
    };                                                                                              \
    if (nk <= 1) go(std::integral_constant<int, 1>{});                                              \
    else if (nk <= 2) go(std::integral_constant<int, 2>{});                                         \
    else if (nk <= 4) go(std::integral_constant<int, 4>{});                                         \
    else if (nk <= 8) go(std::integral_constant<int, 8>{});                                         \
    else go(std::integral_constant<int, 32>{});                                                     \
  } while (0)

int vk_jd_shift(forte_ctx *ctx, double *q, const double *p, double theta, const double *V, int nk, long long n,
                double *out) {
  if (nk < 1 || nk > 32) { set_error("correction solve: %d vectors", nk); return FORTE_ERR_ARG; }
  const JdShape sh = jd_shape(ctx, n, n, {q, p, V});
  double *part;
  unsigned *cnt;
  int rc = part_buffer(ctx, (size_t)sh.nb * nk, &part, &cnt);
  if (rc) return rc;
  FORTE_PROF(ctx, "jd_shift");
  FORTE_JD(k_jd_shift, q, p, theta, V, nk, n, sh.n, part, out, cnt);
  FORTE_LAUNCH_CHECK();
  return FORTE_OK;
}
int vk_jd_project(forte_ctx *ctx, double *q, const double *p, const double *V, int nk, const double *c, long long n,
                  double *out) {
  const JdShape sh = jd_shape(ctx, n, n, {q, p, V});
  double *part;
  unsigned *cnt;
  int rc = part_buffer(ctx, (size_t)sh.nb, &part, &cnt);
  if (rc) return rc;
  FORTE_PROF(ctx, "jd_project");
  FORTE_JD(k_jd_project, q, p, V, nk, n, c, sh.n, part, out, cnt);
  FORTE_LAUNCH_CHECK();
  return FORTE_OK;
}
int vk_jd_step(forte_ctx *ctx, double alpha, const double *p, const double *q, double *x, double *r, const double *rinv,
               double *z, const double *V, int nk, long long n, double *out) {
  const JdShape sh = jd_shape(ctx, n, n, {p, q, x, r, rinv, z, V});
  double *part;
  unsigned *cnt;
  int rc = part_buffer(ctx, (size_t)sh.nb * (nk + 2), &part, &cnt);
  if (rc) return rc;
  FORTE_PROF(ctx, "jd_step");
  FORTE_JD(k_jd_step, alpha, p, q, x, r, rinv, z, V, nk, n, sh.n, part, out, cnt);
  FORTE_LAUNCH_CHECK();
  return FORTE_OK;
}
int vk_jd_turn(forte_ctx *ctx, double *p, const double *z, double beta, const double *V, int nk, const double *d,
               long long n) {
  const JdShape sh = jd_shape(ctx, n, n, {p, z, V});
  FORTE_PROF(ctx, "jd_turn");
  FORTE_JD(k_jd_turn, p, z, beta, V, nk, n, d, sh.n);
  FORTE_LAUNCH_CHECK();
  return FORTE_OK;
}
#undef FORTE_JD

int vk_precond_inv(forte_ctx *ctx, double theta, double guard, double *rinv, long long n) {
  FORTE_PROF(ctx, "precond_inv");
  k_precond_inv<<<(unsigned)std::min<long long>((n + 255) / 256, 152LL * 16), 256, 0, ctx->stream>>>(
      ctx->d_hdiag, theta, guard, rinv, n);
  FORTE_LAUNCH_CHECK();
  return FORTE_OK;
}

// k smallest entries (ties: lowest index), host output idx_out[k].
int vk_argmin_k(forte_ctx *ctx, const double *x, long long n, int k, long long *idx_out) {
  const unsigned nb = (unsigned)std::min<long long>((n + VK_THREADS - 1) / VK_THREADS, 1024);
  size_t need = sizeof(double) * nb + sizeof(long long) * nb + sizeof(long long) * (k + 1);
  int rc = ctx->sc_small.ensure(need + 256);
  if (rc) return rc;
  double *bval = (double *)ctx->sc_small.ptr;
  long long *bidx = (long long *)(bval + nb);
  long long *excl = bidx + nb;
  std::vector<double> hv(nb);
  std::vector<long long> hi(nb);
  for (int r = 0; r < k; ++r) {
    if (r > 0)
      FORTE_CUDA_TRY(cudaMemcpyAsync(excl, idx_out, sizeof(long long) * r, cudaMemcpyHostToDevice, ctx->stream));
    {
      FORTE_PROF(ctx, "argmin");
      k_argmin<<<nb, VK_THREADS, 0, ctx->stream>>>(x, n, excl, r, bval, bidx);
    FORTE_LAUNCH_CHECK();
    }
    FORTE_CUDA_TRY(cudaMemcpyAsync(hv.data(), bval, sizeof(double) * nb, cudaMemcpyDeviceToHost, ctx->stream));
    FORTE_CUDA_TRY(cudaMemcpyAsync(hi.data(), bidx, sizeof(long long) * nb, cudaMemcpyDeviceToHost, ctx->stream));
    FORTE_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
    double best = INFINITY;
    long long bi = -1;
    for (unsigned b = 0; b < nb; ++b) {
      if (hi[b] < 0) continue;
      if (bi < 0 || hv[b] < best || (hv[b] == best && hi[b] < bi)) { best = hv[b]; bi = hi[b]; }
    }
    if (bi < 0) { set_error("argmin: fewer than %d entries", k); return FORTE_ERR_ARG; }
    idx_out[r] = bi;
  }
  return FORTE_OK;
}

int vk_any_nonfinite(forte_ctx *ctx, const double *x, long long n, int *flag_host) {
  int rc = ctx->sc_small.ensure(256);
  if (rc) return rc;
  int *flag = (int *)ctx->sc_small.ptr;
  FORTE_CUDA_TRY(cudaMemsetAsync(flag, 0, sizeof(int), ctx->stream));
  unsigned nb = (unsigned)std::min<long long>((n + 255) / 256, 152LL * 8);
  {
    FORTE_PROF(ctx, "nonfinite");
    k_nonfinite<<<nb, 256, 0, ctx->stream>>>(x, n, flag);
  FORTE_LAUNCH_CHECK();
  }
  FORTE_CUDA_TRY(cudaMemcpyAsync(flag_host, flag, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
  FORTE_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
  return FORTE_OK;
}

}  // namespace forte
