// Spin-free 1- and 2-RDMs (step a9), Sec. II.A.1 Eqs. (gamma_1), (gamma_2)
// summed over spin:
//   gamma_pq   = <bra| E_pq |ket>
//   Gamma_pqrs = <bra| E_pq E_rs |ket> - d_qr gamma_ps = <E_qp bra | E_rs ket> - d_qr gamma_ps
// The 2-RDM is a Gram matrix of the one-body images D^{rs} = E_rs |ket>
// (alpha and beta parts added), taken over all determinants.
#include <algorithm>

#include "forte_internal.h"

namespace forte {

__device__ __forceinline__ double warp_sum_r(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// part[row][pq] = sum_{e in L(row), pq_e = pq} s_e * <bra[J_e,:], ket[row,:]>
// (rows of one spin; the other spin's strings run along the columns).
// A warp forms one entry's dot product at a time.  The entries that do not move the row
// (pq = pp) share one dot product, and for bra == ket (sym) those with p < q are left
// out: gamma is symmetric.  FP64 pipe and L2: 25 instead of 56 dots a row at 7 of 14
// orbitals; CAS(14,14), both spins: 3.6 -> 1.33 ms.
__global__ void __launch_bounds__(256) k_g1_part(const Repl *__restrict__ list, int nk, const double *__restrict__ bra,
                                                 const double *__restrict__ ket, long long ncol, int n, int sym,
                                                 double *__restrict__ part) {
  __shared__ double acc[256];
  const long long row = blockIdx.x;
  const int n2 = n * n, lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < n2; i += blockDim.x) acc[i] = 0.0;
  __syncthreads();
  const double *kr = ket + row * ncol;
  const Repl *L = list + row * nk;
  for (int e = threadIdx.x >> 5; e <= nk; e += blockDim.x >> 5) {  // e == nk: the row with itself
    Repl r = {};
    if (e < nk) {
      r = L[e];
      if (r.J == row || (sym && r.pq / n < r.pq % n)) continue;
    } else {
      r.J = (int)row;
    }
    const double *br = bra + (long long)r.J * ncol;
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    long long c = lane;
    for (; c + 96 < ncol; c += 128) {
      s0 = fma(br[c], kr[c], s0);
      s1 = fma(br[c + 32], kr[c + 32], s1);
      s2 = fma(br[c + 64], kr[c + 64], s2);
      s3 = fma(br[c + 96], kr[c + 96], s3);
    }
    for (; c < ncol; c += 32) s0 = fma(br[c], kr[c], s0);
    const double t = warp_sum_r((s0 + s1) + (s2 + s3));
    if (e < nk) {
      if (lane == 0) acc[r.pq] = r.sgn * t;
    } else {
      for (int f = lane; f < nk; f += 32)
        if (L[f].J == row) acc[L[f].pq] = L[f].sgn * t;
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n2; i += blockDim.x) part[row * n2 + i] = acc[i];
}

// out[j] = sum_b part[b][j] + sum_b part2[b][j]   (grid.x = n * n; sym: the lower
// triangle stands for both)
__global__ void k_sum_cols2(const double *__restrict__ part, long long nb1, const double *__restrict__ part2,
                            long long nb2, int n, int sym, double *__restrict__ out) {
  __shared__ double red[32];
  const int m = n * n, p = blockIdx.x / n, q = blockIdx.x % n;
  const int j = sym && p < q ? q * n + p : blockIdx.x;
  double s = 0.0;
  for (long long b = threadIdx.x; b < nb1; b += blockDim.x) s += part[b * m + j];
  for (long long b = threadIdx.x; b < nb2; b += blockDim.x) s += part2[b * m + j];
  s = warp_sum_r(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    out[blockIdx.x] = t;
  }
}

template <typename T>
__global__ void k_transpose_r(const T *__restrict__ X, T *__restrict__ Y, long long R, long long Cc) {
  __shared__ T tile[32][33];
  long long r0 = (long long)blockIdx.y * 32, c0 = (long long)blockIdx.x * 32;
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    long long r = r0 + i, c = c0 + threadIdx.x;
    if (r < R && c < Cc) tile[i][threadIdx.x] = X[r * Cc + c];
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    long long c = c0 + i, r = r0 + threadIdx.x;
    if (r < R && c < Cc) Y[c * R + r] = tile[threadIdx.x][i];
  }
}

// ---- FP64 Grams of the symmetric and antisymmetric one-body images ----------
//
// With S_rs = E_rs + E_sr (r > s), S_rr = E_rr and A_rs = E_rs - E_sr (r > s), a
// normal-ordered RDM of a real state does not change when every pair is transposed,
// so only its components with an even number of A's are not zero:
//   2-RDM: Gamma(S,S), Gamma(A,A);   3-RDM: Gamma(S,S,S), Gamma(A,A,S),
// symmetric in the pairs of one kind.  They are Gram matrices over the determinants,
//   <S_a S_b>     = <S_a C | S_b C>,        <A_a A_b>     = -<A_a C | A_b C>,
//   <S_a S_b S_c> = <S_a C | S_b (S_c C)>,  <A_a A_b S_c> = -<A_a C | A_b (S_c C)>,
// minus the lower-rank terms of the normal ordering, and every element of the full
// RDM is a sum of two (2-RDM) or four (3-RDM) of them.  For r != s at most one of
// E_rs, E_sr acts on a string, so an element of an image is one signed entry of the
// vector per spin.
//
// The FP64 pipe (2 DFMA per clock and SM) bounds this, so the kernel forms as few
// products as it can: n^4 / 4 per determinant for the 2-RDM and about n^6 / 12 for the
// 3-RDM (the full n^2 x n^2 Grams take n^4 and n^6).  Tiles of 3 x 3 waste 3 % on the
// diagonal blocks at n = 12 (4 x 4: 10 %), and shared-memory loads cost little beside
// 9 DFMAs.  The images are built in shared memory, 32 determinants at a time, from the
// vector (L2), so no image is written to memory but the S_c C of the 3-RDM.
// One GB300: CAS(12; 7,5) 1- and 2-RDM 31.1 -> 7.2 ms (image array + 64 x 64 tiles
// before), CAS(9; 5,4) 3-RDM 51.7 -> 2.4 ms (n^2 launches of 64 x 64 tiles before).

constexpr int UV_B = 3;          // tile edge
constexpr int UV_KS = 32;        // determinants per slab
constexpr int UV_THREADS = 320;  // tiles (threads) per block at most
constexpr int UV_KG = 16;        // slab parts within a block at most (few tiles: small n)

// Rows of a slab: S pairs (r >= s), padded to a multiple of the tile edge, then the A
// pairs (r > s), padded the same way.
struct UvShape {
  int n, U, V, Up, Vp, ld;  // ld: odd row stride of a slab (conflict-free column writes)
};

static UvShape uv_shape(int n) {
  UvShape q;
  q.n = n;
  q.U = n * (n + 1) / 2;
  q.V = n * (n - 1) / 2;
  q.Up = (q.U + UV_B - 1) / UV_B * UV_B;
  q.Vp = (q.V + UV_B - 1) / UV_B * UV_B;
  q.ld = (q.Up + q.Vp) | 1;
  return q;
}

// Tiles (bi >= bj) of the S-S block with bj >= c / 3 come first (descending bj, so that
// the tiles a third index c needs, b >= c, are a prefix), then those of the A-A block.
__host__ __device__ __forceinline__ int uv_tiles_s(const UvShape &q, int c) {
  const int m = q.Up / UV_B - c / UV_B;
  return m * (m + 1) / 2;
}
__host__ __device__ __forceinline__ int uv_tiles(const UvShape &q, int c) {
  const int m = q.Vp / UV_B;
  return uv_tiles_s(q, c) + m * (m + 1) / 2;
}
__device__ __forceinline__ void uv_tile(const UvShape &q, int c, int t, int &bi, int &bj, bool &anti) {
  const int ns = uv_tiles_s(q, c);
  anti = t >= ns;
  const int nb = anti ? q.Vp / UV_B : q.Up / UV_B;
  const int x = anti ? t - ns : t;
  int m = (int)((sqrtf(8.0f * (float)x + 1.0f) - 1.0f) * 0.5f);
  while (m * (m + 1) / 2 > x) --m;
  while ((m + 1) * (m + 2) / 2 <= x) ++m;
  bj = nb - 1 - m;
  bi = bj + (x - m * (m + 1) / 2);
}
// Slab parts a block of `threads` threads splits its determinants into when it has `tiles`.
__device__ __forceinline__ int uv_kparts(int threads, int tiles) {
  const int k = threads / (tiles > 0 ? tiles : 1);
  return k < 1 ? 1 : (k > UV_KG ? UV_KG : k);
}

// One spin's part of (S_rs X)[I] or (A_rs X)[I]: entry code of the string it takes,
// (J << 1) | negative, or -1.
__device__ __forceinline__ int uv_source(const int *__restrict__ t, int n, int r, int s, bool anti) {
  int x = t[s * n + r];  // E_sr I: the term of E_rs
  if (x < 0 && r != s) {
    x = t[r * n + s];    // the term of E_sr
    if (x >= 0 && anti) x ^= 1;
  }
  return x;
}

__device__ __forceinline__ double uv_image(const int *__restrict__ ta, const int *__restrict__ tb, int n, int r, int s,
                                           bool anti, const double *__restrict__ X, long long NB, long long ia,
                                           long long ib) {
  const int xa = uv_source(ta, n, r, s, anti), xb = uv_source(tb, n, r, s, anti);
  double a = 0.0, b = 0.0;
  if (xa >= 0) a = X[(long long)(xa >> 1) * NB + ib];
  if (xb >= 0) b = X[ia * NB + (xb >> 1)];
  return ((xa & 1) ? -a : a) + ((xb & 1) ? -b : b);
}

// F[c] = S_c C for every symmetric pair c (grid.y).
__global__ void k_uv_images(const int *__restrict__ denseA, const int *__restrict__ denseB, int n,
                            const double *__restrict__ C, long long NB, long long ND, double *__restrict__ F) {
  int r = 0, c = blockIdx.y;
  while (c > r) c -= ++r;
  const int s = c, n2 = n * n;
  double *Fc = F + (long long)blockIdx.y * ND;
  for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < ND; k += (long long)gridDim.x * blockDim.x) {
    const long long ia = k / NB, ib = k - ia * NB;
    Fc[k] = uv_image(denseA + ia * n2, denseB + ib * n2, n, r, s, false, C, NB, ia, ib);
  }
}

// Block (x, y, z): slabs of split x, third index c0 + y (THREE), tile group z.
//   part[(x * gridDim.y + y) * maxtiles + tile][9]
template <bool THREE>
__global__ void __launch_bounds__(UV_THREADS) k_uv_gram(const int *__restrict__ denseA, const int *__restrict__ denseB,
                                                        UvShape q, const double *__restrict__ C,
                                                        const double *__restrict__ F, long long NB, long long ND,
                                                        int group, int maxtiles, double *__restrict__ part) {
  extern __shared__ double uv_smem[];
  double *Xs = uv_smem;                                       // [UV_KS][ld]
  double *Ys = THREE ? Xs + (size_t)UV_KS * q.ld : Xs;        // [UV_KS][ld]
  __shared__ uint8_t s_r[256 + 2 * UV_B], s_s[256 + 2 * UV_B];
  const int n = q.n, n2 = n * n, rows = q.Up + q.Vp;
  const int c = THREE ? blockIdx.y : 0;
  const int tiles = min(group, uv_tiles(q, c) - (int)blockIdx.z * group);  // of this block
  if (tiles <= 0) return;
  for (int i = threadIdx.x; i < rows; i += blockDim.x) {
    const bool anti = i >= q.Up;
    int x = anti ? i - q.Up : i, r = anti ? 1 : 0;
    const bool pad = x >= (anti ? q.V : q.U);
    while (!pad && x > r - (anti ? 1 : 0)) x -= (anti ? r : r + 1), ++r;
    s_r[i] = pad ? 255 : (uint8_t)r;
    s_s[i] = pad ? 0 : (uint8_t)x;
  }
  const int kparts = uv_kparts(blockDim.x, tiles);
  const int g = threadIdx.x / tiles, t = threadIdx.x - g * tiles;
  const bool active = g < kparts;
  int bi = 0, bj = 0;
  bool anti = false;
  if (active) uv_tile(q, c, blockIdx.z * group + t, bi, bj, anti);
  const double *xr = Xs + (anti ? q.Up : 0) + UV_B * bi, *yr = Ys + (anti ? q.Up : 0) + UV_B * bj;
  double acc[UV_B][UV_B];
#pragma unroll
  for (int i = 0; i < UV_B; ++i)
#pragma unroll
    for (int j = 0; j < UV_B; ++j) acc[i][j] = 0.0;
  const double *Fc = THREE ? F + (long long)c * ND : nullptr;
  const long long nslab = (ND + UV_KS - 1) / UV_KS;
  const long long b0 = nslab * blockIdx.x / gridDim.x, b1 = nslab * (blockIdx.x + 1) / gridDim.x;
  for (long long b = b0; b < b1; ++b) {
    __syncthreads();
    // a warp takes one row of the slab at a time: a lane owns one determinant
    const int lane = threadIdx.x & 31;
    const long long k = b * UV_KS + lane, ia = k / NB, ib = k - ia * NB;
    for (int row = threadIdx.x >> 5; row < rows; row += blockDim.x >> 5) {
      const int r = s_r[row], s = s_s[row];
      const bool an = row >= q.Up;
      double x = 0.0, y = 0.0;
      if (r != 255 && k < ND) {
        x = uv_image(denseA + ia * n2, denseB + ib * n2, n, r, s, an, C, NB, ia, ib);
        if (THREE) y = uv_image(denseA + ia * n2, denseB + ib * n2, n, r, s, an, Fc, NB, ia, ib);
      }
      Xs[lane * q.ld + row] = x;
      if (THREE) Ys[lane * q.ld + row] = y;
    }
    __syncthreads();
    if (active)
      for (int kk = g; kk < UV_KS; kk += kparts) {
        double x[UV_B], y[UV_B];
#pragma unroll
        for (int i = 0; i < UV_B; ++i) x[i] = xr[kk * q.ld + i];
#pragma unroll
        for (int j = 0; j < UV_B; ++j) y[j] = yr[kk * q.ld + j];
#pragma unroll
        for (int i = 0; i < UV_B; ++i)
#pragma unroll
          for (int j = 0; j < UV_B; ++j) acc[i][j] = fma(x[i], y[j], acc[i][j]);
      }
  }
  // the slab parts of the block, added in order
  for (int gg = 1; gg < kparts; ++gg) {
    __syncthreads();
    if (active && g == gg)
#pragma unroll
      for (int e = 0; e < UV_B * UV_B; ++e) uv_smem[t * UV_B * UV_B + e] = acc[e / UV_B][e % UV_B];
    __syncthreads();
    if (g == 0)
#pragma unroll
      for (int e = 0; e < UV_B * UV_B; ++e) acc[e / UV_B][e % UV_B] += uv_smem[t * UV_B * UV_B + e];
  }
  if (g != 0) return;
  double *P = part + (((long long)blockIdx.x * gridDim.y + blockIdx.y) * maxtiles + blockIdx.z * group + t) *
                         (UV_B * UV_B);
#pragma unroll
  for (int e = 0; e < UV_B * UV_B; ++e) P[e] = acc[e / UV_B][e % UV_B];
}

// Pair operator over E: S_rs = E_rs + E_sr, S_rr = E_rr, A_rs = E_rs - E_sr.
struct UvPair {
  int p[2], q[2], cnt;
  double sg[2];
};
__device__ __forceinline__ UvPair uv_pair(int idx, bool anti) {
  int r = anti ? 1 : 0, x = idx;
  while (x > r - (anti ? 1 : 0)) x -= (anti ? r : r + 1), ++r;
  UvPair u;
  u.p[0] = r; u.q[0] = x; u.sg[0] = 1.0;
  u.p[1] = x; u.q[1] = r; u.sg[1] = anti ? -1.0 : 1.0;
  u.cnt = r == x ? 1 : 2;
  return u;
}

// Sum of the partial Gram elements in split order, minus the lower-rank terms of the
// normal ordering: comp = Gamma(S,S[,S]) as [U][U]([U]) and Gamma(A,A[,S]) as
// [V][V]([U]) behind it, all index orders of a component filled.  One thread per tile
// element of one third index (grid.y).
template <bool THREE>
__global__ void k_uv_comp(const double *__restrict__ part, int nsplit, UvShape q, int maxtiles,
                          const double *__restrict__ g1, const double *__restrict__ g2, double *__restrict__ comp) {
  const int n = q.n, c = THREE ? blockIdx.y : 0;
  const int e = blockIdx.x * blockDim.x + threadIdx.x, total = uv_tiles(q, c);
  if (e >= total * UV_B * UV_B) return;
  const int t = e / (UV_B * UV_B), ij = e % (UV_B * UV_B);
  int bi, bj;
  bool anti;
  uv_tile(q, c, t, bi, bj, anti);
  const int a = bi * UV_B + ij / UV_B, b = bj * UV_B + ij % UV_B;
  if (a < b || a >= (anti ? q.V : q.U) || (THREE && !anti && b < c)) return;
  double v = 0.0;
  for (int x = 0; x < nsplit; ++x)
    v += part[(((long long)x * gridDim.y + blockIdx.y) * maxtiles + t) * (UV_B * UV_B) + ij];
  if (anti) v = -v;
  const UvPair A = uv_pair(a, anti), B = uv_pair(b, anti), Cp = uv_pair(c, false);
  for (int i = 0; i < A.cnt; ++i)
    for (int j = 0; j < B.cnt; ++j) {
      const int p = A.p[i], qq = A.q[i], r = B.p[j], s = B.q[j];
      if constexpr (!THREE) {  // E_pq E_rs = Gamma_pqrs + d_qr gamma_ps
        if (qq == r) v -= A.sg[i] * B.sg[j] * g1[p * n + s];
      } else
      // E_pq E_rs E_tu = Gamma3 + d_qt Gamma_purs + d_st Gamma_pqru + d_qr (Gamma_pstu + d_st gamma_pu)
      for (int l = 0; l < Cp.cnt; ++l) {
        const int tt = Cp.p[l], u = Cp.q[l];
        double w = 0.0;
        if (qq == tt) w += g2[((p * n + u) * n + r) * n + s];
        if (s == tt) w += g2[((p * n + qq) * n + r) * n + u];
        if (qq == r) {
          w += g2[((p * n + s) * n + tt) * n + u];
          if (s == tt) w += g1[p * n + u];
        }
        v -= A.sg[i] * B.sg[j] * w;
      }
    }
  if (!THREE) {
    double *M = anti ? comp + (long long)q.U * q.U : comp;
    const int ld = anti ? q.V : q.U;
    M[(long long)a * ld + b] = v;
    M[(long long)b * ld + a] = v;
    return;
  }
  const long long U = q.U;
  if (anti) {
    double *M = comp + U * U * U;
    M[((long long)a * q.V + b) * U + c] = v;
    M[((long long)b * q.V + a) * U + c] = v;
  } else {
    comp[(a * U + b) * U + c] = v;
    comp[(a * U + c) * U + b] = v;
    comp[(b * U + a) * U + c] = v;
    comp[(b * U + c) * U + a] = v;
    comp[(c * U + a) * U + b] = v;
    comp[(c * U + b) * U + a] = v;
  }
}

// E_pq = w (S + sg A): index of the symmetric and antisymmetric pair, weight, sign.
struct UvExpand {
  int u, v;
  double w, sg;
};
__device__ __forceinline__ UvExpand uv_expand(int p, int q) {
  const int r = max(p, q), s = min(p, q);
  UvExpand e;
  e.u = r * (r + 1) / 2 + s;
  e.v = r == s ? 0 : r * (r - 1) / 2 + s;
  e.w = r == s ? 1.0 : 0.5;
  e.sg = r == s ? 0.0 : (p > q ? 1.0 : -1.0);
  return e;
}

// Gamma_pqrs = w w (Gamma(S,S) + sg sg Gamma(A,A))
__global__ void k_uv_expand2(const double *__restrict__ comp, UvShape q, double *__restrict__ g2) {
  const int n = q.n, i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n * n * n * n) return;
  const UvExpand a = uv_expand(i / (n * n * n), (i / (n * n)) % n), b = uv_expand((i / n) % n, i % n);
  double v = comp[a.u * q.U + b.u];
  const double sg = a.sg * b.sg;
  if (sg != 0.0) v += sg * comp[(long long)q.U * q.U + a.v * q.V + b.v];
  g2[i] = a.w * b.w * v;
}

// Gamma3_pqrstu = w w w (Gamma(S,S,S) + the three Gamma(A,A,S) with their signs)
__global__ void k_uv_expand3(const double *__restrict__ comp, UvShape q, double *__restrict__ g3) {
  const int n = q.n, n2 = n * n;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x, U = q.U, V = q.V;
  if (i >= (long long)n2 * n2 * n2) return;
  const int tu = (int)(i % n2), rs = (int)((i / n2) % n2), pq = (int)(i / ((long long)n2 * n2));
  const UvExpand a = uv_expand(pq / n, pq % n), b = uv_expand(rs / n, rs % n), c = uv_expand(tu / n, tu % n);
  const double *M = comp + U * U * U;
  double v = comp[(a.u * U + b.u) * U + c.u];
  const double ab = a.sg * b.sg, ac = a.sg * c.sg, bc = b.sg * c.sg;
  if (ab != 0.0) v += ab * M[(a.v * V + b.v) * U + c.u];
  if (ac != 0.0) v += ac * M[(a.v * V + c.v) * U + b.u];
  if (bc != 0.0) v += bc * M[(b.v * V + c.v) * U + a.u];
  g3[i] = a.w * b.w * c.w * v;
}

// Launch shape of k_uv_gram: threads per block, tiles per group, groups, and the number
// of slab splits that gives `waves` blocks per resident slot.
struct UvPlan {
  UvShape q;
  int threads, group, groups, maxtiles, nsplit, ny;
  size_t smem, part_bytes, comp_bytes;
};

template <bool THREE>
static int uv_plan(int n, long long ND, UvPlan &p) {
  p.q = uv_shape(n);
  p.maxtiles = uv_tiles(p.q, 0);
  p.groups = (p.maxtiles + UV_THREADS - 1) / UV_THREADS;
  p.group = (p.maxtiles + p.groups - 1) / p.groups;
  const int k = std::max(1, std::min(UV_KG, UV_THREADS / p.group));
  p.threads = std::min(UV_THREADS, (p.group * k + 31) / 32 * 32);
  p.ny = THREE ? p.q.U : 1;
  p.smem = sizeof(double) * (size_t)UV_KS * p.q.ld * (THREE ? 2 : 1);
  FORTE_CUDA_TRY(set_smem_optin_max((const void *)k_uv_gram<THREE>));
  int per_sm = 1, dev = 0, nsm = 1;
  FORTE_CUDA_TRY(cudaGetDevice(&dev));
  FORTE_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  FORTE_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_uv_gram<THREE>, p.threads, p.smem));
  // the 2-RDM's blocks are alike: one wave.  The third index makes those of the 3-RDM
  // uneven (tiles b >= c): about four waves, the largest first
  const long long slots = (long long)std::max(1, per_sm) * nsm * (THREE ? 4 : 1);
  const long long nslab = (ND + UV_KS - 1) / UV_KS;
  p.nsplit = (int)std::max(1LL, std::min({nslab, slots / ((long long)p.groups * p.ny), 65535LL}));
  p.part_bytes = sizeof(double) * (size_t)p.nsplit * p.ny * p.maxtiles * UV_B * UV_B;
  const size_t U = p.q.U, V = p.q.V;
  p.comp_bytes = sizeof(double) * (THREE ? U * U * U + V * V * U : U * U + V * V);
  return FORTE_OK;
}

// Adjoint of the state-averaged energy E_SA = sum_k w_k E_k (Sec. II.B):
// dh += c1 gamma^k, deri += c2 Gamma^k for one state (c1 = scale w_k, c2 = scale w_k / 2).
__global__ void k_sa_accum(const double *__restrict__ g1, const double *__restrict__ g2, int n, double c1,
                           double c2, double *__restrict__ dh, double *__restrict__ deri) {
  const int n2 = n * n, n4 = n2 * n2;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += gridDim.x * blockDim.x) {
    deri[i] += c2 * g2[i];
    if (i < n2) dh[i] += c1 * g1[i];
  }
}

int sa_gradient(forte_ctx *ctx, int nstates, const double *weights, const double *C, double scale, double *dh,
                double *deri) {
  const int n = ctx->n, n2 = n * n;
  int rc = ctx->sc_grad.ensure(sizeof(double) * ((size_t)n2 + (size_t)n2 * n2) + 256);
  if (rc) return rc;
  double *g1 = (double *)ctx->sc_grad.ptr, *g2 = g1 + n2;
  for (int k = 0; k < nstates; ++k) {
    const double *ck = C + (size_t)k * ctx->Ndet;
    if ((rc = rdm12_fp64(ctx, ck, ck, g1, g2))) return rc;
    const double c1 = scale * weights[k], c2 = 0.5 * scale * weights[k];
    {
      FORTE_PROF(ctx, "sa_accum");
      k_sa_accum<<<(unsigned)std::min(1024, (n2 * n2 + 255) / 256), 256, 0, ctx->stream>>>(g1, g2, n, c1, c2, dh,
                                                                                          deri);
      FORTE_LAUNCH_CHECK();
    }
  }
  return FORTE_OK;
}

int rdm12_fp64(forte_ctx *ctx, const double *bra, const double *ket, double *g1, double *g2, bool tensor_ok) {
  cudaStream_t st = ctx->stream;
  const int n = ctx->n, n2 = n * n;
  const long long NA = ctx->Na, NB = ctx->Nb, ND = ctx->Ndet;
  // workspace: transposes of bra/ket, g1 partials, g1 (when the caller passed none)
  size_t off_T = 0;
  size_t sz_T = sizeof(double) * ND * 2;
  size_t off_P = off_T + sz_T;
  size_t sz_P = sizeof(double) * (size_t)(NA + NB) * n2;
  size_t off_g1 = off_P + sz_P;
  size_t sz_g1 = sizeof(double) * n2;
  size_t base_bytes = off_g1 + sz_g1 + 256;
  // 2-RDM: partial Grams and components of the FP64 path; the reduced-precision modes
  // take the tensor-core Gram (rdm_oz.cu).  Both are for bra == ket.
  const bool same = (bra == ket);
  if (g2 && !same) { set_error("the 2-RDM needs one state"); return FORTE_ERR_ARG; }
  // Small spaces keep the FP64 Gram in every mode (one GB300, forte_rdms: 27 M products, 9
  // orbitals with 5 + 4 electrons, 161 us against 202 us; 163 M, 10 with 5 + 5, 485
  // against 361).
  const double uv_products = (double)ND * (n2 * (n2 + 1.0) / 4);
  const bool oz = tensor_ok && g2 && ctx->precision != FORTE_FP64 && rdm2_oz_supported(ctx) &&
                  !(uv_products <= 80e6 && small_route(ctx, true));
  UvPlan pl = {};
  int rc;
  if (g2 && !oz && (rc = uv_plan<false>(n, ND, pl))) return rc;
  size_t off_D = (base_bytes + 255) & ~(size_t)255;
  size_t off_G = off_D + ((pl.part_bytes + 255) & ~(size_t)255);
  size_t sz_G = pl.comp_bytes;
  rc = ctx->sc_rdm.ensure(off_G + sz_G + 256);
  if (rc) return rc;
  char *w = (char *)ctx->sc_rdm.ptr;
  double *Tb = (double *)(w + off_T), *Tk = Tb + ND;
  double *P = (double *)(w + off_P);
  double *g1w = g1 ? g1 : (double *)(w + off_g1);
  if (oz && !g1) {  // the Gram step reallocates sc_rdm: keep the 1-RDM elsewhere
    if (!ctx->d_g1tmp) FORTE_CUDA_TRY(dev_alloc(&ctx->d_g1tmp, sizeof(double) * n2));
    g1w = ctx->d_g1tmp;
  }

  // gamma: alpha rows, then beta rows on the transposed vectors
  {
    FORTE_PROF(ctx, "g1_part");
    k_g1_part<<<(unsigned)NA, 256, 0, st>>>(ctx->sd[0].list, ctx->sh[0].nk, bra, ket, NB, n, same, P);
  FORTE_LAUNCH_CHECK();
  }
  dim3 tb(32, 8), tg((unsigned)((NB + 31) / 32), (unsigned)((NA + 31) / 32));
  {
    FORTE_PROF(ctx, "transpose_r");
    k_transpose_r<double><<<tg, tb, 0, st>>>(ket, Tk, NA, NB);
  FORTE_LAUNCH_CHECK();
  }
  const double *TbraP = Tk;
  if (!same) {
    {
      FORTE_PROF(ctx, "transpose_r");
      k_transpose_r<double><<<tg, tb, 0, st>>>(bra, Tb, NA, NB);
    FORTE_LAUNCH_CHECK();
    }
    TbraP = Tb;
  }
  const int nkB = ctx->sh[ctx->same_strings ? 0 : 1].nk;
  {
    FORTE_PROF(ctx, "g1_part");
    k_g1_part<<<(unsigned)NB, 256, 0, st>>>(ctx->sd[1].list, nkB, TbraP, Tk, NA, n, same, P + NA * n2);
  FORTE_LAUNCH_CHECK();
  }
  {
    FORTE_PROF(ctx, "sum_cols2");
    k_sum_cols2<<<n2, 256, 0, st>>>(P, NA, P + NA * n2, NB, n, same, g1w);
  FORTE_LAUNCH_CHECK();
  }
  if (!g2) return FORTE_OK;
  if (oz) {
    if ((rc = rdm2_oz(ctx, ket, g1w, g2))) return rc;
    return mixed_status(ctx);  // bounded waits of the tensor-core kernel (synchronises the stream)
  }

  double *P2 = (double *)(w + off_D), *comp = (double *)(w + off_G);
  {
    FORTE_PROF(ctx, "gram");
    k_uv_gram<false><<<dim3((unsigned)pl.nsplit, 1, (unsigned)pl.groups), pl.threads, pl.smem, st>>>(
        ctx->sd[0].dense, ctx->sd[1].dense, pl.q, ket, nullptr, NB, ND, pl.group, pl.maxtiles, P2);
    FORTE_LAUNCH_CHECK();
  }
  {
    FORTE_PROF(ctx, "finish_g2");
    const int ne = pl.maxtiles * UV_B * UV_B;
    k_uv_comp<false><<<(ne + 63) / 64, 64, 0, st>>>(P2, pl.nsplit, pl.q, pl.maxtiles, g1w, nullptr,
                                                    comp);
    FORTE_LAUNCH_CHECK();
    k_uv_expand2<<<(n2 * n2 + 255) / 256, 256, 0, st>>>(comp, pl.q, g2);
    FORTE_LAUNCH_CHECK();
  }
  return FORTE_OK;
}

// Spin-free 3-RDM of one state (Sec. II.A.1, gamma_3 summed over spin), FP64: the
// components Gamma(S,S,S) and Gamma(A,A,S) from <S_a C | S_b F_c> and <A_a C | A_b F_c>,
// F_c = S_c C, with the FP64 1- and 2-RDMs in the lower-rank terms of the normal
// ordering; one launch covers every third index c.
int rdm3_fp64(forte_ctx *ctx, const double *C, double *g3) {
  cudaStream_t st = ctx->stream;
  const int n = ctx->n, n2 = n * n;
  const long long NB = ctx->Nb, ND = ctx->Ndet;
  UvPlan pl = {};
  int rc = uv_plan<true>(n, ND, pl);
  if (rc) return rc;
  auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
  const size_t off_g2 = up(sizeof(double) * n2);
  const size_t off_F = off_g2 + up(sizeof(double) * n2 * n2);
  const size_t off_P = off_F + up(sizeof(double) * (size_t)pl.q.U * ND);
  const size_t off_c = off_P + up(pl.part_bytes);
  if ((rc = ctx->sc_rdm3.ensure(off_c + pl.comp_bytes + 256))) return rc;
  char *w = (char *)ctx->sc_rdm3.ptr;
  double *g1 = (double *)w, *g2 = (double *)(w + off_g2), *F = (double *)(w + off_F), *P = (double *)(w + off_P),
         *comp = (double *)(w + off_c);
  if ((rc = rdm12_fp64(ctx, C, C, g1, g2, false))) return rc;
  const int *dA = ctx->sd[0].dense, *dB = ctx->sd[1].dense;
  {
    FORTE_PROF(ctx, "build_D");
    const dim3 g((unsigned)std::min<long long>((ND + 255) / 256, 152LL * 8), (unsigned)pl.q.U);
    k_uv_images<<<g, 256, 0, st>>>(dA, dB, n, C, NB, ND, F);
    FORTE_LAUNCH_CHECK();
  }
  {
    FORTE_PROF(ctx, "gram");
    k_uv_gram<true><<<dim3((unsigned)pl.nsplit, (unsigned)pl.ny, (unsigned)pl.groups), pl.threads, pl.smem, st>>>(
        dA, dB, pl.q, C, F, NB, ND, pl.group, pl.maxtiles, P);
    FORTE_LAUNCH_CHECK();
  }
  {
    FORTE_PROF(ctx, "finish_g3");
    const int ne = pl.maxtiles * UV_B * UV_B;
    k_uv_comp<true><<<dim3((unsigned)((ne + 63) / 64), (unsigned)pl.ny), 64, 0, st>>>(
        P, pl.nsplit, pl.q, pl.maxtiles, g1, g2, comp);
    FORTE_LAUNCH_CHECK();
    const long long n6 = (long long)n2 * n2 * n2;
    k_uv_expand3<<<(unsigned)((n6 + 255) / 256), 256, 0, st>>>(comp, pl.q, g3);
    FORTE_LAUNCH_CHECK();
  }
  return FORTE_OK;
}

}  // namespace forte
