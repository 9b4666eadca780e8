// Sigma over an arbitrary list of determinants (the selected-CI data path of
// Sec. II.A.2, adaptive CI): S[v][i] = sum_j <D_i|H|D_j> C[v][j], H of Eq. 1.
//
// Determinants are 64-bit words over 2n spin orbitals (n <= 32): alpha orbital p
// at bit p, beta orbital p at bit n + p, creation operators ordered by spin
// orbital index (alpha before beta).  The list is arbitrary (any order, any mix of
// (n_alpha, n_beta) sectors); the matrix elements follow the Slater-Condon rules,
// evaluated on the device from the spin-free integrals.
//
// Design (one GPU, lists of ~1e2 .. 1e6 determinants): a warp owns one determinant i and
// runs over the whole list.  Two steps, so that neither waits for the other's lanes:
//   screen   bit-sliced: plane b holds, 32 determinants to a word, the complement of
//            bit b.  For the occupied spin orbitals of D_i alone, a carry-save count of
//            these words tells for 32 pairs at once whether at most two electrons of
//            D_i are missing in D_j: about 1.75 logic instructions a lane per orbital
//            and 32 pairs, no population count (which runs at an eighth of their rate).
//   elements the pairs that pass go through a queue in shared memory, so that 32 lanes
//            evaluate 32 connected pairs; singles (a sum over the occupied orbitals) and
//            the diagonal have their own step, since one of them among 31 doubles
//            would hold up the warp.
// About 1.3 % of the pairs of a grown list are connected, so the old form (one thread a
// row, two population counts a pair, elements evaluated where they turned up) ran
// its elements with one or two lanes.
// One GB300, 50,001 determinants of 30 orbitals and 10 + 10 electrons: 20.4 -> 1.57 ms.
// The order of a row's sum follows from the list alone, so results repeat exactly.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "forte_internal.h"

struct forte_sci {
  int n = 0;
  int device = 0;
  cudaStream_t stream = nullptr;
  double *d_h = nullptr;    // [n][n]
  double *d_eri = nullptr;  // [n][n][n][n], chemist order
  forte::Scratch planes;    // bit planes [65][words]
};

namespace forte {
namespace {

constexpr int SCI_WARPS = 8;   // determinants (rows) per block
constexpr int SCI_NV = 4;      // vectors per launch
constexpr unsigned SCI_FULL = 0xffffffffu;

__device__ __forceinline__ int below(uint64_t d, int P) {  // occupied spin orbitals below P
  return __popcll(d & ((1ull << P) - 1ull));
}

struct SciInts {
  const double *h, *eri;
  int n;
  int inv;  // 65536 / n + 1: P / n = P inv / 65536 for P < 64
  __device__ __forceinline__ double g(int p, int q, int r, int s) const {
    return __ldg(eri + ((((long long)p * n + q) * n + r) * n + s));
  }
  __device__ __forceinline__ int spin(int P) const { return (P * inv) >> 16; }
  __device__ __forceinline__ int orb(int P) const { return P - spin(P) * n; }
};

// Elements <D_I|H|D_J> for words of one (n_alpha, n_beta) sector.  Spin orbital P:
// spatial P % n, spin P / n; <PQ||RS> = <PQ|RS> - <PQ|SR>, <PQ|RS> = (pr|qs) when
// spin(P) = spin(R) and spin(Q) = spin(S), else 0.

// One replacement: D_I = phase a+_M a_R D_J (M in I only, R in J only; 0 across spins).
__device__ double sc_single(const SciInts &H, uint64_t I, uint64_t J) {
  const uint64_t x = I ^ J;
  const int M = __ffsll((long long)(x & I)) - 1, R = __ffsll((long long)(x & J)) - 1;
  if (H.spin(M) != H.spin(R)) return 0.0;
  const int m = H.orb(M), r = H.orb(R);
  const uint64_t t = J & ~(1ull << R);
  double v = __ldg(H.h + m * H.n + r);
  for (uint64_t a = t; a; a &= a - 1) {  // K in J, K != R
    const int K = __ffsll((long long)a) - 1, k = H.orb(K);
    v += H.g(m, r, k, k);
    if (H.spin(K) == H.spin(M)) v -= H.g(m, k, k, r);
  }
  return ((below(J, R) + below(t, M)) & 1) ? -v : v;
}

// Two replacements: D_I = phase a+_M a+_O a_S a_R D_J with M < O in I only, R < S in J
// only: <MO||RS> times the phase of the operator string applied to D_J.
__device__ double sc_double(const SciInts &H, uint64_t I, uint64_t J) {
  const uint64_t x = I ^ J;
  uint64_t mi = x & I, rj = x & J;
  const int M = __ffsll((long long)mi) - 1, R = __ffsll((long long)rj) - 1;
  mi &= mi - 1;
  rj &= rj - 1;
  const int O = __ffsll((long long)mi) - 1, S = __ffsll((long long)rj) - 1;
  uint64_t t = J;
  int c = below(t, R);
  t &= ~(1ull << R);
  c += below(t, S);
  t &= ~(1ull << S);
  c += below(t, O);
  t |= 1ull << O;
  c += below(t, M);
  const int sM = H.spin(M), sO = H.spin(O), sR = H.spin(R), sS = H.spin(S);
  const int m = H.orb(M), o = H.orb(O), r = H.orb(R), s = H.orb(S);
  double v = 0.0;
  if (sM == sR && sO == sS) v += H.g(m, r, o, s);  // <MO|RS> = (mr|os)
  if (sM == sS && sO == sR) v -= H.g(m, s, o, r);  // <MO|SR> = (ms|or)
  return (c & 1) ? -v : v;
}

// planes[b][w]: bit k is set when spin orbital b is empty in determinant 32 w + k (and
// past the end of the list); plane 64 is zero.  W: words per plane, a multiple of 128
// (16-byte loads of a whole warp).
__global__ void k_sci_planes(long long nd, const uint64_t *__restrict__ dets, long long W,
                             uint32_t *__restrict__ planes) {
  const long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= W) return;
  const long long j = w * 32 + lane;
  const uint64_t D = j < nd ? dets[j] : 0ull;
  uint32_t lo = 0, hi = 0;  // lane b (and 32 + b) keeps plane b's word
  for (int b = 0; b < 64; ++b) {
    const uint32_t m = __ballot_sync(SCI_FULL, !((D >> b) & 1ull));
    if (lane == (b & 31)) {
      if (b < 32) lo = m; else hi = m;
    }
  }
  planes[lane * W + w] = lo;
  planes[(lane + 32) * W + w] = hi;
  if (lane == 0) planes[64 * W + w] = 0;
}

__device__ __forceinline__ void csa(uint32_t &s, uint32_t &c, uint32_t a, uint32_t b, uint32_t d) {
  s = a ^ b ^ d;
  c = (a & b) | (a & d) | (b & d);
}

// S[v0 + v][i] = sum_j <D_i|H|D_j> C[v0 + v][j], v < NV; one warp per i.
template <int NV>
__global__ void __launch_bounds__(32 * SCI_WARPS) k_sci_sigma(SciInts H, long long nd, const uint64_t *__restrict__ dets,
                                                              const uint32_t *__restrict__ planes, long long W,
                                                              const double *__restrict__ C, double *__restrict__ S) {
  __shared__ uint32_t s_q[SCI_WARPS][64], s_q1[SCI_WARPS][64];  // rings of pairs, of single replacements
  __shared__ __align__(4) uint8_t s_occ[SCI_WARPS][68];                     // occupied spin orbitals of the row
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long i = (long long)blockIdx.x * SCI_WARPS + wid;
  if (i >= nd) return;  // (whole warps; no block barrier below)
  uint32_t *q = s_q[wid], *q1 = s_q1[wid];
  uint8_t *occ = s_occ[wid];
  const uint64_t I = dets[i], amask = (1ull << H.n) - 1ull;
  const int na = __popcll(I & amask), no = __popcll(I);
  // occupied list, padded to a multiple of four with the zero plane
  for (int b = lane; b < 64; b += 32)
    if ((I >> b) & 1ull) occ[below(I, b)] = (uint8_t)b;
  if (lane < 4) occ[no + lane] = 64;
  __syncwarp();

  double acc[NV], dsum[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = dsum[v] = 0.0;
  bool hasd = false;
  unsigned head = 0, cnt = 0, head1 = 0, cnt1 = 0;

  auto singles = [&](unsigned m) {  // the first m queued single replacements
    if (lane < m) {
      const uint32_t j = q1[(head1 + lane) & 63];
      const double e = sc_single(H, I, dets[j]);
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] = fma(e, C[(long long)v * nd + j], acc[v]);
    }
    __syncwarp();
    head1 += m;
    cnt1 -= m;
  };
  auto pairs = [&](unsigned m) {  // the first m queued pairs
    bool one = false;
    uint32_t j = 0;
    if (lane < m) {
      j = q[(head + lane) & 63];
      if (j < nd) {
        const uint64_t J = dets[j];
        const int d = __popcll(I ^ J);
        const bool sector = __popcll(J & amask) == na && __popcll(J) == no;
        if (sector && d == 4) {
          const double e = sc_double(H, I, J);
#pragma unroll
          for (int v = 0; v < NV; ++v) acc[v] = fma(e, C[(long long)v * nd + j], acc[v]);
        }
        one = sector && d == 2;
        if (sector && d == 0) {
          hasd = true;
#pragma unroll
          for (int v = 0; v < NV; ++v) dsum[v] += C[(long long)v * nd + j];
        }
      }
    }
    const unsigned b1 = __ballot_sync(SCI_FULL, one);
    if (one) q1[(head1 + cnt1 + __popc(b1 & ((1u << lane) - 1u))) & 63] = j;
    __syncwarp();
    head += m;
    cnt -= m;
    cnt1 += __popc(b1);
    if (cnt1 >= 32) singles(32);
  };

  for (long long w0 = 0; w0 < W; w0 += 128) {
    const uint4 *P = reinterpret_cast<const uint4 *>(planes + w0) + lane;
    uint32_t ones[4] = {0, 0, 0, 0}, twos[4] = {0, 0, 0, 0}, fours[4] = {0, 0, 0, 0};
    for (int k = 0; k < no; k += 4) {
      const uint32_t o4 = *reinterpret_cast<const uint32_t *>(occ + k);
      uint4 x[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) x[t] = __ldg(P + ((o4 >> (8 * t)) & 255u) * (W / 4));
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const uint32_t a = e == 0 ? x[0].x : e == 1 ? x[0].y : e == 2 ? x[0].z : x[0].w;
        const uint32_t b = e == 0 ? x[1].x : e == 1 ? x[1].y : e == 2 ? x[1].z : x[1].w;
        const uint32_t c = e == 0 ? x[2].x : e == 1 ? x[2].y : e == 2 ? x[2].z : x[2].w;
        const uint32_t d = e == 0 ? x[3].x : e == 1 ? x[3].y : e == 2 ? x[3].z : x[3].w;
        uint32_t t1, t2, f;
        csa(ones[e], t1, ones[e], a, b);
        csa(ones[e], t2, ones[e], c, d);
        csa(twos[e], f, twos[e], t1, t2);
        fours[e] |= f;
      }
    }
    uint32_t m[4];  // at most two electrons missing
#pragma unroll
    for (int e = 0; e < 4; ++e) m[e] = ~(fours[e] | (ones[e] & twos[e]));
    const uint32_t j0 = (uint32_t)((w0 + 4 * lane) * 32);
    for (;;) {
      const int e = m[0] ? 0 : m[1] ? 1 : m[2] ? 2 : 3;
      const uint32_t cur = m[0] ? m[0] : m[1] ? m[1] : m[2] ? m[2] : m[3];
      const unsigned bal = __ballot_sync(SCI_FULL, cur != 0);
      if (!bal) break;
      if (cur) {
        q[(head + cnt + __popc(bal & ((1u << lane) - 1u))) & 63] = j0 + 32 * e + (uint32_t)(__ffs((int)cur) - 1);
        const uint32_t rest = cur & (cur - 1);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (k == e) m[k] = rest;
      }
      __syncwarp();
      cnt += __popc(bal);
      if (cnt >= 32) pairs(32);
    }
  }
  if (cnt) pairs(cnt);
  if (cnt1) singles(cnt1);
  if (__any_sync(SCI_FULL, hasd)) {
    // <D_I|H|D_I> = sum_P h_PP + sum_{Q<P} <PQ||PQ>: a lane takes every 32nd P
    double e = 0.0;
    for (int a = lane; a < no; a += 32) {
      const int P = occ[a], p = H.orb(P);
      e += __ldg(H.h + p * H.n + p);
      for (int b = 0; b < a; ++b) {
        const int Q = occ[b], qo = H.orb(Q);
        e += H.g(qo, qo, p, p);
        if (H.spin(P) == H.spin(Q)) e -= H.g(qo, p, p, qo);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(SCI_FULL, e, o);
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[v] = fma(e, dsum[v], acc[v]);
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc[v] += __shfl_xor_sync(SCI_FULL, acc[v], o);
    if (lane == 0) S[(long long)v * nd + i] = acc[v];
  }
}

}  // namespace
}  // namespace forte

using namespace forte;

extern "C" {

forte_sci *forte_sci_create(int norb, const double *h, const double *eri) {
  clear_error();
  if (norb < 1 || norb > 32) {
    set_error("forte_sci_create: norb must be in 1..32 (2 norb spin orbitals in a 64-bit word)");
    return nullptr;
  }
  if (!h || !eri) {
    set_error("forte_sci_create: NULL integrals");
    return nullptr;
  }
  const size_t n = (size_t)norb, n4 = n * n * n * n;
  for (size_t k = 0; k < n * n; ++k)
    if (!std::isfinite(h[k])) { set_error("forte_sci_create: h contains NaN/Inf"); return nullptr; }
  for (size_t k = 0; k < n4; ++k)
    if (!std::isfinite(eri[k])) { set_error("forte_sci_create: eri contains NaN/Inf"); return nullptr; }
  forte_sci *s = new forte_sci();
  s->n = norb;
  if (cudaGetDevice(&s->device) != cudaSuccess || dev_alloc(&s->d_h, sizeof(double) * n * n) != cudaSuccess ||
      dev_alloc(&s->d_eri, sizeof(double) * n4) != cudaSuccess ||
      cudaMemcpy(s->d_h, h, sizeof(double) * n * n, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(s->d_eri, eri, sizeof(double) * n4, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaStreamSynchronize(nullptr) != cudaSuccess) {  // (the handle's stream may not wait for the default one)
    set_error("forte_sci_create: device allocation or copy failed");
    cudaFree(s->d_h);
    cudaFree(s->d_eri);
    delete s;
    return nullptr;
  }
  return s;
}

void forte_sci_destroy(forte_sci *s) {
  if (!s) return;
  if (s->stream) cudaStreamSynchronize(s->stream);
  cudaFree(s->d_h);
  cudaFree(s->d_eri);
  s->planes.release();
  delete s;
}

int forte_sci_set_stream(forte_sci *s, void *cuda_stream) {
  if (!s) { set_error("NULL handle"); return FORTE_ERR_ARG; }
  s->stream = (cudaStream_t)cuda_stream;
  return FORTE_OK;
}

int forte_sci_sigma(forte_sci *s, long long ndet, const uint64_t *dets, const double *C, double *S, int nvec) {
  if (!s) { set_error("NULL handle"); return FORTE_ERR_ARG; }
  if (ndet < 0 || nvec < 0) { set_error("forte_sci_sigma: ndet and nvec must be >= 0"); return FORTE_ERR_ARG; }
  if (ndet == 0 || nvec == 0) return FORTE_OK;
  if (!dets || !C || !S) { set_error("forte_sci_sigma: NULL argument"); return FORTE_ERR_ARG; }
  if (ndet > (1LL << 31)) { set_error("forte_sci_sigma: at most 2^31 determinants"); return FORTE_ERR_ARG; }
  const long long W = (ndet + 4095) / 4096 * 128;  // words per plane
  int rc = s->planes.ensure(sizeof(uint32_t) * (size_t)W * 65);
  if (rc) return rc;
  uint32_t *planes = (uint32_t *)s->planes.ptr;
  k_sci_planes<<<(unsigned)((W + 7) / 8), 256, 0, s->stream>>>(ndet, dets, W, planes);
  FORTE_LAUNCH_CHECK();
  const SciInts H = {s->d_h, s->d_eri, s->n, 65536 / s->n + 1};
  const unsigned nb = (unsigned)((ndet + SCI_WARPS - 1) / SCI_WARPS);
  for (int v0 = 0; v0 < nvec; v0 += SCI_NV) {
    const double *Cv = C + (long long)v0 * ndet;
    double *Sv = S + (long long)v0 * ndet;
    switch (std::min(SCI_NV, nvec - v0)) {
      case 1: k_sci_sigma<1><<<nb, 32 * SCI_WARPS, 0, s->stream>>>(H, ndet, dets, planes, W, Cv, Sv); break;
      case 2: k_sci_sigma<2><<<nb, 32 * SCI_WARPS, 0, s->stream>>>(H, ndet, dets, planes, W, Cv, Sv); break;
      case 3: k_sci_sigma<3><<<nb, 32 * SCI_WARPS, 0, s->stream>>>(H, ndet, dets, planes, W, Cv, Sv); break;
      default: k_sci_sigma<4><<<nb, 32 * SCI_WARPS, 0, s->stream>>>(H, ndet, dets, planes, W, Cv, Sv); break;
    }
    FORTE_LAUNCH_CHECK();
  }
  return FORTE_OK;
}

}  // extern "C"
