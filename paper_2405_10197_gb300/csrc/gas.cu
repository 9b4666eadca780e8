// Occupation-restricted CI (GAS / RAS), Sec. II.A.1: the active orbitals are
// split into consecutive spaces A_1 .. A_G and a determinant |Ia>|Ib> is kept
// when gmin[g] <= n_alpha(A_g) + n_beta(A_g) <= gmax[g] for every g.  The
// restriction is applied, as in the paper, at the level of the strings (each
// string's per-space occupation is its class) and of the allowed combinations
// of string classes (a small table ok[class_a][class_b]).
//
// The restricted Hamiltonian is P H P.  Vectors keep the [N_alpha][N_beta]
// layout of the full space, zero outside the kept determinants, and the diagonal
// is +inf there, so that guesses and preconditioned corrections stay inside the
// restricted space.  When at most a quarter of the determinants is kept, sigma is
// formed over the kept determinants only (k_gas_sigma: each output from its
// same-spin Hamiltonian rows and its alpha-beta replacement pairs, skipping the
// source determinants of excluded class pairs), so its cost follows the kept
// space; otherwise the full-grid kernels run and a pass zeroes the excluded
// entries (write-only: it reads the class table and stores a zero where a
// determinant is excluded).
#include <algorithm>
#include <map>
#include <vector>

#include "forte_internal.h"

namespace forte {

// x[row][ib] = value wherever ok[clsA[ia]][clsB[ib]] == 0, rows = nvec * NA
// (ia = row % NA).  One block per row in a grid-stride loop, threads along ib.
template <typename T>
__global__ void k_gas_fill(T *__restrict__ x, long long rows, long long NA, long long NB,
                           const int *__restrict__ clsA, const int *__restrict__ clsB,
                           const uint8_t *__restrict__ ok, int ncB, T value) {
  for (long long row = blockIdx.x; row < rows; row += gridDim.x) {
    const uint8_t *okr = ok + (long long)clsA[row % NA] * ncB;
    T *xr = x + row * NB;
    for (long long ib = threadIdx.x; ib < NB; ib += blockDim.x)
      if (!okr[clsB[ib]]) xr[ib] = value;
  }
}

// x[v][i] = value wherever mask[i] == 0 (an arbitrary determinant mask).
template <typename T>
__global__ void k_det_fill(T *__restrict__ x, long long total, long long nd, const uint8_t *__restrict__ mask,
                           T value) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x)
    if (!mask[i % nd]) x[i] = value;
}

// ---- the restricted sigma over the kept determinants ----------------------------
//
// All strings of one class (per-space occupations) have the same number of single
// replacements into every class, and the same number of same-spin Hamiltonian entries
// from every class.  With each string's lists ordered by target class, the entries that
// a restriction allows are therefore the same positions for every string of a class:
// one short position list per block and class compacts the work, and every lane of a warp
// has an allowed product to form.
//   gas_off   [N_beta][no]: moving replacements of a beta string, by target class
//   gas_tcls  [class][no]: target class of each position
//   gas_ellc / gas_ellv (and FP32 values): H_bb rows by column class, entry-major within a
//             class (base nnz coff[class], then [nnz][strings of the class])
//   gas_ccls  [class][nnz]: column class of each position
// Built on the device, from rows of nnz entries each; one thread per beta string (in class
// order).
constexpr int GAS_MAXCLS = 64;

__global__ void k_gas_order(const uint32_t *__restrict__ off, int no, const int *__restrict__ ptr,
                            const int *__restrict__ col, const double *__restrict__ val, int nnz,
                            const int *__restrict__ cls, int nc, const int *__restrict__ coff,
                            const int *__restrict__ cstr, int N, uint32_t *__restrict__ goff,
                            uint8_t *__restrict__ tcls, int *__restrict__ ellc, double *__restrict__ ellv,
                            float *__restrict__ ellv32, uint8_t *__restrict__ ccls) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const int J = cstr[i], b = cls[J], i0 = coff[b], nb = coff[b + 1] - i0, ii = i - i0;
  int at[GAS_MAXCLS + 1];
  auto starts = [&](auto target, int cnt) {  // counting sort: at[c] = first position of class c
    for (int c = 0; c <= nc; ++c) at[c] = 0;
    for (int e = 0; e < cnt; ++e) ++at[target(e) + 1];
    for (int c = 0; c < nc; ++c) at[c + 1] += at[c];
  };
  auto ot = [&](int e) { return cls[off[(long long)J * no + e] & 0xFFFFu]; };
  starts(ot, no);
  for (int e = 0; e < no; ++e) {
    const int c = ot(e), p = at[c]++;
    goff[(long long)J * no + p] = off[(long long)J * no + e];
    if (ii == 0) tcls[b * no + p] = (uint8_t)c;
  }
  auto ct = [&](int e) { return cls[col[ptr[J] + e]]; };
  starts(ct, nnz);
  for (int e = 0; e < nnz; ++e) {
    const int c = ct(e), p = at[c]++;
    const long long w = (long long)nnz * i0 + (long long)p * nb + ii;
    ellc[w] = col[ptr[J] + e];
    ellv[w] = val[ptr[J] + e];
    ellv32[w] = (float)val[ptr[J] + e];
    if (ii == 0) ccls[b * nnz + p] = (uint8_t)c;
  }
}
// Every string of a class has its class's position lists (the counting argument above).
__global__ void k_gas_check(const uint32_t *__restrict__ goff, int no, const uint8_t *__restrict__ tcls,
                            const int *__restrict__ ellc, int nnz, const uint8_t *__restrict__ ccls,
                            const int *__restrict__ cls, const int *__restrict__ coff, const int *__restrict__ cstr, int N,
                            int *__restrict__ flag) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const int J = cstr[i], b = cls[J], i0 = coff[b], nb = coff[b + 1] - i0, ii = i - i0;
  bool bad = false;
  for (int p = 0; p < no; ++p) bad |= cls[goff[(long long)J * no + p] & 0xFFFFu] != tcls[b * no + p];
  for (int p = 0; p < nnz; ++p) bad |= cls[ellc[(long long)nnz * i0 + (long long)p * nb + ii]] != ccls[b * nnz + p];
  if (bad) *flag = 1;
}

constexpr int GAS_THREADS = 256;

// list = the p < cnt with ok(p), ascending, compacted by warp `w` of the block; the count
// goes to *n.  The caller synchronises before the list is read.
template <typename F>
__device__ __forceinline__ void gas_compact(int w, int cnt, F ok, uint16_t *list, int *n) {
  if ((int)(threadIdx.x >> 5) != w) return;
  const int lane = threadIdx.x & 31;
  int m = 0;
  for (int p0 = 0; p0 < cnt; p0 += 128) {  // four tests at a time: their loads overlap
    bool k[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) k[u] = p0 + 32 * u + lane < cnt && ok(p0 + 32 * u + lane);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const unsigned bal = __ballot_sync(0xffffffffu, k[u]);
      if (k[u]) list[m + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)(p0 + 32 * u + lane);
      m += __popc(bal);
    }
  }
  if (lane == 0) *n = m;
}

// P H P C for the kept determinants of the kept alpha row Ia = rows[blockIdx.x]
// (vector blockIdx.y), every other entry of S left as it is (zero).
//  (1) alpha-beta, driven by the source beta strings, class by class: tiles of TJ strings Jb
//      of class cb are gathered as D[k][j] = C[J_k][Jb_j] for the rows J_k that carry
//      weight there (k in L(Ia) with an allowed (class(J_k), cb) pair; k = 0 stands for
//      all replacements that move no electron, as in k_ab_fp64), and every replacement
//      E_rs Jb = s I_b with an allowed output adds s sum_k s_k (pq_k|rs) D[k][j] to the row
//      accumulator (shared memory); the unmoved replacements of Jb go to Jb itself
//      with the integral sums W;
//  (2) per kept output: the accumulator plus the same-spin terms
//      sum_Ja H_aa[Ia][Ja] C[Ja][Ib] + sum_Jb H_bb[Ib][Jb] C[Ia][Jb] over allowed sources.
// The FP64 pipe bounds it.  One GB300, CAS(14,14) with at most 2 holes in orbitals 0-3
// and 2 particles in 10-13 (369,712 of 11.8 M determinants): 4.73 -> 2.75 ms (before, a lane
// whose replacement was not allowed idled, and the same-spin sums ran over all entries).
// Small spaces wait on memory latency, many classes holding a few strings each; there the
// lanes of a warp share an output: 5 + 6 electrons in 12 orbitals, 1 hole in 0-3, 2 particles
// in 9-11: 167 us before the class lists, 285 us with a thread per output, 137 us so.
// T: FP64, or FP32 for the FP32 vectors of the reduced-precision phase.
template <typename T>
__global__ void __launch_bounds__(GAS_THREADS) k_gas_sigma(
    const T *__restrict__ C, T *__restrict__ S, long long NB, long long vstride, const uint32_t *__restrict__ strA,
    const uint32_t *__restrict__ offA, int noA, const int *__restrict__ ptrA, const int *__restrict__ colA,
    const T *__restrict__ valA, int maxnnzA, const uint32_t *__restrict__ goffB, int noB,
    const uint8_t *__restrict__ tcls, const int *__restrict__ ellc, const T *__restrict__ ellv, int nnzB,
    const uint8_t *__restrict__ ccls, const T *__restrict__ gpair, const double *__restrict__ W, int npair,
    const int *__restrict__ clsA, const unsigned long long *__restrict__ okm, int ncB, const int *__restrict__ rows,
    const int *__restrict__ coff, const int *__restrict__ cstr, int TJ) {
  extern __shared__ __align__(16) uint8_t gsm[];
  const int Ia = rows[blockIdx.x], nk = noA + 1;
  const int rb = ptrA[Ia], nnz = ptrA[Ia + 1] - rb;
  T *G = (T *)gsm;                                // [nk][npair] signed integral rows
  T *srow = G + (size_t)nk * npair;               // [NB] alpha-beta accumulator
  T *D = srow + NB;                               // [nk][TJ] gathered C rows
  T *sval = D + (size_t)nk * TJ;                  // [maxnnzA] CSR row Ia of H_aa
  int *scol = (int *)(sval + maxnnzA);            // [maxnnzA]
  int *sJ = scol + maxnnzA;                       // [nk] rows of C
  int *sj = sJ + nk;                              // [TJ] strings of the tile
  // class masks (bit b: beta class b is allowed) of the rows that k and the H_aa entries read
  unsigned long long *kmask = (unsigned long long *)(((uintptr_t)(sj + TJ) + 7) & ~(uintptr_t)7);  // [nk]
  unsigned long long *emask = kmask + nk;         // [maxnnzA]
  uint16_t *klist = (uint16_t *)(emask + maxnnzA);  // [nk]: allowed k
  uint16_t *plist = klist + nk;                   // [max(noB, 1)]: allowed positions of the sources' lists
  uint16_t *elist = plist + noB + 1;              // [maxnnzA]: allowed entries of H_aa[Ia]
  uint16_t *flist = elist + maxnnzA;              // [nnzB]: allowed positions of H_bb rows
  __shared__ int s_pp[16], s_n[2];
  const uint32_t *la = offA + (long long)Ia * noA;
  const uint32_t occ = strA[Ia];
  const int npp = __popc(occ);
  const unsigned long long okA = okm[clsA[Ia]];
  if (threadIdx.x < 32 && ((occ >> threadIdx.x) & 1u))
    s_pp[__popc(occ & ((1u << threadIdx.x) - 1u))] = threadIdx.x * (threadIdx.x + 3) / 2;  // pair (r, r)
  for (int e = threadIdx.x; e < nk; e += GAS_THREADS) {
    sJ[e] = e ? (int)(la[e - 1] & 0xFFFFu) : Ia;
    kmask[e] = okm[clsA[sJ[e]]];
  }
  for (int i = threadIdx.x; i < noA * npair; i += GAS_THREADS) {
    const uint32_t w = la[i / npair];
    const T g = gpair[(size_t)((w >> 16) & 0xFFu) * npair + i % npair];
    G[npair + i] = (w >> 31) ? -g : g;
  }
  for (long long i = threadIdx.x; i < NB; i += GAS_THREADS) srow[i] = T(0);
  for (int i = threadIdx.x; i < nnz; i += GAS_THREADS) {
    sval[i] = valA[rb + i];
    scol[i] = colA[rb + i];
    emask[i] = okm[clsA[scol[i]]];
  }
  __syncthreads();
  for (int rs = threadIdx.x; rs < npair; rs += GAS_THREADS) {
    T v = T(0);
    for (int m = 0; m < npp; ++m) v += gpair[(size_t)s_pp[m] * npair + rs];
    G[rs] = v;
  }
  const T *Cv = C + (long long)blockIdx.y * vstride;
  T *Sv = S + (long long)blockIdx.y * vstride + (long long)Ia * NB;
  for (int cb = 0; cb < ncB; ++cb) {
    if (coff[cb] == coff[cb + 1]) continue;
    __syncthreads();
    gas_compact(0, nk, [&](int e) { return (kmask[e] >> cb) & 1ull; }, klist, &s_n[0]);
    gas_compact(1, noB, [&](int p) { return (okA >> tcls[cb * noB + p]) & 1ull; }, plist, &s_n[1]);
    __syncthreads();
    const int kc = s_n[0], pc = s_n[1];
    const bool self = (okA >> cb) & 1ull;
    if (kc == 0 || (pc == 0 && !self)) continue;
    for (int s0 = coff[cb]; s0 < coff[cb + 1]; s0 += TJ) {
      const int tj = min(TJ, coff[cb + 1] - s0);
      __syncthreads();
      for (int i = threadIdx.x; i < kc * tj; i += GAS_THREADS) {
        const int kk = i / tj, j = i - kk * tj;
        D[kk * TJ + j] = Cv[(long long)sJ[klist[kk]] * NB + cstr[s0 + j]];
      }
      for (int j = threadIdx.x; j < tj; j += GAS_THREADS) sj[j] = cstr[s0 + j];
      __syncthreads();
      for (int w = threadIdx.x; w < tj * pc; w += GAS_THREADS) {
        const int j = w / pc;
        const uint32_t f = goffB[(long long)sj[j] * noB + plist[w - j * pc]];
        const T *g = G + ((f >> 16) & 0xFFu), *d = D + j;
        T acc = T(0);
#pragma unroll 4
        for (int kk = 0; kk < kc; ++kk) acc += g[klist[kk] * npair] * d[kk * TJ];
        atomicAdd(&srow[f & 0xFFFFu], (f >> 31) ? -acc : acc);
      }
      if (self) {
        // the unmoved replacements of Jb: npp integral sums with row Ia itself (k = 0) and one
        // with each other row, split over up to 16 threads a string
        const int parts = min(16, GAS_THREADS / tj), part = threadIdx.x / tj, j = threadIdx.x - part * tj;
        const int z = klist[0] == 0 ? npp : 0, lead = z ? 1 : 0;
        if (part < parts) {
          T acc = T(0);
#pragma unroll 2
          for (int u = part; u < z + kc - lead; u += parts) {
            if (u < z) {
              acc += (T)W[(size_t)s_pp[u] * NB + sj[j]] * D[j];
            } else {
              const int kk = u - z + lead;
              const uint32_t w = la[klist[kk] - 1];
              const T x = (T)W[(size_t)((w >> 16) & 0xFFu) * NB + sj[j]];
              acc += ((w >> 31) ? -x : x) * D[kk * TJ + j];
            }
          }
          atomicAdd(&srow[sj[j]], acc);
        }
      }
    }
  }
  for (int b = 0; b < ncB; ++b) {
    const int i0 = coff[b], nb = coff[b + 1] - i0;
    if (!((okA >> b) & 1ull) || nb == 0) continue;
    __syncthreads();
    gas_compact(0, nnz, [&](int e) { return (emask[e] >> b) & 1ull; }, elist, &s_n[0]);
    gas_compact(1, nnzB, [&](int p) { return (okA >> ccls[b * nnzB + p]) & 1ull; }, flist, &s_n[1]);
    __syncthreads();
    const int ne = s_n[0], nf = s_n[1];
    // small classes: up to 32 neighbouring lanes share an output's terms
    int parts = 1;
    while (parts < 32 && 2 * parts * nb <= GAS_THREADS) parts *= 2;
    const int q = threadIdx.x % parts;
    for (int i1 = 0; i1 < nb; i1 += GAS_THREADS / parts) {
      const int i = i1 + threadIdx.x / parts, Ib = i < nb ? cstr[i0 + i] : 0;
      T acc = T(0), acc2 = T(0);
      if (i < nb) {
#pragma unroll 4
        for (int e = q; e < ne; e += parts) acc += sval[elist[e]] * Cv[(long long)scol[elist[e]] * NB + Ib];
        const int *ec = ellc + (long long)nnzB * i0 + i;
        const T *ev = ellv + (long long)nnzB * i0 + i;
#pragma unroll 4
        for (int f = q; f < nf; f += parts) {
          const long long p = (long long)flist[f] * nb;
          acc2 += ev[p] * Cv[(long long)Ia * NB + ec[p]];
        }
      }
      acc += acc2;
      for (int o = parts >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (i < nb && q == 0) Sv[Ib] = srow[Ib] + acc;
    }
  }
}

static size_t gas_smem_bytes(size_t tsz, int nk, int noB, int npair, long long NB, int maxnnz, int nnzB, int TJ) {
  return tsz * ((size_t)nk * npair + NB + (size_t)nk * TJ + maxnnz) + sizeof(int) * ((size_t)maxnnz + nk + TJ) +
         8 * ((size_t)nk + maxnnz) + sizeof(uint16_t) * ((size_t)nk + noB + 1 + maxnnz + nnzB) + 24;
}

bool gas_sparse(const forte_ctx *ctx) {
  if (!ctx->gas_on || ctx->detmask_on || !ctx->d_gas_rows || !ctx->d_gas_off || ctx->gas_route == 0) return false;
  return ctx->gas_route == 1 || 4 * ctx->gas_ndet <= ctx->Ndet;
}

template <typename T>
static int gas_sigma_t(forte_ctx *ctx, const T *C, T *S, int nvec) {
  if (nvec <= 0) return FORTE_OK;
  cudaStream_t st = ctx->stream;
  FORTE_CUDA_TRY(cudaMemsetAsync(S, 0, sizeof(T) * ctx->Ndet * nvec, st));
  if (ctx->gas_nrows == 0) return FORTE_OK;
  const int n = ctx->n, noA = ctx->na * (n - ctx->na), noB = ctx->nb * (n - ctx->nb);
  const int np = ctx->npair, ncB = ctx->gas_nc[1], nnzB = ctx->sh[1].csr_ptr[1];
  // the widest source tile that keeps two blocks per SM, else one
  auto bytes = [&](int TJ) {
    return gas_smem_bytes(sizeof(T), noA + 1, noB, np, ctx->Nb, ctx->gas_maxnnz, nnzB, TJ);
  };
  int TJ = 64;
  while (TJ > 16 && bytes(TJ) > 113 * 1024) TJ /= 2;
  while (TJ > 8 && bytes(TJ) > 220 * 1024) TJ /= 2;
  const size_t smem = bytes(TJ);
  if (smem > 220 * 1024) {
    set_error("restricted sigma needs %zu bytes of shared memory", smem);
    return FORTE_ERR_ARG;
  }
  FORTE_CUDA_TRY(set_smem_optin_max((const void *)k_gas_sigma<T>));
  const bool f32 = sizeof(T) == 4;
  const T *valA = f32 ? (const T *)(const void *)ctx->sd[0].csr_val32 : (const T *)(const void *)ctx->sd[0].csr_val;
  const T *ellv = f32 ? (const T *)(const void *)ctx->d_gas_ellv32 : (const T *)(const void *)ctx->d_gas_ellv;
  const T *gp = f32 ? (const T *)(const void *)ctx->d_gpair32 : (const T *)(const void *)ctx->d_gpair;
  dim3 grid((unsigned)ctx->gas_nrows, (unsigned)nvec);
  FORTE_PROF(ctx, f32 ? "gas_sigma_f32" : "gas_sigma");
  k_gas_sigma<T><<<grid, GAS_THREADS, smem, st>>>(
      C, S, ctx->Nb, ctx->Ndet, ctx->sd[0].str, ctx->sd[0].off, noA, ctx->sd[0].csr_ptr, ctx->sd[0].csr_col, valA,
      ctx->gas_maxnnz, ctx->d_gas_off, noB, ctx->d_gas_tcls, ctx->d_gas_ellc, ellv, nnzB, ctx->d_gas_ccls, gp, ctx->d_W,
      np, ctx->d_gas_cls[0], ctx->d_gas_okm, ncB, ctx->d_gas_rows, ctx->d_gas_coff, ctx->d_gas_cstr, TJ);
  FORTE_LAUNCH_CHECK();
  return FORTE_OK;
}
int gas_sigma(forte_ctx *ctx, const double *C, double *S, int nvec) { return gas_sigma_t(ctx, C, S, nvec); }
int gas_sigma(forte_ctx *ctx, const float *C, float *S, int nvec) { return gas_sigma_t(ctx, C, S, nvec); }

template <typename T>
static int gas_fill(forte_ctx *ctx, T *x, int nvec, T value) {
  if (nvec <= 0) return FORTE_OK;
  if (ctx->detmask_on) {
    const long long total = (long long)nvec * ctx->Ndet;
    const unsigned nb = (unsigned)std::min<long long>((total + 255) / 256, 152LL * 16);
    FORTE_PROF(ctx, "det_mask");
    k_det_fill<T><<<nb, 256, 0, ctx->stream>>>(x, total, ctx->Ndet, ctx->d_detmask, value);
    FORTE_LAUNCH_CHECK();
  }
  if (!ctx->gas_on) return FORTE_OK;
  const long long rows = (long long)nvec * ctx->Na;
  const unsigned nb = (unsigned)std::min<long long>(rows, 152LL * 16);
  const int nt = ctx->Nb >= 256 ? 256 : (ctx->Nb >= 64 ? 64 : 32);
  FORTE_PROF(ctx, "gas_mask");
  k_gas_fill<T><<<nb, nt, 0, ctx->stream>>>(x, rows, ctx->Na, ctx->Nb, ctx->d_gas_cls[0], ctx->d_gas_cls[1],
                                            ctx->d_gas_ok, ctx->gas_nc[1], value);
  FORTE_LAUNCH_CHECK();
  return FORTE_OK;
}

int gas_mask(forte_ctx *ctx, double *x, int nvec) { return gas_fill<double>(ctx, x, nvec, 0.0); }
int gas_mask(forte_ctx *ctx, float *x, int nvec) { return gas_fill<float>(ctx, x, nvec, 0.0f); }

int det_mask_fill(forte_ctx *ctx, double *x, int nvec, double value) { return gas_fill<double>(ctx, x, nvec, value); }

long long space_dim(const forte_ctx *ctx) {
  if (ctx->detmask_on) {  // (no occupation restriction besides it; the mask is mirror-closed with a sector)
    if (ctx->spin_parity == 0) return ctx->detmask_n;
    const long long D = ctx->detmask_ndiag;
    return (ctx->detmask_n - D) / 2 + (ctx->spin_parity > 0 ? D : 0);
  }
  const long long K = ctx->gas_on ? ctx->gas_ndet : ctx->Ndet;
  if (ctx->spin_parity == 0) return K;
  // the kept set is symmetric under I_alpha <-> I_beta: mirror pairs plus the diagonal
  const long long D = ctx->gas_on ? ctx->gas_ndiag : ctx->Na;
  return (K - D) / 2 + (ctx->spin_parity > 0 ? D : 0);
}

// The lists of the kept-determinant kernel; without them sigma runs on the full grid.
static void gas_lists_release(forte_ctx *ctx) {
  auto drop = [](auto *&p) {
    cudaFree(p);
    p = nullptr;
  };
  drop(ctx->d_gas_coff);
  drop(ctx->d_gas_cstr);
  drop(ctx->d_gas_off);
  drop(ctx->d_gas_okm);
  drop(ctx->d_gas_tcls);
  drop(ctx->d_gas_ellc);
  drop(ctx->d_gas_ellv);
  drop(ctx->d_gas_ellv32);
  drop(ctx->d_gas_ccls);
}

static void gas_release(forte_ctx *ctx) {
  for (int s = 0; s < 2; ++s) {
    cudaFree(ctx->d_gas_cls[s]);
    ctx->d_gas_cls[s] = nullptr;
    ctx->gas_nc[s] = 0;
  }
  cudaFree(ctx->d_gas_ok);
  ctx->d_gas_ok = nullptr;
  cudaFree(ctx->d_gas_rows);
  ctx->d_gas_rows = nullptr;
  gas_lists_release(ctx);
  ctx->gas_nrows = 0;
  for (int t = 0; t < 2; ++t) ctx->gas_pick[t] = ctx->gas_pick_mode[t] = -1;
  ctx->gas_on = false;
  ctx->gas_ndet = 0;
  ctx->gas_ndiag = 0;
}

void gas_free(forte_ctx *ctx) { gas_release(ctx); }

// Beta strings by class (ascending), and their lists by target class.  Where the memory
// for them (16 bytes an entry of H_bb, 175 MB at 16 orbitals) cannot be had, there are no
// lists.
static int gas_lists(forte_ctx *ctx, const std::vector<int> &cls, const std::vector<long long> &cnt,
                     const std::vector<uint8_t> &ok, int ncA) {
  const SpinHost &B = ctx->sh[1];
  const int n = ctx->n, ncB = (int)cnt.size();
  if (!rows_alike(B.csr_ptr)) {  // before any kernel takes nnz entries from a row
    set_error("internal: string Hamiltonian rows of different lengths");
    return FORTE_ERR_ARG;
  }
  std::vector<int> coff(ncB + 1, 0), cstr(B.N);
  for (int b = 0; b < ncB; ++b) coff[b + 1] = coff[b] + (int)cnt[b];
  {
    std::vector<int> at(coff.begin(), coff.end() - 1);
    for (long long j = 0; j < B.N; ++j) cstr[at[cls[j]]++] = (int)j;
  }
  const int noB = ctx->nb * (n - ctx->nb), nnz = B.csr_ptr[1];
  const size_t ell = (size_t)nnz * B.N;
  std::vector<unsigned long long> okm(ncA, 0ull);
  for (int a = 0; a < ncA; ++a)
    for (int b = 0; b < ncB; ++b)
      if (ok[(size_t)a * ncB + b]) okm[a] |= 1ull << b;
  DevTemp tmp;
  int flag = 0;
  if (dev_alloc(&ctx->d_gas_coff, sizeof(int) * coff.size()) != cudaSuccess ||
      dev_alloc(&ctx->d_gas_cstr, sizeof(int) * cstr.size()) != cudaSuccess ||
      dev_alloc(&ctx->d_gas_okm, sizeof(okm[0]) * okm.size()) != cudaSuccess ||
      dev_alloc(&ctx->d_gas_off, sizeof(uint32_t) * std::max<size_t>(1, (size_t)B.N * noB)) != cudaSuccess ||
      dev_alloc(&ctx->d_gas_tcls, (size_t)ncB * noB + 1) != cudaSuccess ||
      dev_alloc(&ctx->d_gas_ellc, sizeof(int) * ell) != cudaSuccess ||
      dev_alloc(&ctx->d_gas_ellv, sizeof(double) * ell) != cudaSuccess ||
      dev_alloc(&ctx->d_gas_ellv32, sizeof(float) * ell) != cudaSuccess ||
      dev_alloc(&ctx->d_gas_ccls, (size_t)ncB * nnz) != cudaSuccess || dev_alloc(&tmp.ptr, sizeof(int)) != cudaSuccess) {
    gas_lists_release(ctx);
    return FORTE_OK;
  }
  FORTE_CUDA_TRY(copy_in(ctx, ctx->d_gas_coff, coff.data(), sizeof(int) * coff.size()));
  FORTE_CUDA_TRY(copy_in(ctx, ctx->d_gas_cstr, cstr.data(), sizeof(int) * cstr.size()));
  FORTE_CUDA_TRY(copy_in(ctx, ctx->d_gas_okm, okm.data(), sizeof(okm[0]) * okm.size()));
  int *d_flag = (int *)tmp.ptr;
  FORTE_CUDA_TRY(copy_in(ctx, d_flag, &flag, sizeof(int)));
  const unsigned nbk = (unsigned)((B.N + 63) / 64);
  k_gas_order<<<nbk, 64, 0, ctx->stream>>>(ctx->sd[1].off, noB, ctx->sd[1].csr_ptr, ctx->sd[1].csr_col,
                                           ctx->sd[1].csr_val, nnz, ctx->d_gas_cls[1], ncB, ctx->d_gas_coff,
                                           ctx->d_gas_cstr, (int)B.N, ctx->d_gas_off, ctx->d_gas_tcls, ctx->d_gas_ellc,
                                           ctx->d_gas_ellv, ctx->d_gas_ellv32, ctx->d_gas_ccls);
  FORTE_LAUNCH_CHECK();
  k_gas_check<<<nbk, 64, 0, ctx->stream>>>(ctx->d_gas_off, noB, ctx->d_gas_tcls, ctx->d_gas_ellc, nnz, ctx->d_gas_ccls,
                                           ctx->d_gas_cls[1], ctx->d_gas_coff, ctx->d_gas_cstr, (int)B.N, d_flag);
  FORTE_LAUNCH_CHECK();
  FORTE_CUDA_TRY(cudaMemcpyAsync(&flag, d_flag, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
  FORTE_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
  if (flag) {
    set_error("internal: strings of one class differ in their replacements");
    return FORTE_ERR_ARG;
  }
  return FORTE_OK;
}

int gas_set(forte_ctx *ctx, int nspace, const int *size, const int *gmin, const int *gmax, long long *ndet_out) {
  const int n = ctx->n;
  if (nspace < 0 || nspace > n) { set_error("nspace must be in [0, norb]"); return FORTE_ERR_ARG; }
  if (nspace > 0 && (!size || !gmin || !gmax)) { set_error("NULL space arrays"); return FORTE_ERR_ARG; }
  int tot = 0;
  for (int g = 0; g < nspace; ++g) {
    if (size[g] < 1) { set_error("space %d is empty", g); return FORTE_ERR_ARG; }
    if (gmin[g] < 0 || gmax[g] < gmin[g]) { set_error("space %d: need 0 <= gmin <= gmax", g); return FORTE_ERR_ARG; }
    tot += size[g];
  }
  if (nspace > 0 && tot != n) { set_error("space sizes add up to %d, not norb = %d", tot, n); return FORTE_ERR_ARG; }

  // classes of the strings of each spin: their per-space occupation vectors
  std::vector<int> cls[2];
  std::vector<std::vector<int>> occ[2];
  std::vector<long long> cnt[2];
  for (int s = 0; s < 2 && nspace > 0; ++s) {
    const SpinHost &H = ctx->sh[s];
    std::map<std::vector<int>, int> id;
    cls[s].resize(H.N);
    for (long long i = 0; i < H.N; ++i) {
      std::vector<int> o(nspace, 0);
      int orb = 0;
      for (int g = 0; g < nspace; ++g)
        for (int k = 0; k < size[g]; ++k, ++orb) o[g] += (int)((H.str[i] >> orb) & 1u);
      auto it = id.find(o);
      if (it == id.end()) {
        it = id.emplace(o, (int)occ[s].size()).first;
        occ[s].push_back(o);
        cnt[s].push_back(0);
      }
      cls[s][i] = it->second;
      ++cnt[s][it->second];
    }
  }
  const int ncA = (int)occ[0].size(), ncB = (int)occ[1].size();
  std::vector<uint8_t> ok((size_t)ncA * ncB, 0);
  long long ndet = 0;
  for (int a = 0; a < ncA; ++a)
    for (int b = 0; b < ncB; ++b) {
      bool keep = true;
      for (int g = 0; g < nspace; ++g) {
        const int e = occ[0][a][g] + occ[1][b][g];
        keep = keep && e >= gmin[g] && e <= gmax[g];
      }
      ok[(size_t)a * ncB + b] = keep;
      if (keep) ndet += cnt[0][a] * cnt[1][b];
    }
  if (nspace > 0 && ndet == 0) { set_error("the occupation restriction keeps no determinant"); return FORTE_ERR_ARG; }
  long long ndiag = 0;  // determinants |I>|I> (same string sets only)
  if (nspace > 0 && ctx->same_strings)
    for (size_t i = 0; i < cls[0].size(); ++i) ndiag += ok[(size_t)cls[0][i] * ncB + cls[1][i]];

  FORTE_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
  gas_release(ctx);
  int rc = hdiag_build(ctx);  // the unrestricted diagonal; excluded entries are set below
  if (rc) return rc;
  if (nspace == 0) {
    if (ndet_out) *ndet_out = ctx->Ndet;
    return FORTE_OK;
  }
  for (int s = 0; s < 2; ++s) {
    if (dev_alloc(&ctx->d_gas_cls[s], sizeof(int) * cls[s].size()) != cudaSuccess) {
      gas_release(ctx);
      set_error("cudaMalloc of the string classes failed");
      return FORTE_ERR_ALLOC;
    }
    FORTE_CUDA_TRY(copy_in(ctx, ctx->d_gas_cls[s], cls[s].data(), sizeof(int) * cls[s].size()));
  }
  if (dev_alloc(&ctx->d_gas_ok, ok.size()) != cudaSuccess) {
    gas_release(ctx);
    set_error("cudaMalloc of the class table failed");
    return FORTE_ERR_ALLOC;
  }
  FORTE_CUDA_TRY(copy_in(ctx, ctx->d_gas_ok, ok.data(), ok.size()));
  // kept alpha rows, those with the most kept beta strings first (they take longest)
  {
    std::vector<long long> kept(ncA, 0);
    for (int a = 0; a < ncA; ++a)
      for (int b = 0; b < ncB; ++b)
        if (ok[(size_t)a * ncB + b]) kept[a] += cnt[1][b];
    std::vector<int> rowsv;
    int maxnnz = 0;
    for (long long i = 0; i < ctx->sh[0].N; ++i) {
      if (kept[cls[0][i]] > 0) rowsv.push_back((int)i);
      maxnnz = std::max(maxnnz, ctx->sh[0].csr_ptr[i + 1] - ctx->sh[0].csr_ptr[i]);
    }
    std::stable_sort(rowsv.begin(), rowsv.end(), [&](int x, int y) { return kept[cls[0][x]] > kept[cls[0][y]]; });
    if (dev_alloc(&ctx->d_gas_rows, sizeof(int) * std::max<size_t>(1, rowsv.size())) != cudaSuccess) {
      gas_release(ctx);
      set_error("cudaMalloc of the restricted-sigma rows failed");
      return FORTE_ERR_ALLOC;
    }
    if (!rowsv.empty())
      FORTE_CUDA_TRY(copy_in(ctx, ctx->d_gas_rows, rowsv.data(), sizeof(int) * rowsv.size()));
    ctx->gas_nrows = (long long)rowsv.size();
    ctx->gas_maxnnz = maxnnz;
  }
  if (ncB <= GAS_MAXCLS && (rc = gas_lists(ctx, cls[1], cnt[1], ok, ncA))) {
    gas_release(ctx);
    return rc;
  }
  ctx->gas_nc[0] = ncA;
  ctx->gas_nc[1] = ncB;
  ctx->gas_ndet = ndet;
  ctx->gas_ndiag = ndiag;
  ctx->gas_on = true;
  if ((rc = gas_fill<double>(ctx, ctx->d_hdiag, 1, (double)INFINITY))) return rc;
  if (ctx->nguess > 0 && (rc = gas_mask(ctx, ctx->d_guess, ctx->nguess))) return rc;
  ctx->nroots_done = 0;  // earlier roots belong to another space
  FORTE_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
  if (ndet_out) *ndet_out = ndet;
  return FORTE_OK;
}

}  // namespace forte
