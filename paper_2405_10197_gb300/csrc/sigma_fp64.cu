// FP64 sigma build  sigma = H C  in the alpha-string x beta-string basis
// (Sec. II.A.1; Hamiltonian Eq. 1 in the spin-free form
//  H = sum_pq k_pq E_pq + 1/2 sum_pqrs (pq|rs) E_pq E_rs,  k_pq = h_pq - 1/2 sum_r (pr|rq)).
//
// Split by spin:
//   sigma_aa[Ia,Ib] = sum_Ja  H_aa[Ia,Ja] C[Ja,Ib]      (same-spin string Hamiltonian, CSR)
//   sigma_bb[Ia,Ib] = sum_Jb  H_bb[Ib,Jb] C[Ia,Jb]      (same kernel on C transposed)
//   sigma_ab[Ia,Ib] = sum_{e in L(Ia)} sum_{f in L(Jb)} s_e s_f (pq_e|rs_f) C[J_e, Jb],
//                     scattered to Ib = J_f for every Jb
// where L(I) is the signed single-replacement list of string I.
#include <algorithm>

#include "forte_internal.h"

namespace forte {

constexpr int SS_THREADS = 256;
constexpr int SS_CPT = 2;              // output columns per thread
constexpr int SS_SEG = 512;            // CSR entries staged per pass

// Y[row, c] (+)= sum_nz val * X[col, c]; rows of X and Y are ncol long.
// grid.x = nrow * nchunk, grid.y = vector.
template <typename T>
__global__ void __launch_bounds__(SS_THREADS) k_ss_spmm(const int *__restrict__ ptr,
                                                        const int *__restrict__ col,
                                                        const T *__restrict__ val,
                                                        const T *__restrict__ X, T *__restrict__ Y,
                                                        long long nrow, long long ncol, int nchunk,
                                                        long long vstride, int accumulate) {
  __shared__ int s_col[SS_SEG];
  __shared__ T s_val[SS_SEG];
  const long long row = blockIdx.x / nchunk;
  const int chunk = blockIdx.x % nchunk;
  const T *Xv = X + (long long)blockIdx.y * vstride;
  T *Yv = Y + (long long)blockIdx.y * vstride;
  long long c0 = (long long)chunk * SS_THREADS * SS_CPT + threadIdx.x;
  T acc[SS_CPT];
#pragma unroll
  for (int k = 0; k < SS_CPT; ++k) acc[k] = T(0);
  const int b = ptr[row], e = ptr[row + 1];
  for (int s0 = b; s0 < e; s0 += SS_SEG) {
    int cnt = min(SS_SEG, e - s0);
    __syncthreads();
    for (int i = threadIdx.x; i < cnt; i += SS_THREADS) {
      s_col[i] = col[s0 + i];
      s_val[i] = val[s0 + i];
    }
    __syncthreads();
#pragma unroll 4
    for (int i = 0; i < cnt; ++i) {
      const T v = s_val[i];
      const T *xr = Xv + (long long)s_col[i] * ncol;
#pragma unroll
      for (int k = 0; k < SS_CPT; ++k) {
        long long c = c0 + (long long)k * SS_THREADS;
        if (c < ncol) acc[k] += v * xr[c];
      }
    }
  }
#pragma unroll
  for (int k = 0; k < SS_CPT; ++k) {
    long long c = c0 + (long long)k * SS_THREADS;
    if (c < ncol) {
      T *y = Yv + row * ncol + c;
      *y = accumulate ? *y + acc[k] : acc[k];
    }
  }
}

// Y[c][r] (+)= X[r][c] for an R x Cc matrix per vector.
template <typename T>
__global__ void k_transpose(const T *__restrict__ X, T *__restrict__ Y, long long R, long long Cc,
                            long long vstride, int accumulate) {
  __shared__ T tile[32][33];
  const T *Xv = X + (long long)blockIdx.z * vstride;
  T *Yv = Y + (long long)blockIdx.z * vstride;
  long long r0 = (long long)blockIdx.y * 32, c0 = (long long)blockIdx.x * 32;
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    long long r = r0 + i, c = c0 + threadIdx.x;
    if (r < R && c < Cc) tile[i][threadIdx.x] = Xv[r * Cc + c];
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    long long c = c0 + i, r = r0 + threadIdx.x;
    if (r < R && c < Cc) {
      T v = tile[threadIdx.x][i];
      T *y = Yv + c * R + r;
      *y = accumulate ? *y + v : v;
    }
  }
}

// ---- FP64 alpha-beta term ------------------------------------------------------
//
// sigma[Ia, E_rs Jb] += s F[rs][Jb], F[rs][Jb] = sum_e s_e (pq_e|rs) C[J_e, Jb].
// The replacements that move no electron are taken together: all of Ia's read the row
// C[Ia] and all of Jb's write Jb, so they make one row (integrals summed over the
// orbitals of Ia) and one output (integrals summed over those of Jb, d_W).  At 7 of 14
// orbitals 50 x 50 instead of 56 x 56 products a determinant; the FP64 pipe (2 DFMA per
// clock and SM) bounds the rest.  One GB300, CAS(12,12), 4 vectors: 13.2 -> 8.9 ms.
// (Two replacements a thread, for two independent sums, measured 9.1 ms.)
//
// Shared memory: G[nk][npair] signed integral rows (row 0: the unmoved ones), row[NB] the
// output row, D[nk][TJ] gathered rows of C.  A thread takes one (string, replacement)
// of the tile at a time; the entry order of SpinDev::off gives the lanes' integral
// loads different banks.
constexpr int AB_THREADS = 256;

__global__ void __launch_bounds__(AB_THREADS) k_ab_fp64(const uint32_t *__restrict__ strA,
                                                        const uint32_t *__restrict__ offA, int noA,
                                                        const uint32_t *__restrict__ offB, int noB, long long NB,
                                                        const double *__restrict__ gpair, const double *__restrict__ W,
                                                        int npair, const double *__restrict__ C,
                                                        double *__restrict__ S, long long vstride, int TJ) {
  extern __shared__ double ab_smem[];
  const int nk = noA + 1;
  double *row = ab_smem;                   // NB
  double *G = row + NB;                    // nk * npair
  double *D = G + (size_t)nk * npair;      // nk * TJ
  __shared__ int s_J[80], s_pp[16];        // C rows; pair indices of Ia's unmoved replacements
  const long long Ia = blockIdx.x;
  const double *Cv = C + (long long)blockIdx.y * vstride;
  double *Sv = S + (long long)blockIdx.y * vstride;
  const uint32_t *la = offA + Ia * noA;
  for (int e = threadIdx.x; e < noA; e += AB_THREADS) s_J[e + 1] = la[e] & 0xFFFFu;
  const uint32_t occ = strA[Ia];
  const int npp = __popc(occ);
  if (threadIdx.x == 0) s_J[0] = (int)Ia;
  if (threadIdx.x < 32 && ((occ >> threadIdx.x) & 1u))
    s_pp[__popc(occ & ((1u << threadIdx.x) - 1u))] = threadIdx.x * (threadIdx.x + 3) / 2;  // pair (r, r)
  for (int i = threadIdx.x; i < noA * npair; i += AB_THREADS) {
    const uint32_t w = la[i / npair];
    const double g = gpair[(size_t)((w >> 16) & 0xFFu) * npair + i % npair];
    G[npair + i] = (w >> 31) ? -g : g;
  }
  for (long long i = threadIdx.x; i < NB; i += AB_THREADS) row[i] = 0.0;
  __syncthreads();
  for (int rs = threadIdx.x; rs < npair; rs += AB_THREADS) {
    double v = 0.0;
    for (int m = 0; m < npp; ++m) v += gpair[(size_t)s_pp[m] * npair + rs];
    G[rs] = v;
  }
  for (long long j0 = 0; j0 < NB; j0 += TJ) {
    const int tj = (int)min((long long)TJ, NB - j0);
    for (int i = threadIdx.x; i < nk * tj; i += AB_THREADS) {
      const int e = i / tj, j = i - e * tj;
      D[e * TJ + j] = Cv[(long long)s_J[e] * NB + j0 + j];
    }
    __syncthreads();
    const uint32_t *lb = offB + j0 * noB;
    for (int w = threadIdx.x; w < tj * noB; w += AB_THREADS) {
      const uint32_t f = lb[w];
      const double *g = G + ((f >> 16) & 0xFFu), *d = D + w / noB;
      double v = 0.0;
#pragma unroll 8
      for (int e = 0; e < nk; ++e) v = fma(g[e * npair], d[e * TJ], v);
      atomicAdd(&row[f & 0xFFFFu], (f >> 31) ? -v : v);
    }
    // the unmoved replacements of the tile's strings: output j itself, rows split over
    // the threads
    const int parts = AB_THREADS / TJ, part = threadIdx.x / TJ, j = threadIdx.x - part * TJ;
    if (part < parts && j < tj) {
      double v = 0.0;
      for (int e = 1 + part; e < nk; e += parts) {
        const uint32_t w = la[e - 1];
        const double x = W[(size_t)((w >> 16) & 0xFFu) * NB + j0 + j];
        v = fma((w >> 31) ? -x : x, D[e * TJ + j], v);
      }
      for (int m = part; m < npp; m += parts) v = fma(W[(size_t)s_pp[m] * NB + j0 + j], D[j], v);
      atomicAdd(&row[j0 + j], v);
    }
    __syncthreads();
  }
  for (long long i = threadIdx.x; i < NB; i += AB_THREADS) Sv[Ia * NB + i] += row[i];
}

static int ab_fp64(forte_ctx *ctx, const double *C, double *S, int nvec) {
  const int n = ctx->n, noA = ctx->na * (n - ctx->na), noB = ctx->nb * (n - ctx->nb);
  const long long NA = ctx->Na, NB = ctx->Nb;
  auto bytes = [&](int TJ) { return sizeof(double) * ((size_t)NB + (size_t)(noA + 1) * (ctx->npair + TJ)); };
  int TJ = 64;
  while (bytes(TJ) > 220 * 1024 && TJ > 8) TJ /= 2;
  if (bytes(TJ) > 220 * 1024) {
    set_error("alpha-beta FP64 kernel needs %zu bytes of shared memory", bytes(TJ));
    return FORTE_ERR_ARG;
  }
  FORTE_CUDA_TRY(set_smem_optin_max((const void *)k_ab_fp64));
  FORTE_PROF(ctx, "ab_fp64");
  k_ab_fp64<<<dim3((unsigned)NA, (unsigned)nvec), AB_THREADS, bytes(TJ), ctx->stream>>>(
      ctx->sd[0].str, ctx->sd[0].off, noA, ctx->sd[1].off, noB, NB, ctx->d_gpair, ctx->d_W, ctx->npair, C, S,
      ctx->Ndet, TJ);
  FORTE_LAUNCH_CHECK();
  return FORTE_OK;
}

// ---- small spaces (sigma_small) ------------------------------------------------
//
// Up to about 10 orbitals a sigma is a few microseconds of FP64 work, so the launches,
// the idle SMs and the latency of their chains count.  Every output is gathered by a few
// threads that split its sum and add their parts in a fixed order: no transposes, no
// atomics, and enough blocks for every SM.  One GB300, CAS(8,8), one vector: 53 -> 22 us
// (the general kernels: a 70-block grid, 21 us for the alpha-beta term alone).

constexpr int SM_THREADS = 256;

// Sum over the `parts` thread groups of a block of their values for column i of CH.
__device__ __forceinline__ double sm_sum(double v, double *red, int CH, int parts) {
  red[threadIdx.x] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < CH)
    for (int p = 0; p < parts; ++p) t += red[p * CH + threadIdx.x];
  return t;
}

// Alpha-alpha (ALPHA: S = H_aa C) or beta-beta (S += C H_bb) part of row blockIdx.y,
// columns blockIdx.x * CH .., vector blockIdx.z.
template <bool ALPHA>
__global__ void __launch_bounds__(SM_THREADS) k_ss_small(const int *__restrict__ ptr, const int *__restrict__ col,
                                                         const double *__restrict__ val, int nnz,
                                                         const double *__restrict__ C, double *__restrict__ S,
                                                         long long NB, long long vstride, int CH) {
  __shared__ double red[SM_THREADS];
  const int parts = SM_THREADS / CH, part = threadIdx.x / CH;
  const long long Ia = blockIdx.y, Ib = (long long)blockIdx.x * CH + threadIdx.x % CH;
  const double *Cv = C + (long long)blockIdx.z * vstride;
  cudaTriggerProgrammaticLaunchCompletion();
  double a = 0.0;
  if (Ib < NB) {
    if (ALPHA) {
      const int b = ptr[Ia], e = ptr[Ia + 1];
#pragma unroll 4
      for (int k = b + part; k < e; k += parts) a = fma(val[k], Cv[(long long)col[k] * NB + Ib], a);
    } else {
      const double *Cr = Cv + Ia * NB;
#pragma unroll 4
      for (int k = part; k < nnz; k += parts) a = fma(val[k * NB + Ib], Cr[col[k * NB + Ib]], a);
    }
  }
  a = sm_sum(a, red, CH, parts);
  if (!ALPHA) cudaGridDependencySynchronize();  // S of the kernel before
  if (threadIdx.x < CH && Ib < NB) {
    double *s = S + (long long)blockIdx.z * vstride + Ia * NB + Ib;
    *s = ALPHA ? a : *s + a;
  }
}

// Alpha-beta part of row blockIdx.y: D holds the rows C[J_e] whole, G the signed
// integrals, so that output Ib gathers F[rs][J] from every replacement J of Ib.
__global__ void __launch_bounds__(SM_THREADS) k_ab_small(const uint32_t *__restrict__ strA,
                                                         const uint32_t *__restrict__ offA, int noA,
                                                         const uint32_t *__restrict__ offB, int noB, int NB,
                                                         const double *__restrict__ gpair, const double *__restrict__ W,
                                                         int npair, const double *__restrict__ C,
                                                         double *__restrict__ S, long long vstride, int CH) {
  extern __shared__ double ab_smem[];
  __shared__ double red[SM_THREADS];
  __shared__ int s_pp[16];
  const int nk = noA + 1;
  double *G = ab_smem, *D = G + nk * npair;  // [nk][npair], [nk][NB]
  const int Ia = blockIdx.y;
  const double *Cv = C + (long long)blockIdx.z * vstride;
  const uint32_t *la = offA + (long long)Ia * noA;
  const uint32_t occ = strA[Ia];
  const int npp = __popc(occ);
  if (threadIdx.x < 32 && ((occ >> threadIdx.x) & 1u))
    s_pp[__popc(occ & ((1u << threadIdx.x) - 1u))] = threadIdx.x * (threadIdx.x + 3) / 2;  // pair (r, r)
  for (int i = threadIdx.x; i < noA * npair; i += SM_THREADS) {
    const uint32_t w = la[i / npair];
    const double g = gpair[((w >> 16) & 0xFFu) * npair + i % npair];
    G[npair + i] = (w >> 31) ? -g : g;
  }
  for (int i = threadIdx.x; i < nk * NB; i += SM_THREADS) {
    const int e = i / NB;
    D[i] = Cv[(long long)(e ? (int)(la[e - 1] & 0xFFFFu) : Ia) * NB + (i - e * NB)];
  }
  __syncthreads();
  for (int rs = threadIdx.x; rs < npair; rs += SM_THREADS) {
    double v = 0.0;
    for (int m = 0; m < npp; ++m) v += gpair[s_pp[m] * npair + rs];
    G[rs] = v;
  }
  __syncthreads();
  const int parts = SM_THREADS / CH, part = threadIdx.x / CH;
  const int Ib = blockIdx.x * CH + threadIdx.x % CH;
  double out = 0.0;
  if (Ib < NB) {
    const uint32_t *lb = offB + (long long)Ib * noB;
    for (int f = part; f < noB; f += parts) {  // <Ib|E|J> = <J|E|Ib>, same pair and sign
      const uint32_t w = lb[f];
      const double *g = G + ((w >> 16) & 0xFFu), *d = D + (w & 0xFFFFu);
      double a = 0.0, b = 0.0;
      int e = 0;
#pragma unroll 4
      for (; e + 1 < nk; e += 2) {
        a = fma(g[e * npair], d[e * NB], a);
        b = fma(g[(e + 1) * npair], d[(e + 1) * NB], b);
      }
      if (e < nk) a = fma(g[e * npair], d[e * NB], a);
      out += (w >> 31) ? -(a + b) : a + b;
    }
    // the unmoved replacements of Ib
    for (int e = 1 + part; e < nk; e += parts) {
      const uint32_t w = la[e - 1];
      const double x = W[(long long)((w >> 16) & 0xFFu) * NB + Ib];
      out = fma((w >> 31) ? -x : x, D[e * NB + Ib], out);
    }
    for (int m = part; m < npp; m += parts) out = fma(W[(long long)s_pp[m] * NB + Ib], D[Ib], out);
  }
  out = sm_sum(out, red, CH, parts);
  cudaGridDependencySynchronize();  // S of the kernels before
  if (threadIdx.x < CH && Ib < NB) S[(long long)blockIdx.z * vstride + (long long)Ia * NB + Ib] += out;
}

double fp64_products(const forte_ctx *ctx) {
  const SpinHost &A = ctx->sh[0], &B = ctx->sh[ctx->same_strings ? 0 : 1];
  const double ka = A.nel * (ctx->n - A.nel) + 1, kb = B.nel * (ctx->n - B.nel) + 1;
  return (double)ctx->Ndet * (ka * kb + (double)A.csr_ptr[1] + (double)B.csr_ptr[1]);
}

// The small-space FP64 kernels against the double-FP32 / digit-slice ones, us on one GB300:
// 9.6 M products (9 orbitals, 5 + 4) 48 against 85 / 139, 38 M (four vectors of it) 100
// against 119 / 242, 59 M (10, 5 + 5) 166 against 144 / 223, 236 M 579 against 275 / 472.
// The line is where FP64 and double-FP32 meet, and serves the digit-slice mode too, whose
// own crossing with FP64 lies at about 100 M.  Between 40 M and some 4 G products that mode
// is slower than the double-FP32 one (188 M 406 against 276, 1.6 G 1257 against 1246, 5.4 G
// 2988 against 3517): FORTE_OZ64 runs the kernels it names all the same.
bool fp64_small(const forte_ctx *ctx, int nvec) {
  return ctx->sd[1].ell_col && fp64_products(ctx) * nvec <= 40e6;
}

bool small_route(const forte_ctx *ctx, bool waits) {
  // (a longer wait changes nothing but the time of a failure; a shorter one is for the
  // kernels that wait, so they run)
  const bool cut = ctx->wait_budget != 0 && ctx->wait_budget < WAIT_BUDGET_DEFAULT;
  return ctx->small_route == 1 || (ctx->small_route == -1 && !(waits && cut));
}

// Columns per block: as many threads share an output as leave two blocks an SM busy, and
// 32 columns once the grid is larger than that.
static int sm_columns(long long NA, long long NB, int nvec) {
  int CH = 32;
  while (CH > 8 && NA * ((NB + CH - 1) / CH) * nvec < 2 * 152) CH /= 2;
  return CH;
}

static bool sd_small(const forte_ctx *ctx) { return ctx->sd[1].ell_col != nullptr; }

static int sigma_fp64_small(forte_ctx *ctx, const double *C, double *S, int nvec) {
  cudaStream_t st = ctx->stream;
  const int n = ctx->n, noA = ctx->na * (n - ctx->na), noB = ctx->nb * (n - ctx->nb);
  const long long NA = ctx->Na, NB = ctx->Nb, ND = ctx->Ndet;
  const int CH = sm_columns(NA, NB, nvec);
  const SpinDev &A = ctx->sd[0], &B = ctx->sd[1];
  const dim3 grid((unsigned)((NB + CH - 1) / CH), (unsigned)NA, (unsigned)nvec);
  // The second and third kernel may start while the one before runs (they read C and the
  // tables) and wait for it only where they add to S: their launch and first loads
  // overlap its tail.
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(SM_THREADS);
  cfg.stream = st;
  {
    FORTE_PROF(ctx, "ss_spmm");
    k_ss_small<true><<<grid, SM_THREADS, 0, st>>>(A.csr_ptr, A.csr_col, A.csr_val, 0, C, S, NB, ND, CH);
    FORTE_LAUNCH_CHECK();
  }
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  {
    FORTE_PROF(ctx, "ss_spmm");
    FORTE_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_ss_small<false>, (const int *)nullptr, (const int *)B.ell_col,
                                      (const double *)B.ell_val, (int)ctx->sh[ctx->same_strings ? 0 : 1].csr_ptr[1], C, S,
                                      NB, ND, CH));
  }
  if (ctx->sh[0].nk > 0 && ctx->sh[ctx->same_strings ? 0 : 1].nk > 0) {
    const size_t smem = sizeof(double) * (size_t)(noA + 1) * (NB + ctx->npair);
    if (smem > 44 * 1024) FORTE_CUDA_TRY(set_smem_optin_max((const void *)k_ab_small));
    cfg.dynamicSmemBytes = smem;
    FORTE_PROF(ctx, "ab_fp64");
    FORTE_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_ab_small, (const uint32_t *)A.str, (const uint32_t *)A.off, noA,
                                      (const uint32_t *)B.off, noB, (int)NB, (const double *)ctx->d_gpair,
                                      (const double *)ctx->d_W, ctx->npair, C, S, ND, CH));
  }
  return FORTE_OK;
}

int sigma_fp64(forte_ctx *ctx, const double *C, double *S, int nvec) {
  if (sd_small(ctx)) return sigma_fp64_small(ctx, C, S, nvec);
  // beta-beta scratch: T1 = C^T, T2 = H_bb T1 (grown on demand)
  const long long ND = ctx->Ndet;
  int rc = ctx->sc_t1.ensure(sizeof(double) * ND * nvec);
  if (rc) return rc;
  rc = ctx->sc_t2.ensure(sizeof(double) * ND * nvec);
  if (rc) return rc;
  return sigma_fp64_scratch(ctx, C, S, nvec, (double *)ctx->sc_t1.ptr, (double *)ctx->sc_t2.ptr);
}

// The FP64 sigma with caller-provided scratch T1, T2 (each >= nvec * Ndet
// doubles); allocates nothing.  Shared by forte_sigma (context scratch) and
// forte_sigma_fp64_noalloc (the library's fixed array).
int sigma_fp64_scratch(forte_ctx *ctx, const double *C, double *S, int nvec, double *T1, double *T2) {
  if (sd_small(ctx)) return sigma_fp64_small(ctx, C, S, nvec);
  cudaStream_t st = ctx->stream;
  const long long NA = ctx->Na, NB = ctx->Nb, ND = ctx->Ndet;
  // alpha-alpha: S = H_aa C
  {
    int nchunk = (int)((NB + SS_THREADS * SS_CPT - 1) / (SS_THREADS * SS_CPT));
    dim3 grid((unsigned)(NA * nchunk), nvec);
    FORTE_PROF(ctx, "ss_spmm");
    k_ss_spmm<double><<<grid, SS_THREADS, 0, st>>>(ctx->sd[0].csr_ptr, ctx->sd[0].csr_col,
                                                   ctx->sd[0].csr_val, C, S, NA, NB, nchunk, ND, 0);
    FORTE_LAUNCH_CHECK();
  }
  // beta-beta: T1 = C^T, T2 = H_bb T1, S += T2^T
  {
    dim3 tb(32, 8);
    dim3 g1((unsigned)((NB + 31) / 32), (unsigned)((NA + 31) / 32), nvec);
    {
      FORTE_PROF(ctx, "transpose");
      k_transpose<double><<<g1, tb, 0, st>>>(C, T1, NA, NB, ND, 0);
      FORTE_LAUNCH_CHECK();
    }
    int nchunk = (int)((NA + SS_THREADS * SS_CPT - 1) / (SS_THREADS * SS_CPT));
    dim3 grid((unsigned)(NB * nchunk), nvec);
    {
      FORTE_PROF(ctx, "ss_spmm");
      k_ss_spmm<double><<<grid, SS_THREADS, 0, st>>>(ctx->sd[1].csr_ptr, ctx->sd[1].csr_col,
                                                     ctx->sd[1].csr_val, T1, T2, NB, NA, nchunk, ND, 0);
      FORTE_LAUNCH_CHECK();
    }
    dim3 g2((unsigned)((NA + 31) / 32), (unsigned)((NB + 31) / 32), nvec);
    {
      FORTE_PROF(ctx, "transpose");
      k_transpose<double><<<g2, tb, 0, st>>>(T2, S, NB, NA, ND, 1);
      FORTE_LAUNCH_CHECK();
    }
  }
  // alpha-beta
  if (ctx->sh[0].nk > 0 && ctx->sh[ctx->same_strings ? 0 : 1].nk > 0)
    return ab_fp64(ctx, C, S, nvec);
  return FORTE_OK;
}

// FP32 same-spin term for the reduced-precision path:
//   S32 = H_aa C32  then  S32 += (H_bb C32^T)^T,  via the scratch buffers T1/T2.
int same_spin_f32(forte_ctx *ctx, const float *C32, float *S32, float *T1, float *T2, int nvec) {
  cudaStream_t st = ctx->stream;
  const long long NA = ctx->Na, NB = ctx->Nb, ND = ctx->Ndet;
  {
    int nchunk = (int)((NB + SS_THREADS * SS_CPT - 1) / (SS_THREADS * SS_CPT));
    dim3 grid((unsigned)(NA * nchunk), nvec);
    {
      FORTE_PROF(ctx, "ss_spmm_f32");
      k_ss_spmm<float><<<grid, SS_THREADS, 0, st>>>(ctx->sd[0].csr_ptr, ctx->sd[0].csr_col,
                                                    ctx->sd[0].csr_val32, C32, S32, NA, NB, nchunk, ND, 0);
      FORTE_LAUNCH_CHECK();
    }
  }
  dim3 tb(32, 8);
  dim3 g1((unsigned)((NB + 31) / 32), (unsigned)((NA + 31) / 32), nvec);
  {
    FORTE_PROF(ctx, "transpose_f32");
    k_transpose<float><<<g1, tb, 0, st>>>(C32, T1, NA, NB, ND, 0);
    FORTE_LAUNCH_CHECK();
  }
  {
    int nchunk = (int)((NA + SS_THREADS * SS_CPT - 1) / (SS_THREADS * SS_CPT));
    dim3 grid((unsigned)(NB * nchunk), nvec);
    FORTE_PROF(ctx, "ss_spmm_f32");
    k_ss_spmm<float><<<grid, SS_THREADS, 0, st>>>(ctx->sd[1].csr_ptr, ctx->sd[1].csr_col,
                                                  ctx->sd[1].csr_val32, T1, T2, NB, NA, nchunk, ND, 0);
    FORTE_LAUNCH_CHECK();
  }
  dim3 g2((unsigned)((NA + 31) / 32), (unsigned)((NB + 31) / 32), nvec);
  {
    FORTE_PROF(ctx, "transpose_f32");
    k_transpose<float><<<g2, tb, 0, st>>>(T2, S32, NB, NA, ND, 1);
    FORTE_LAUNCH_CHECK();
  }
  return FORTE_OK;
}

// H_II = H_aa[Ia,Ia] + H_bb[Ib,Ib] + sum_{i in Ia, j in Ib} (ii|jj)
__global__ void k_hdiag(const double *__restrict__ dA, const double *__restrict__ dB,
                        const double *__restrict__ W, const uint32_t *__restrict__ strB, int n,
                        long long NA, long long NB, double *__restrict__ out) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= NA * NB) return;
  long long ia = i / NB, ib = i % NB;
  uint32_t s = strB[ib];
  double v = dA[ia] + dB[ib];
  const double *w = W + ia * n;
  while (s) {
    int j = __ffs(s) - 1;
    v += w[j];
    s &= s - 1;
  }
  out[i] = v;
}

int hdiag_build(forte_ctx *ctx) {
  const int n = ctx->n;
  const SpinHost &A = ctx->sh[0];
  std::vector<double> W((size_t)A.N * n, 0.0);
  for (long long ia = 0; ia < A.N; ++ia)
    for (int j = 0; j < n; ++j) {
      double v = 0.0;
      for (int i = 0; i < n; ++i)
        if ((A.str[ia] >> i) & 1u) v += ctx->eri[(((size_t)i * n + i) * n + j) * n + j];
      W[(size_t)ia * n + j] = v;
    }
  DevTemp tmp;
  FORTE_CUDA_TRY(dev_alloc(&tmp.ptr, sizeof(double) * W.size()));
  double *dW = (double *)tmp.ptr;
  FORTE_CUDA_TRY(copy_in(ctx, dW, W.data(), sizeof(double) * W.size()));
  if (!ctx->d_hdiag) {
    cudaError_t e = dev_alloc(&ctx->d_hdiag, sizeof(double) * ctx->Ndet);
    if (e != cudaSuccess) {
      set_error("cudaMalloc hdiag failed: %s", cudaGetErrorString(e));
      return FORTE_ERR_ALLOC;
    }
  }
  long long nt = ctx->Ndet;
  k_hdiag<<<(unsigned)((nt + 255) / 256), 256, 0, ctx->stream>>>(
      ctx->sd[0].diag, ctx->sd[1].diag, dW, ctx->sd[1].str, n, ctx->Na, ctx->Nb, ctx->d_hdiag);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  if (e != cudaSuccess) {
    set_error("hdiag kernel failed: %s", cudaGetErrorString(e));
    return FORTE_ERR_CUDA;
  }
  return FORTE_OK;
}

// ============================================================================
// FP64-class sigma in double-FP32 arithmetic (precision FORTE_DF32, and the
// refinement operator of the reduced-precision modes).
//
// Every FP64 operand x is held as an unevaluated pair x = hi + lo of FP32 values
// (hi = fl32(x), lo = fl32(x - hi); |x - hi - lo| <= 2^-48 |x|).  A product term
// a b adds hi_a hi_b exactly (the FMA residual of the FP32 product), the cross
// terms hi_a lo_b + lo_a hi_b in FP32, and drops lo_a lo_b (2^-48 relative); the
// running sum is a compensated pair (TwoSum of Knuth, TAOCP vol. 2, Sec. 4.2.2).
// Relative error per product about 2^-46.  The FP32 pipe of this GPU issues 64
// times the FP64 pipe's operations, so ~12 FP32 operations per term beat one DFMA.
// ============================================================================

// Two such sums side by side in the packed FP32 instructions (add / mul / fma .f32x2), which
// issue twice the operations of the single ones: measured on one GB300, the same-spin
// product of one spin at CAS(14,14) takes 2.5 ms with them, 3.64 ms without.  The
// operations and their rounding are those of a TwoSum with FMA product residual.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pk2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpk2(f32x2 v, float &a, float &b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
constexpr f32x2 F32X2_M1 = 0xBF800000BF800000ull;  // (-1, -1)
constexpr f32x2 F32X2_SIGN = 0x8000000080000000ull;

// (ah, al) += (gh + gl)(xh + xl)
__device__ __forceinline__ void df_fma2(f32x2 &ah, f32x2 &al, f32x2 gh, f32x2 gl, f32x2 xh, f32x2 xl) {
  const f32x2 p = mul2(gh, xh);
  const f32x2 npe = fma2(gh ^ F32X2_SIGN, xh, p);  // p - gh xh: minus the product's residual
  const f32x2 c = fma2(gh, xl, mul2(gl, xh));
  const f32x2 s = add2(ah, p);
  const f32x2 bb = fma2(ah, F32X2_M1, s);
  const f32x2 e = add2(fma2(fma2(bb, F32X2_M1, s), F32X2_M1, ah), fma2(bb, F32X2_M1, p));
  ah = s;
  al = add2(al, add2(e, fma2(npe, F32X2_M1, c)));
}

// The operands are planar: hi [rows][ld] and lo behind it, rows padded with zeros to a
// multiple of four, so that two neighbours are one packed operand.
__device__ __forceinline__ void df_split(double v, float &h, float &l) {
  h = (float)v;
  l = (float)(v - (double)h);
}
// FP32 to FP64 with integer operations for normal numbers (the conversion instruction
// shares the narrow FP64 pipe).
__device__ __forceinline__ double to_double(float x) {
  const uint32_t b = __float_as_uint(x), e = (b >> 23) & 255u;
  if (e == 0u || e == 255u) return (double)x;  // zero, subnormal, infinity, NaN
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + (896u << 20))), (int)(b << 29));
}
static long long df_ld(long long ncol) { return (ncol + 3) & ~3LL; }

// hi, lo [vector][R][ld] of X [vector][R][Cc].
__global__ void k_df_split(const double *__restrict__ X, float *__restrict__ hi, float *__restrict__ lo, long long rows,
                           long long Cc, long long ld) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < rows * ld; i += (long long)gridDim.x * blockDim.x) {
    const long long r = i / ld, c = i - r * ld;
    float h = 0.f, l = 0.f;
    if (c < Cc) df_split(X[r * Cc + c], h, l);
    hi[i] = h;
    lo[i] = l;
  }
}

// hi, lo [vector][Cc][ld] of the transpose of X [vector][R][Cc].
__global__ void k_df_split_t(const double *__restrict__ X, float *__restrict__ hi, float *__restrict__ lo, long long R,
                             long long Cc, long long ld) {
  __shared__ double tile[32][33];
  const double *Xv = X + (long long)blockIdx.z * R * Cc;
  const long long r0 = (long long)blockIdx.y * 32, c0 = (long long)blockIdx.x * 32, o = (long long)blockIdx.z * Cc * ld;
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const long long r = r0 + i, c = c0 + threadIdx.x;
    tile[i][threadIdx.x] = (r < R && c < Cc) ? Xv[r * Cc + c] : 0.0;
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const long long c = c0 + i, r = r0 + threadIdx.x;
    if (r < ld && c < Cc) {
      float h, l;
      df_split(tile[threadIdx.x][i], h, l);
      hi[o + c * ld + r] = h;
      lo[o + c * ld + r] = l;
    }
  }
}

// (hi, lo) pairs of a table
__global__ void k_df_pairs(const double *__restrict__ x, float2 *__restrict__ y, long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    float h, l;
    df_split(x[i], h, l);
    y[i] = make_float2(h, l);
  }
}

// Same-spin CSR product in double-FP32: Y[row, c] = sum_nz val * X[col, c], Y FP64 [nrow][ncol].
// grid.x = nrow * nchunk, grid.y = vector.  A thread takes four neighbouring columns (two
// 16-byte loads a term); blockDim and nchunk are chosen so that few lanes lie beyond the
// last column.
constexpr int SSD_SEG = 256;  // CSR entries staged per pass
__global__ void __launch_bounds__(256) k_ss_spmm_df(const int *__restrict__ ptr, const int *__restrict__ col,
                                                    const float2 *__restrict__ val, const float *__restrict__ Xhi,
                                                    const float *__restrict__ Xlo, double *__restrict__ Y,
                                                    long long nrow, long long ncol, long long ld, int nchunk) {
  __shared__ float2 sv[SSD_SEG];
  __shared__ unsigned srow[SSD_SEG];  // row start in units of four columns
  const long long row = blockIdx.x / nchunk;
  const int chunk = blockIdx.x % nchunk, nt = blockDim.x;
  const long long q = (long long)chunk * nt + threadIdx.x;          // columns 4q .. 4q + 3
  const long long vo = (long long)blockIdx.y * nrow * (ld / 4), qs = min(q, ld / 4 - 1);  // (past the end: the last)
  const ulonglong2 *hp = reinterpret_cast<const ulonglong2 *>(Xhi) + vo + qs;
  const ulonglong2 *lp = reinterpret_cast<const ulonglong2 *>(Xlo) + vo + qs;
  f32x2 ah0 = 0, ah1 = 0, al0 = 0, al1 = 0;
  const int b = ptr[row], e = ptr[row + 1];
  for (int s0 = b; s0 < e; s0 += SSD_SEG) {
    const int cnt = min(SSD_SEG, e - s0);
    __syncthreads();
    for (int i = threadIdx.x; i < cnt; i += nt) {
      sv[i] = val[s0 + i];
      srow[i] = (unsigned)(col[s0 + i] * (ld / 4));
    }
    __syncthreads();
#pragma unroll 4
    for (int i = 0; i < cnt; ++i) {
      const float2 v = sv[i];
      const f32x2 gh = pk2(v.x, v.x), gl = pk2(v.y, v.y);
      const ulonglong2 h = __ldg(hp + srow[i]), l = __ldg(lp + srow[i]);
      df_fma2(ah0, al0, gh, gl, h.x, l.x);
      df_fma2(ah1, al1, gh, gl, h.y, l.y);
    }
  }
  if (4 * q >= ncol) return;
  float h[4], l[4];
  unpk2(ah0, h[0], h[1]);
  unpk2(ah1, h[2], h[3]);
  unpk2(al0, l[0], l[1]);
  unpk2(al1, l[2], l[3]);
  double *y = Y + ((long long)blockIdx.y * nrow + row) * ncol + 4 * q;
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (4 * q + k < ncol) y[k] = (double)h[k] + (double)l[k];
}

static int ss_spmm_df(forte_ctx *ctx, const SpinDev &sp, const float2 *val, const float *Xhi, const float *Xlo, double *Y,
                      long long nrow, long long ncol, int nvec) {
  // the block size (whole warps, 64 .. 256) with the fewest idle lanes
  const long long ld = df_ld(ncol);
  int nt = 256, nchunk = 1;
  long long best = 1LL << 62;
  for (int t = 256; t >= 64; t -= 32) {
    const long long n = (ld / 4 + t - 1) / t;
    if (n * t < best) {
      best = n * t;
      nt = t;
      nchunk = (int)n;
    }
  }
  FORTE_PROF(ctx, "ss_spmm_df");
  k_ss_spmm_df<<<dim3((unsigned)(nrow * nchunk), (unsigned)nvec), nt, 0, ctx->stream>>>(sp.csr_ptr, sp.csr_col, val, Xhi,
                                                                                        Xlo, Y, nrow, ncol, ld, nchunk);
  FORTE_LAUNCH_CHECK();
  return FORTE_OK;
}

// The alpha-beta term in double-FP32 (the sums of k_ab_fp64).  A thread's sum over the rows e
// runs as two packed ones over even and odd e, so G[pair] and D[string] hold 16-byte quads
// (hi_e, hi_e+1, lo_e, lo_e+1), e padded with zeros to nkp, nkp / 2 odd: quads of different
// pair mod 8 lie in different banks, the order SpinDev::off deals the replacements in.
// Bound by those shared-memory loads and the 13 packed operations of two terms.  One
// GB300, CAS(13; 7,5): 4.06 -> 2.69 ms.
constexpr int AB_DF_THREADS = 512;
__global__ void __launch_bounds__(AB_DF_THREADS) k_ab_df(const uint32_t *__restrict__ strA,
                                                         const uint32_t *__restrict__ offA, int noA,
                                                         const uint32_t *__restrict__ offB, int noB, long long NB,
                                                         const double *__restrict__ gpair,
                                                         const float2 *__restrict__ gpair2,
                                                         const float2 *__restrict__ W2, int npair, int nkp,
                                                         const float *__restrict__ Chi, const float *__restrict__ Clo,
                                                         long long ld, double *__restrict__ S, long long vstride,
                                                         int TJ) {
  constexpr int NT = AB_DF_THREADS;
  extern __shared__ double ab_smem[];
  const int nk = noA + 1;
  double *row = ab_smem;                                    // NB
  float *G = reinterpret_cast<float *>(row + ((NB + 1) & ~1LL));  // [npair][nkp / 2] quads
  float *D = G + 2 * (size_t)npair * nkp;                         // [TJ][nkp / 2] quads
  // element e of row r: hi at quad(r, e), lo two floats further
  auto quad = [nkp](int r, int e) { return (r * (nkp >> 1) + (e >> 1)) * 4 + (e & 1); };
  __shared__ int s_J[80], s_pp[16];
  const long long Ia = blockIdx.x;
  const float *Ch = Chi + (long long)blockIdx.y * gridDim.x * ld, *Cl = Clo + (long long)blockIdx.y * gridDim.x * ld;
  double *Sv = S + (long long)blockIdx.y * vstride;
  const uint32_t *la = offA + Ia * noA;
  for (int e = threadIdx.x; e < noA; e += NT) s_J[e + 1] = la[e] & 0xFFFFu;
  const uint32_t occ = strA[Ia];
  const int npp = __popc(occ);
  if (threadIdx.x == 0) s_J[0] = (int)Ia;
  if (threadIdx.x < 32 && ((occ >> threadIdx.x) & 1u))
    s_pp[__popc(occ & ((1u << threadIdx.x) - 1u))] = threadIdx.x * (threadIdx.x + 3) / 2;  // pair (r, r)
  for (int i = threadIdx.x; i < npair * (nkp - 1); i += NT) {
    const int e = 1 + i / npair, rs = i % npair;  // (the padding rows e >= nk are zero)
    float2 g = make_float2(0.f, 0.f);
    if (e < nk) {
      const uint32_t w = la[e - 1];
      g = gpair2[(size_t)((w >> 16) & 0xFFu) * npair + rs];
      if (w >> 31) g = make_float2(-g.x, -g.y);
    }
    G[quad(rs, e)] = g.x;
    G[quad(rs, e) + 2] = g.y;
  }
  for (long long i = threadIdx.x; i < NB; i += NT) row[i] = 0.0;
  for (int i = threadIdx.x; i < TJ * (nkp - nk); i += NT) {
    const int j = i / (nkp - nk), e = nk + i % (nkp - nk);
    D[quad(j, e)] = D[quad(j, e) + 2] = 0.f;
  }
  __syncthreads();
  for (int rs = threadIdx.x; rs < npair; rs += NT) {
    double v = 0.0;
    for (int m = 0; m < npp; ++m) v += gpair[(size_t)s_pp[m] * npair + rs];
    df_split(v, G[quad(rs, 0)], G[quad(rs, 0) + 2]);
  }
  for (long long j0 = 0; j0 < NB; j0 += TJ) {
    const int tj = (int)min((long long)TJ, NB - j0);
    for (int i = threadIdx.x; i < nk * tj; i += NT) {
      const int e = i / tj, j = i - e * tj;
      const long long at = (long long)s_J[e] * ld + j0 + j;
      D[quad(j, e)] = Ch[at];
      D[quad(j, e) + 2] = Cl[at];
    }
    __syncthreads();
    const uint32_t *lb = offB + j0 * noB;
    for (int w = threadIdx.x; w < tj * noB; w += NT) {
      const uint32_t f = lb[w];
      const ulonglong2 *g = reinterpret_cast<const ulonglong2 *>(G) + (int)((f >> 16) & 0xFFu) * (nkp / 2);
      const ulonglong2 *d = reinterpret_cast<const ulonglong2 *>(D) + w / noB * (nkp / 2);
      f32x2 ah = 0, al = 0;
#pragma unroll 4
      for (int e = 0; e < nkp / 2; ++e) {
        const ulonglong2 x = g[e], y = d[e];
        df_fma2(ah, al, x.x, x.y, y.x, y.y);
      }
      // the two sums joined in FP32 (TwoSum), one FP64 addition: a conversion or addition
      // on the FP64 pipe takes a warp 16 clocks, as long as four terms
      float h0, h1, l0, l1;
      unpk2(ah, h0, h1);
      unpk2(al, l0, l1);
      const float h = h0 + h1, b = h - h0;
      const double v = to_double(h) + to_double(((h0 - (h - b)) + (h1 - b)) + (l0 + l1));
      atomicAdd(&row[f & 0xFFFFu], (f >> 31) ? -v : v);
    }
    // the unmoved replacements of the tile's strings: output j itself, rows split over
    // the threads
    const int parts = NT / TJ, part = threadIdx.x / TJ, j = threadIdx.x - part * TJ;
    if (part < parts && j < tj) {
      f32x2 ah = 0, al = 0;
      auto term = [&](float2 x, int e) { df_fma2(ah, al, pk2(x.x, 0.f), pk2(x.y, 0.f), pk2(D[quad(j, e)], 0.f), pk2(D[quad(j, e) + 2], 0.f)); };
      for (int e = 1 + part; e < nk; e += parts) {
        const uint32_t w = la[e - 1];
        const float2 x = W2[(size_t)((w >> 16) & 0xFFu) * NB + j0 + j];
        term((w >> 31) ? make_float2(-x.x, -x.y) : x, e);
      }
      for (int m = part; m < npp; m += parts) term(W2[(size_t)s_pp[m] * NB + j0 + j], 0);
      float h, l, z;
      unpk2(ah, h, z);
      unpk2(al, l, z);
      atomicAdd(&row[j0 + j], (double)h + (double)l);
    }
    __syncthreads();
  }
  for (long long i = threadIdx.x; i < NB; i += NT) Sv[Ia * NB + i] += row[i];
}

static int ab_df(forte_ctx *ctx, const float *Chi, const float *Clo, double *S, int nvec) {
  const int n = ctx->n, noA = ctx->na * (n - ctx->na), noB = ctx->nb * (n - ctx->nb);
  const long long NA = ctx->Na, NB = ctx->Nb;
  int nkp = (noA + 2) & ~1;
  if ((nkp / 2) % 2 == 0) nkp += 2;
  auto bytes = [&](int TJ) { return sizeof(double) * (((size_t)NB + 1) / 2 * 2 + (size_t)nkp * (ctx->npair + TJ)); };
  int TJ = 64;  // (narrower where that lets a second block onto the SM)
  if (bytes(64) > 112 * 1024 && bytes(32) <= 112 * 1024) TJ = 32;
  while (bytes(TJ) > 220 * 1024 && TJ > 8) TJ /= 2;
  if (bytes(TJ) > 220 * 1024) {
    set_error("alpha-beta double-FP32 kernel needs %zu bytes of shared memory", bytes(TJ));
    return FORTE_ERR_ARG;
  }
  FORTE_CUDA_TRY(set_smem_optin_max((const void *)k_ab_df));
  FORTE_PROF(ctx, "ab_df");
  k_ab_df<<<dim3((unsigned)NA, (unsigned)nvec), AB_DF_THREADS, bytes(TJ), ctx->stream>>>(
      ctx->sd[0].str, ctx->sd[0].off, noA, ctx->sd[1].off, noB, NB, ctx->d_gpair, (const float2 *)ctx->d_gpair2,
      (const float2 *)ctx->d_W2, ctx->npair, nkp, Chi, Clo, df_ld(NB), S, ctx->Ndet, TJ);
  FORTE_LAUNCH_CHECK();
  return FORTE_OK;
}

static int df_setup(forte_ctx *ctx) {
  if (ctx->df_ready) return FORTE_OK;
  const int np = ctx->npair;
  FORTE_CUDA_TRY(alloc_once(&ctx->d_gpair2, sizeof(float2) * (size_t)np * np));
  k_df_pairs<<<(unsigned)std::min<long long>(((long long)np * np + 255) / 256, 1024), 256, 0, ctx->stream>>>(
      ctx->d_gpair, (float2 *)ctx->d_gpair2, (long long)np * np);
  FORTE_LAUNCH_CHECK();
  const long long nw = (long long)np * ctx->Nb;
  FORTE_CUDA_TRY(alloc_once(&ctx->d_W2, sizeof(float2) * (size_t)nw));
  k_df_pairs<<<(unsigned)std::min<long long>((nw + 255) / 256, 152LL * 16), 256, 0, ctx->stream>>>(
      ctx->d_W, (float2 *)ctx->d_W2, nw);
  FORTE_LAUNCH_CHECK();
  const int nsp = ctx->same_strings ? 1 : 2;
  for (int s = 0; s < nsp; ++s) {
    const long long nnz = (long long)ctx->sh[s].csr_col.size();
    FORTE_CUDA_TRY(alloc_once(&ctx->d_csr_val2[s], sizeof(float2) * (size_t)std::max(1LL, nnz)));
    if (nnz > 0) {
      k_df_pairs<<<(unsigned)std::min<long long>((nnz + 255) / 256, 152LL * 16), 256, 0, ctx->stream>>>(
          ctx->sd[s].csr_val, (float2 *)ctx->d_csr_val2[s], nnz);
      FORTE_LAUNCH_CHECK();
    }
  }
  if (ctx->same_strings) ctx->d_csr_val2[1] = ctx->d_csr_val2[0];
  ctx->df_ready = true;
  return FORTE_OK;
}

int sigma_df(forte_ctx *ctx, const double *C, double *S, int nvec, bool with_ab) {
  if (with_ab && small_route(ctx, false) && fp64_small(ctx, nvec))
    return sigma_fp64(ctx, C, S, nvec);  // faster and more exact there
  int rc = df_setup(ctx);
  if (rc) return rc;
  cudaStream_t st = ctx->stream;
  const long long NA = ctx->Na, NB = ctx->Nb, ND = ctx->Ndet;
  const long long ldb = df_ld(NB), lda = df_ld(NA);
  const size_t nc = (size_t)nvec * NA * ldb, nt = (size_t)nvec * NB * lda;
  if ((rc = ctx->sc_df.ensure(2 * sizeof(float) * nc + 256))) return rc;
  if ((rc = ctx->sc_t1.ensure(2 * sizeof(float) * nt + 256))) return rc;
  if ((rc = ctx->sc_t2.ensure(sizeof(double) * (size_t)nvec * ND + 256))) return rc;
  float *Chi = (float *)ctx->sc_df.ptr, *Clo = Chi + nc, *Thi = (float *)ctx->sc_t1.ptr, *Tlo = Thi + nt;
  double *T2 = (double *)ctx->sc_t2.ptr;
  {
    FORTE_PROF(ctx, "df_split");
    k_df_split<<<(unsigned)std::min<size_t>((nc + 255) / 256, 152 * 16), 256, 0, st>>>(C, Chi, Clo, (long long)nvec * NA,
                                                                                      NB, ldb);
    FORTE_LAUNCH_CHECK();
  }
  if ((rc = ss_spmm_df(ctx, ctx->sd[0], (const float2 *)ctx->d_csr_val2[0], Chi, Clo, S, NA, NB, nvec))) return rc;
  {
    const dim3 tb(32, 8);
    const dim3 g1((unsigned)((NB + 31) / 32), (unsigned)((lda + 31) / 32), nvec);
    {
      FORTE_PROF(ctx, "transpose");
      k_df_split_t<<<g1, tb, 0, st>>>(C, Thi, Tlo, NA, NB, lda);
      FORTE_LAUNCH_CHECK();
    }
    if ((rc = ss_spmm_df(ctx, ctx->sd[1], (const float2 *)ctx->d_csr_val2[1], Thi, Tlo, T2, NB, NA, nvec))) return rc;
    const dim3 g2((unsigned)((NA + 31) / 32), (unsigned)((NB + 31) / 32), nvec);
    {
      FORTE_PROF(ctx, "transpose");
      k_transpose<double><<<g2, tb, 0, st>>>(T2, S, NB, NA, ND, 1);
      FORTE_LAUNCH_CHECK();
    }
  }
  if (with_ab && ctx->sh[0].nk > 0 && ctx->sh[ctx->same_strings ? 0 : 1].nk > 0) return ab_df(ctx, Chi, Clo, S, nvec);
  return FORTE_OK;
}

}  // namespace forte
