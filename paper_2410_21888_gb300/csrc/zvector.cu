// The step of the RI-MP2 gradient after the unrelaxed densities (Appendix), one fragment,
// FP64 (include/rimp2_grad.h):
//   Gamma^P = Gamma^Q J^{-1/2};  L'_iq = sum_aQ Gamma^Q_ia B^Q_qa;  L''_aq = sum_iQ Gamma^Q_ia B^Q_iq
//   and the Z-vector equation for D_ai by preconditioned conjugate gradients.
//
// With x[i][a] = D_ai, the operator of the Z-vector equation is
//   (A x)_ia = (e_a - e_i)/2 x_ia + 2 sum_Q B^Q_ia c^Q - sum_jQ B^Q_ja W^Q_ij,
//   c^Q = sum_jb B^Q_jb x_jb,  W^Q_ij = sum_b B^Q_ib x_jb,
// the Coulomb part 2 (ai|bj) and the exchange part (aj|bi) of G^{bj}_ai.  The right-hand
// side L''_ai - L'_ia - sum_pq G^{pq}_ai Dbar_pq expands the same way:
//   sum_kl G^{kl}_ai D_kl = 2 sum_Q B^Q_ia d^Q - sum_lQ B^Q_la U^Q_il,
//   sum_bc G^{bc}_ai D_bc = 2 sum_Q B^Q_ia e^Q - sum_cQ B^Q_ac V^Q_ic,
//   d^Q = sum_kl B^Q_kl D_kl, e^Q = sum_bc B^Q_bc D_bc, U^Q_il = sum_k B^Q_ik D_kl,
//   V^Q_ic = sum_b B^Q_ib D_bc.
// The contractions with a K of naux or more run on the grouped FP64 GEMM (PK_GEN problems
// on caller pointers); the sums over one index run as column or row sums; the whole
// conjugate-gradient solve is one cooperative kernel (k_cg).
#include <algorithm>
#include <atomic>
#include <cstring>
#include <vector>

#include <cuda_runtime.h>

#include "fp64_gemm.cuh"
#include "rimp2_grad.h"
#include "rimp2_testing.h"

namespace rimp2 {
namespace {

constexpr int kColRows = 16;      // rows per CTA of the column sums (at least)

size_t al256(size_t x) { return (x + 255) / 256 * 256; }

// out[Q] += sum_r w[r] M[r][Q] over the rows [rb, re) of r = (r1, r0) at base + r1 s1 + r0 s0,
// w[r1 * R0 + r0], for one Q; eight rows' loads in flight
__device__ __forceinline__ void colsum_rows(const double* base, long long s1, long long s0, int R0,
                                            const double* w, int Q, long long rb, long long re,
                                            double* out) {
  int a = (int)(rb / R0), b = (int)(rb - (long long)a * R0);
  double s = 0.0;
  for (long long r = rb; r < re; r += 8) {
    double m[8], f[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const bool in = r + k < re;
      m[k] = in ? base[a * s1 + b * s0 + Q] : 0.0;
      f[k] = in ? w[r + k] : 0.0;
      if (++b == R0) { b = 0; ++a; }
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) s = fma(f[k], m[k], s);
  }
  atomicAdd(out + Q, s);
}

__global__ void __launch_bounds__(256)
k_colsum(const double* base, long long s1, long long s0, int R1, int R0, const double* w, int X,
         int rows_per, double* out) {
  const int Q = blockIdx.x * blockDim.x + threadIdx.x;
  if (Q >= X) return;
  const long long R = (long long)R1 * R0, r0 = (long long)blockIdx.y * rows_per;
  colsum_rows(base, s1, s0, R0, w, Q, r0, min(R, r0 + rows_per), out);
}

// Warp sums over row (i,a) of the ov block of B: s1 = sum_Q B^Q_ia vec[Q] and, where asked for,
// s2 = sum_Q (B^Q_ia)^2
template <bool SQ>
__device__ __forceinline__ void row_sums(const double* Bf, int o, int n, int i, int a, int X,
                                         const double* vec, int lane, double& s1, double& s2) {
  const double* row = Bf + ((long long)i * n + o + a) * X;
  s1 = s2 = 0.0;
#pragma unroll 4
  for (int Q = lane; Q < X; Q += 32) {
    const double b = row[Q];
    s1 = fma(b, vec[Q], s1);
    if (SQ) s2 = fma(b, b, s2);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    s1 += __shfl_xor_sync(0xffffffffu, s1, off);
    if (SQ) s2 += __shfl_xor_sync(0xffffffffu, s2, off);
  }
}

// rhs[r] = L''_ai - L'_ia - 2 sum_Q B^Q_ia vec[Q] (vec = d + e); diag[r] = (e_a - e_i)/2 + sum_Q B^2
__global__ void __launch_bounds__(256)
k_rhs_rows(const double* Bf, const double* eps, int o, int v, int X, const double* vec,
           const double* lp, const double* lpp, double* rhs, double* diag) {
  const long long r = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31, n = o + v;
  if (r >= (long long)o * v) return;
  const int i = (int)(r / v), a = (int)(r - (long long)i * v);
  double s1, s2;
  row_sums<true>(Bf, o, n, i, a, X, vec, lane, s1, s2);
  if (lane != 0) return;
  rhs[r] = lpp[(long long)a * n + i] - lp[(long long)i * n + o + a] - 2.0 * s1;
  diag[r] = 0.5 * (eps[o + a] - eps[i]) + s2;
}

// ------------------------------------------------------------------ conjugate gradients
//
// The whole solve in one cooperative launch (every CTA resident, at most four per SM).  An
// iteration is bound by the FP64 work of its two exchange products (4 nocc^2 nvir naux
// FLOPs); as five launches an iteration, all max_iter of them enqueued, the launches after
// convergence (about 2 us each) and the single-CTA vector updates cost 3 of 9.7 ms at nocc=30
// nvir=120 naux=450, now 6.6 ms: 230 us an iteration, of which the products' FMAs take 170 and
// the uneven ends of phases A and B most of the rest.  Here an iteration is five phases separated by grid barriers:
//   A  W = B p by GEMM items and c = sum_jb B_jb p_jb by row blocks, from one work queue
//   B  Ap = (e_a - e_i)/2 p + 2 B c by blocks of rows - sum_jQ B W by GEMM items, added by
//      atomics into a zeroed Ap
//   C  p.Ap      D  x, r, ||r||, r.z      E  p, and c = Ap = 0 for the next product
// Dot products are summed per CTA and the CTAs' sums in a fixed order by every CTA, so all
// CTAs take the same decisions.

struct CgArgs {
  const GemmProb *pw, *px;        // phase A and B products
  int nw, nx;
  long long tw, tx;               // their work items
  const double *Bf, *eps, *rhs, *diag;
  double *x, *r, *p, *Ap, *c, *part, *info;
  int o, v, X, max_iter;
  double tol;
  unsigned* ctr;                  // two queue counters per iteration, zero
  unsigned long long* bar;        // barrier arrivals, zero
  unsigned* abort;                // zero; set when a barrier's wait expires
  unsigned long long limit_ns;
};

constexpr int kCgColRows = 32;    // rows per column-sum item (times 256 columns)
constexpr int kCgRows = 32;       // rows per row-sum item

// All CTAs of the grid; false when the wait expires (the caller leaves the kernel).
__device__ __forceinline__ bool grid_barrier(const CgArgs& A, unsigned long long& arrivals) {
  __shared__ int ok;
  __syncthreads();
  arrivals += gridDim.x;
  if (threadIdx.x == 0) {
    int good = 1;
    __threadfence();
    atomicAdd(A.bar, 1ull);
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    if (A.limit_ns == 0 && *(volatile unsigned long long*)A.bar < arrivals) {   // the test hook's
      atomicExch(A.abort, 1u);
      good = 0;
    }
    for (unsigned it = 1; good; ++it) {
      if (*(volatile unsigned long long*)A.bar >= arrivals) break;
      if ((it & 255u) == 0) {
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (*(volatile unsigned*)A.abort || t - t0 > A.limit_ns) {
          atomicExch(A.abort, 1u);
          good = 0;
          break;
        }
      }
    }
    __threadfence();
    ok = good;
  }
  __syncthreads();
  return ok != 0;
}

// The CTA's sums of (a, b) to part_a / part_b [blockIdx.x], in a fixed order.  has: whether
// the thread's warp holds any term (FP64 additions of idle warps would only load the unit).
__device__ __forceinline__ void cta_sums(double a, double b, bool has, double* part_a, double* part_b) {
  __shared__ double sh[2][8];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (__any_sync(0xffffffffu, has)) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, off);
      b += __shfl_xor_sync(0xffffffffu, b, off);
    }
  }
  __syncthreads();
  if (lane == 0) { sh[0][w] = a; sh[1][w] = b; }
  __syncthreads();
  if (threadIdx.x < 2) {
    double t = 0.0;
    for (int k = 0; k < 8; ++k) t += sh[threadIdx.x][k];
    (threadIdx.x ? part_b : part_a)[blockIdx.x] = t;
  }
}

// Sum over the CTAs of part[0..gridDim.x), in a fixed order, by one warp
__device__ __forceinline__ double grid_total(const double* part) {
  const int lane = threadIdx.x & 31;
  double t = 0.0;
#pragma unroll 4
  for (int k = lane; k < (int)gridDim.x; k += 32) t += part[k];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
  return t;
}

__global__ void __launch_bounds__(256, F64_CTAS) k_cg(CgArgs A) {
  __shared__ F64Smem sm;
  __shared__ F64Entry e;
  const long long N = (long long)A.o * A.v;
  // vector elements dealt to the CTAs one by one: the divisions of D and E then spread over
  // every SM's FP64 unit
  const long long first = blockIdx.x + (long long)gridDim.x * threadIdx.x, step = (long long)gridDim.x * 256;
  const int n = A.o + A.v, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int colx = (A.X + 255) / 256;
  const long long cols = (long long)colx * ((N + kCgColRows - 1) / kCgColRows);
  const long long rows = (N + kCgRows - 1) / kCgRows;
  // CTA sums: p.Ap (and a copy), then ||r||^2 and r.z
  double* const part = A.part;
  const int G = (int)gridDim.x;
  __shared__ double s_rz, s_bnorm, s_rnorm, s_alpha, s_beta;   // set by the first warp
  __shared__ int s_conv;
  unsigned long long arrivals = 0;
  Bases bs{};

  // x = 0, r = rhs, z = r / diag, p = z
  double rz = 0.0, rr = 0.0;
  for (long long k = first; k < N; k += step) {
    const double b = A.rhs[k], z = b / A.diag[k];
    A.x[k] = 0.0; A.r[k] = b; A.p[k] = z; A.Ap[k] = 0.0;
    rz = fma(b, z, rz);
    rr = fma(b, b, rr);
  }
  for (long long q = first; q < A.X; q += step) A.c[q] = 0.0;
  cta_sums(rr, rz, first < N, part + 2 * G, part + 3 * G);
  const bool alive = grid_barrier(A, arrivals);
  if (warp == 0) {
    rr = grid_total(part + 2 * G);
    rz = grid_total(part + 3 * G);
    if (lane == 0) {
      s_rz = rz;
      s_bnorm = s_rnorm = sqrt(rr);
      s_conv = alive && rr == 0.0;
    }
  }
  __syncthreads();
  int it = 0;
  while (alive && !s_conv && it < A.max_iter) {
    // A
    for (;;) {
      if (threadIdx.x < 32) f64_next(A.pw, A.nw, A.tw, A.ctr + 2 * it, e);
      __syncthreads();
      const long long t = e.t;
      if (t < A.tw) {
        f64_item<true>(e.P, bs, e.tm, e.tn, e.ks, sm);
      } else if (t - A.tw < cols) {
        const long long u = t - A.tw, rb = u / colx * kCgColRows;
        const int Q = (int)(u % colx) * 256 + threadIdx.x;
        if (Q < A.X)
          colsum_rows(A.Bf + (long long)A.o * A.X, (long long)n * A.X, A.X, A.v, A.p, Q, rb,
                      min(N, rb + kCgColRows), A.c);
      } else {
        break;
      }
      __syncthreads();
    }
    if (!grid_barrier(A, arrivals)) break;
    // B
    for (;;) {
      if (threadIdx.x < 32) f64_next(A.px, A.nx, A.tx, A.ctr + 2 * it + 1, e);
      __syncthreads();
      const long long t = e.t;
      if (t < A.tx) {
        f64_item<true>(e.P, bs, e.tm, e.tn, e.ks, sm);
      } else if (t - A.tx < rows) {
        const long long r1 = min(N, (t - A.tx + 1) * kCgRows);
        for (long long r = (t - A.tx) * kCgRows + warp; r < r1; r += 8) {
          const int i = (int)(r / A.v), a = (int)(r - (long long)i * A.v);
          double s1, s2;
          row_sums<false>(A.Bf, A.o, n, i, a, A.X, A.c, lane, s1, s2);
          if (lane == 0)
            atomicAdd(A.Ap + r, 0.5 * (A.eps[A.o + a] - A.eps[i]) * A.p[r] + 2.0 * s1);
        }
      } else {
        break;
      }
      __syncthreads();
    }
    if (!grid_barrier(A, arrivals)) break;
    // C: alpha = rz / p.Ap.  The scalars are computed by the first warp of every CTA: divisions
    // and square roots by all threads would cost 8 us an iteration on the FP64 units
    double pap = 0.0;
    for (long long k = first; k < N; k += step) pap = fma(A.p[k], A.Ap[k], pap);
    cta_sums(pap, 0.0, first < N, part, part + G);
    if (!grid_barrier(A, arrivals)) break;
    if (warp == 0) {
      pap = grid_total(part);
      if (lane == 0) {
        s_alpha = pap != 0.0 ? s_rz / pap : 0.0;
        s_conv = pap == 0.0;
      }
    }
    __syncthreads();
    // D: x += alpha p; r -= alpha Ap; z = r / diag
    rr = rz = 0.0;
    for (long long k = first; k < N; k += step) {
      const double alpha = s_alpha;
      A.x[k] = fma(alpha, A.p[k], A.x[k]);
      const double rk = fma(-alpha, A.Ap[k], A.r[k]);
      A.r[k] = rk;
      rr = fma(rk, rk, rr);
      rz = fma(rk, rk / A.diag[k], rz);
    }
    cta_sums(rr, rz, first < N, part + 2 * G, part + 3 * G);
    if (!grid_barrier(A, arrivals)) { if (threadIdx.x == 0) s_conv = 0; break; }
    if (warp == 0) {
      rr = grid_total(part + 2 * G);
      rz = grid_total(part + 3 * G);
      if (lane == 0) {
        s_rnorm = sqrt(rr);
        s_conv |= s_rnorm <= A.tol * s_bnorm;
        s_beta = rz / s_rz;
        s_rz = rz;
      }
    }
    __syncthreads();
    ++it;
    if (s_conv) break;
    // E: p = z + beta p
    for (long long k = first; k < N; k += step) {
      A.p[k] = fma(s_beta, A.p[k], A.r[k] / A.diag[k]);
      A.Ap[k] = 0.0;
    }
    for (long long q = first; q < A.X; q += step) A.c[q] = 0.0;
    if (!grid_barrier(A, arrivals)) break;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    // iterations = max_iter + 1 when the tolerance was not met, -1 when a barrier's wait expired
    A.info[0] = s_conv ? (double)it : *(volatile unsigned*)A.abort ? -1.0 : (double)(A.max_iter + 1);
    A.info[1] = s_bnorm > 0.0 ? s_rnorm / s_bnorm : 0.0;
    A.info[2] = s_bnorm;
  }
}

// C(m,n) = alpha sum_{k1,k0} A[m sAm + k0 sAk + k1 sA1] Bop[n sBn + k0 sBk + k1 sB1]
GemmProb gen(int M, int N, int K0, int K1, const double* a, long long sAm, long long sAk,
             long long sA1, const double* b, long long sBn, long long sBk, long long sB1,
             double* c, long long ldc, double alpha, bool accumulate) {
  GemmProb P{};
  P.kind = PK_GEN;
  P.M = M; P.N = N; P.K0 = K0; P.k_total = (long long)K0 * K1;
  P.pa = a; P.sAm = sAm; P.sAk = sAk; P.sA1 = sA1;
  P.pb = b; P.sBn = sBn; P.sBk = sBk; P.sB1 = sB1;
  P.pc = c; P.ldc = ldc; P.alpha = alpha;
  P.accumulate = accumulate ? 1 : 0;
  return P;
}

// part: the CTAs' sums of k_cg; zero .. zero_end: cleared at the start of every solve
struct Layout {
  size_t w, vv, r, p, ap, diag, rhs, c, part, zero, de, bar, ctr, zero_end, desc, total;
};

constexpr int kDescLists = 4;   // Gamma^P, L', L'', U, V; rhs terms; W; exchange product
constexpr size_t kDescBytes = 5 << 18;
constexpr int kPreCtr = 8;      // queue counters of the launches before k_cg
constexpr int kMaxCgGrid = 1024;

Layout layout(long long o, long long v, long long X, int max_iter) {
  Layout L{};
  size_t off = 0;
  const size_t ov = (size_t)(o * v);
  L.w = off; off += al256((size_t)(o * o * X) * 8);
  L.vv = off; off += al256((size_t)(o * v * X) * 8);
  L.r = off; off += al256(ov * 8);
  L.p = off; off += al256(ov * 8);
  L.ap = off; off += al256(ov * 8);
  L.diag = off; off += al256(ov * 8);
  L.rhs = off; off += al256(ov * 8);
  L.c = off; off += al256((size_t)X * 8);
  L.part = off; off += al256((size_t)4 * kMaxCgGrid * 8);
  L.zero = off;
  L.de = off; off += al256((size_t)X * 8);
  L.bar = off; off += 256;
  L.ctr = off; off += al256(((size_t)2 * max_iter + kPreCtr) * 4);
  L.zero_end = off;
  L.desc = off; off += kDescBytes;
  L.total = off;
  return L;
}

std::atomic<long long> g_wait_ns{-1};   // test hook: limit of k_cg's barriers (< 0: the normal one)

int iters_of(const rimp2_zvec_args* a) { return a->max_iter > 0 ? a->max_iter : 100; }

}  // namespace
}  // namespace rimp2

using namespace rimp2;

extern "C" {

int rimp2_testing_set_zvec_wait_limit(int64_t ns) {
  g_wait_ns.store(ns < 0 ? -1 : (long long)ns, std::memory_order_relaxed);
  return RIMP2_OK;
}

int rimp2_zvec_workspace_size(int32_t nocc, int32_t nvir, int32_t naux, int32_t max_iter,
                              size_t* bytes) {
  if (!bytes || nocc < 0 || nvir < 0 || naux < 0 || max_iter < 0) return RIMP2_ERR_BAD_ARG;
  *bytes = layout(nocc, nvir, naux, max_iter > 0 ? max_iter : 100).total;
  return RIMP2_OK;
}

int rimp2_zvec_solve(const rimp2_zvec_args* A, void* workspace, size_t ws_bytes,
                     cudaStream_t s) {
  if (!A || A->nocc < 0 || A->nvir < 0 || A->naux < 0 || A->max_iter < 0 || A->tol < 0)
    return RIMP2_ERR_BAD_ARG;
  const int o = A->nocc, v = A->nvir, X = A->naux, n = o + v;
  const long long ov = (long long)o * v;
  const long long X_ = X;
  // pointers are required where their arrays have elements
  if (!A->info || ((long long)o * n > 0 && !A->lp) || ((long long)v * n > 0 && !A->lpp) ||
      (ov > 0 && !A->dai) || (n > 0 && !A->eps) || ((long long)n * n * X_ > 0 && !A->Bf) ||
      (ov * X_ > 0 && !A->gamma) || (o > 0 && !A->pij) || (v > 0 && !A->pab))
    return RIMP2_ERR_BAD_ARG;
  const int max_iter = iters_of(A);
  const double tol = A->tol > 0 ? A->tol : 1e-12;
  const Layout L = layout(o, v, X, max_iter);
  if (!workspace || ((uintptr_t)workspace & 255u) || ws_bytes < L.total) return RIMP2_ERR_WORKSPACE;
  char* ws = (char*)workspace;
  double* W = (double*)(ws + L.w);
  double* Vv = (double*)(ws + L.vv);
  double* r = (double*)(ws + L.r);
  double* p = (double*)(ws + L.p);
  double* Ap = (double*)(ws + L.ap);
  double* diag = (double*)(ws + L.diag);
  double* rhs = (double*)(ws + L.rhs);
  double* c = (double*)(ws + L.c);
  double* de = (double*)(ws + L.de);
  unsigned* ctr = (unsigned*)(ws + L.ctr);
  cudaError_t e = cudaSuccess;
  auto ok = [&](cudaError_t x) { if (e == cudaSuccess) e = x; return e == cudaSuccess; };

  // outputs written by sums or accumulated
  if ((long long)o * n > 0) ok(cudaMemsetAsync(A->lp, 0, (size_t)o * n * 8, s));
  if ((long long)v * n > 0) ok(cudaMemsetAsync(A->lpp, 0, (size_t)v * n * 8, s));
  if (ov == 0) {
    ok(cudaMemsetAsync(A->info, 0, 3 * 8, s));
    return e == cudaSuccess ? RIMP2_OK : RIMP2_ERR_CUDA;
  }
  ok(cudaMemsetAsync(ws + L.zero, 0, L.zero_end - L.zero, s));

  const int grid = gemm_f64_occupancy_grid();
  const double* Bf = A->Bf;
  const long long nX = (long long)n * X, oX = (long long)o * X;
  std::vector<GemmProb> lists[kDescLists];
  // 0, one launch of independent products.
  // Gamma^P[(i,a)][P] = sum_Q Gamma[(i,a)][Q] J^{-1/2}[P][Q]
  if (A->jmh && A->gamma_p)
    lists[0].push_back(gen((int)ov, X, X, 1, A->gamma, X, 1, 0, A->jmh, X, 1, 0, A->gamma_p, X,
                           1.0, false));
  // L'[i][q] = sum_(a,Q) Gamma[i][a][Q] B[q][o+a][Q]; L''[a][q] = sum_(i,Q) Gamma[i][a][Q] B[i][q][Q]
  lists[0].push_back(gen(o, n, X, v, A->gamma, (long long)v * X, 1, X, Bf + oX, nX, 1, X, A->lp, n,
                         1.0, true));
  lists[0].push_back(gen(v, n, X, o, A->gamma, X, 1, (long long)v * X, Bf, X, 1, nX, A->lpp, n,
                         1.0, true));
  // U[i][l][Q] = sum_k D_kl B[i][k][Q];  V[i][c][Q] = sum_b D_bc B[i][o+b][Q]
  for (int i = 0; i < o; ++i) {
    lists[0].push_back(gen(o, X, o, 1, A->pij, o, 1, 0, Bf + (long long)i * nX, 1, X, 0,
                           W + (long long)i * oX, X, 1.0, false));
    lists[0].push_back(gen(v, X, v, 1, A->pab, v, 1, 0, Bf + (long long)i * nX + oX, 1, X, 0,
                           Vv + (long long)i * v * X, X, 1.0, false));
  }
  // 1: rhs[i][a] += sum_(l,Q) B[l][o+a][Q] U[i][l][Q] + sum_(c,Q) B[o+a][o+c][Q] V[i][c][Q]
  lists[1].push_back(gen(o, v, X, o, W, oX, 1, X, Bf + oX, X, 1, nX, rhs, v, 1.0, true));
  lists[1].push_back(gen(o, v, X, v, Vv, (long long)v * X, 1, X, Bf + (long long)o * nX + oX, nX, 1,
                         X, rhs, v, 1.0, true));
  // 2: W[i][j][Q] = sum_b p[j][b] B[i][o+b][Q]
  for (int i = 0; i < o; ++i)
    lists[2].push_back(gen(o, X, v, 1, p, v, 1, 0, Bf + (long long)i * nX + oX, 1, X, 0,
                           W + (long long)i * oX, X, 1.0, false));
  // 3: Ap[i][a] -= sum_(j,Q) B[j][o+a][Q] W[i][j][Q]
  lists[3].push_back(gen(o, v, X, o, W, oX, 1, X, Bf + oX, X, 1, nX, Ap, v, -1.0, true));

  std::vector<char> host;
  size_t doff[kDescLists];
  long long tiles[kDescLists];
  int grids[kDescLists];
  for (int k = 0; k < kDescLists; ++k) {
    grids[k] = plan_f64_tiles(lists[k], grid, F64_ITEMS_PER_SM, tiles[k]);
    doff[k] = host.size();
    const size_t bytes = lists[k].size() * sizeof(GemmProb);
    if (doff[k] + bytes > kDescBytes) return RIMP2_ERR_UNSUPPORTED;
    host.resize(al256(doff[k] + bytes), 0);
    if (bytes) memcpy(host.data() + doff[k], lists[k].data(), bytes);
  }
  char* desc = ws + L.desc;
  ok(cudaMemcpyAsync(desc, host.data(), std::min(host.size(), kDescBytes), cudaMemcpyHostToDevice, s));
  Bases bs{};
  auto gemm = [&](int k) {
    if (e != cudaSuccess || tiles[k] == 0) return;
    ok(launch_gemm_f64((const GemmProb*)(desc + doff[k]), (int)lists[k].size(), tiles[k], bs, ctr + k,
                       grids[k], s));
  };
  // d + e
  auto colsum = [&](const double* base, long long s1, long long s0, int R1, int R0,
                    const double* w, double* out) {
    const long long R = (long long)R1 * R0;
    if (e != cudaSuccess || X == 0 || R == 0) return;
    const long long per = std::max<long long>(kColRows, (R + 65534) / 65535);
    const dim3 g((unsigned)((X + 255) / 256), (unsigned)((R + per - 1) / per));
    k_colsum<<<g, 256, 0, s>>>(base, s1, s0, R1, R0, w, X, (int)per, out);
    ok(cudaGetLastError());
  };
  colsum(Bf, nX, X, o, o, A->pij, de);
  colsum(Bf + (long long)o * nX + oX, nX, X, v, v, A->pab, de);
  gemm(0);
  if (e == cudaSuccess) {
    k_rhs_rows<<<(unsigned)((ov + 7) / 8), 256, 0, s>>>(Bf, A->eps, o, v, X, de, A->lp, A->lpp, rhs, diag);
    ok(cudaGetLastError());
  }
  gemm(1);
  if (e != cudaSuccess) return RIMP2_ERR_CUDA;

  CgArgs C{};
  C.pw = (const GemmProb*)(desc + doff[2]); C.nw = (int)lists[2].size(); C.tw = tiles[2];
  C.px = (const GemmProb*)(desc + doff[3]); C.nx = (int)lists[3].size(); C.tx = tiles[3];
  C.Bf = Bf; C.eps = A->eps; C.rhs = rhs; C.diag = diag;
  C.x = A->dai; C.r = r; C.p = p; C.Ap = Ap; C.c = c;
  C.part = (double*)(ws + L.part); C.info = A->info;
  C.o = o; C.v = v; C.X = X; C.max_iter = max_iter; C.tol = tol;
  C.ctr = ctr + kPreCtr;
  C.bar = (unsigned long long*)(ws + L.bar);
  C.abort = (unsigned*)(ws + L.bar + 128);
  // a healthy barrier waits for a fraction of one exchange product's time
  const long long limit = g_wait_ns.load(std::memory_order_relaxed);
  C.limit_ns = limit >= 0 ? (unsigned long long)limit
                          : 2000000000ull + (unsigned long long)(2.0 * o * o * v * X * 4e-3);
  // every CTA resident (cooperative), and no more of them than the phases have items: a grid
  // barrier costs less with fewer
  int dev = 0, sms = 0, per = 0;
  if (!ok(cudaGetDevice(&dev)) || !ok(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) ||
      !ok(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_cg, 256, 0)))
    return RIMP2_ERR_CUDA;
  const long long items = std::max(tiles[2], tiles[3]) + (ov + kCgRows - 1) / kCgRows;
  const int g = (int)std::max(1LL, std::min<long long>(std::min(sms * std::max(per, 1), kMaxCgGrid), items));
  void* kargs[1] = {&C};
  ok(cudaLaunchCooperativeKernel((const void*)k_cg, dim3((unsigned)g), dim3(256), kargs, 0, s));
  return e == cudaSuccess ? RIMP2_OK : RIMP2_ERR_CUDA;
}

}  // extern "C"
