// One work item of the grouped FP64 GEMM: a tile of at most 64 x 64 outputs over a piece of
// K, computed by a 256-thread CTA on the FP64 units.
//
// The FP64 units bound it: GB300 issues about two FP64 FMAs a clock and SM, so a warp's FMA
// occupies the SM's pipe for 16 clocks and shared-memory reads, index arithmetic and L2
// traffic fit beside it even at one output a thread.  What costs time is FMAs spent on
// padding and SMs without work.  So:
//   * tiles are 64, 32 or 16 wide (plan_f64_tiles picks one per problem) and a tile's edge
//     is trimmed to 16 rows or columns: a thread owns rows ty + 16 r and columns tx + 16 c,
//     and the k loop is instantiated for every (rows, columns) = 1..4 x 1..4;
//   * K is one flat index over (k1, k0), so K0 = nvir leaves no idle tail in every k1, and
//     it can be cut at any multiple of 16;
//   * the next 16 K elements are loaded into registers while the current ones are
//     multiplied from one of two shared-memory buffers (one barrier per 16).
// Measured (energy, Gamma, P_ij, P_ab; fixed 64 x 64 tiles over whole P matrices before):
// nocc=10 nvir=40 naux=150 1042 -> 155 us, nocc=29 nvir=117 naux=437 19.7 -> 15.2 ms, 64
// monomers (nocc 8..20) 87.8 -> 50.0 ms; V at nocc=50 nvir=250 naux=750 runs at 1.24 TFLOP/s
// of issued FMAs, the rate of a register-only DFMA loop (1.25).
#pragma once

#include "rimp2_internal.cuh"

namespace rimp2 {

constexpr int F64_T = 64;    // widest tile
constexpr int F64_BK = 16;

struct F64Smem {
  double a[2][F64_BK][F64_T + 1];
  double b[2][F64_BK][F64_T + 1];
};

// Upper-triangle enumeration, column by column: t -> (r, c) with r <= c (the estimate in
// FP32, corrected in integers: FP64 square roots would cost more than they decide).
__device__ __forceinline__ void tri_index(long long t, int& r, int& c) {
  long long cc = (long long)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while (cc * (cc + 1) / 2 > t) --cc;
  while ((cc + 1) * (cc + 2) / 2 <= t) ++cc;
  c = (int)cc;
  r = (int)(t - cc * (cc + 1) / 2);
}

// Tile (tm, tn) and K piece ks of work item lt of a problem
__device__ __forceinline__ void f64_decode(const GemmProb& P, long long lt, int& tm, int& tn, int& ks) {
  ks = (int)(lt % P.ksplit);
  const long long tt = lt / P.ksplit;
  if (P.sym) tri_index(tt, tm, tn);
  else { tm = (int)(tt / P.tiles_n); tn = (int)(tt % P.tiles_n); }
}

// One operand's share of a 16-deep K block: R elements a thread, rows row0 + 16 q at one k.
// kc: K is the contiguous index, so lanes run along k; otherwise along the rows.
template <int R>
struct F64Operand {
  const double* p;
  long long srow, sk, s1;
  int row0, nrows, kk, K0;
  int k0;            // k = k1 * K0 + k0 of the thread's next element
  long long k1;
  __device__ __forceinline__ void init(const double* base, long long s_row, long long s_k,
                                       long long s_1, int first, int rows, int K0_, long long kbeg,
                                       int tid) {
    p = base; srow = s_row; sk = s_k; s1 = s_1; K0 = K0_; nrows = rows;
    const bool kc = s_k == 1;
    kk = kc ? (tid & 15) : (tid >> 4);
    row0 = kc ? (tid >> 4) : (tid & 15);
    p += (long long)first * srow;
    const long long k = kbeg + kk;
    k1 = K0 > 0 ? k / K0 : 0;
    k0 = (int)(k - k1 * K0);
  }
  // kleft: K elements left in the piece from this block's start
  __device__ __forceinline__ void load(double (&v)[R], long long kleft) {
    const bool in_k = kk < kleft;
    const double* q = p + (long long)k0 * sk + k1 * s1;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int row = row0 + 16 * r;
      v[r] = in_k && row < nrows ? q[(long long)row * srow] : 0.0;
    }
    k0 += F64_BK;
    while (k0 >= K0) { k0 -= K0; ++k1; }
  }
  __device__ __forceinline__ void store(const double (&v)[R], double (*s)[F64_T + 1]) const {
#pragma unroll
    for (int r = 0; r < R; ++r) s[kk][row0 + 16 * r] = v[r];
  }
};

template <int RR, int CC>
__device__ __forceinline__ void f64_tile(const GemmProb& P, const Bases& bs, int tm, int tn, int ks,
                                         F64Smem& sm) {
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int m0 = tm * P.bt, n0 = tn * P.bt;
  const double* __restrict__ A = P.kind == PK_GEN ? P.pa : (P.kind == PK_V ? bs.B : bs.ws) + P.a_off;
  const double* __restrict__ Bo = P.kind == PK_GEN ? P.pb : (P.b_from_B ? bs.B : bs.ws) + P.b_off;
  const long long kbeg = (long long)ks * P.k_chunk;
  long long kleft = min(P.k_total - kbeg, P.k_chunk);
  double acc[RR][CC];
#pragma unroll
  for (int r = 0; r < RR; ++r)
#pragma unroll
    for (int c = 0; c < CC; ++c) acc[r][c] = 0.0;

  if (kleft > 0) {
    F64Operand<RR> oa;
    F64Operand<CC> ob;
    oa.init(A, P.sAm, P.sAk, P.sA1, m0, P.M - m0, P.K0, kbeg, tid);
    ob.init(Bo, P.sBn, P.sBk, P.sB1, n0, P.N - n0, P.K0, kbeg, tid);
    double va[RR], vb[CC];
    oa.load(va, kleft);
    ob.load(vb, kleft);
    for (int buf = 0;; buf ^= 1) {
      oa.store(va, sm.a[buf]);
      ob.store(vb, sm.b[buf]);
      __syncthreads();
      kleft -= F64_BK;
      if (kleft > 0) {
        oa.load(va, kleft);
        ob.load(vb, kleft);
      }
#pragma unroll
      for (int kk = 0; kk < F64_BK; ++kk) {
        double a[RR], b[CC];
#pragma unroll
        for (int r = 0; r < RR; ++r) a[r] = sm.a[buf][kk][ty + 16 * r];
#pragma unroll
        for (int c = 0; c < CC; ++c) b[c] = sm.b[buf][kk][tx + 16 * c];
#pragma unroll
        for (int r = 0; r < RR; ++r)
#pragma unroll
          for (int c = 0; c < CC; ++c) acc[r][c] = fma(a[r], b[c], acc[r][c]);
      }
      if (kleft <= 0) break;
    }
  }

  if (P.kind == PK_V) {
    double* __restrict__ C = bs.ws + P.c_off;
    const double* eo = bs.eps + P.eo_off;
    const double* ev = bs.eps + P.ev_off;
    // D = (e_i - e_a) + (e_j - e_b): one FP64 addition an element
    double dn[CC];
#pragma unroll
    for (int c = 0; c < CC; ++c) {
      const int n = min(n0 + tx + 16 * c, P.N - 1), j = n / P.v;
      dn[c] = eo[j] - ev[n - j * P.v];
    }
#pragma unroll
    for (int r = 0; r < RR; ++r) {
      const int m = m0 + ty + 16 * r;
      if (m >= P.M) continue;
      const int i = m / P.v;
      const double dm = eo[i] - ev[m - i * P.v];
#pragma unroll
      for (int c = 0; c < CC; ++c) {
        const int n = n0 + tx + 16 * c;
        if (n >= P.N) continue;
        const double T = acc[r][c] / (dm + dn[c]);
        C[(long long)m * P.ldc + n] = T;
        if (tm != tn) C[(long long)n * P.ldc + m] = T;
      }
    }
    return;
  }
  double* __restrict__ C =
      P.kind == PK_GEN ? P.pc
                       : (P.kind == PK_GAMMA ? bs.gamma : P.kind == PK_PAB ? bs.pab : bs.pij) + P.c_off;
  const bool store = P.ksplit == 1 && (P.kind == PK_GAMMA || (P.kind == PK_GEN && !P.accumulate));
#pragma unroll
  for (int r = 0; r < RR; ++r) {
    const int m = m0 + ty + 16 * r;
    if (m >= P.M) continue;
#pragma unroll
    for (int c = 0; c < CC; ++c) {
      const int n = n0 + tx + 16 * c;
      if (n >= P.N) continue;
      const double val = P.alpha * acc[r][c];
      double* p = C + (long long)m * P.ldc + n;
      if (store) { *p = val; continue; }
      if (P.sym) {   // C = C^T: each unordered pair once, added at (m,n) and (n,m)
        if (m > n) continue;
        if (m < n) atomicAdd(C + (long long)n * P.ldc + m, val);
      }
      atomicAdd(p, val);
    }
  }
}

// Work item (tm, tn, ks) of problem P, by the whole CTA.  The caller separates two items by a
// barrier (the item's last reads of sm are not followed by one).
__device__ __forceinline__ void f64_item(const GemmProb& P, const Bases& bs, int tm, int tn, int ks,
                                         F64Smem& sm) {
  const int rr = (min(P.bt, P.M - tm * P.bt) + 15) >> 4, cc = (min(P.bt, P.N - tn * P.bt) + 15) >> 4;
  switch ((rr - 1) * 4 + cc - 1) {
#define RIMP2_F64_CASE(R, C) \
  case (R - 1) * 4 + C - 1: f64_tile<R, C>(P, bs, tm, tn, ks, sm); break;
#define RIMP2_F64_ROW(R) RIMP2_F64_CASE(R, 1) RIMP2_F64_CASE(R, 2) RIMP2_F64_CASE(R, 3) RIMP2_F64_CASE(R, 4)
    RIMP2_F64_ROW(1) RIMP2_F64_ROW(2) RIMP2_F64_ROW(3) RIMP2_F64_ROW(4)
#undef RIMP2_F64_ROW
#undef RIMP2_F64_CASE
    default: break;
  }
}

}  // namespace rimp2
