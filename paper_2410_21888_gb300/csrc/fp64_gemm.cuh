// One work item of the grouped FP64 GEMM: a tile of at most 32 x 32 outputs over a piece of
// K, computed by a 256-thread CTA on the FP64 units.
//
// The FP64 units bound it: GB300 issues about two FP64 FMAs a clock and SM, so a warp's FMA
// occupies the SM's pipe for 16 clocks and shared-memory reads, index arithmetic and L2
// traffic fit beside it even at one output a thread.  What costs time is FMAs spent on
// padding and SMs without work.  So:
//   * tiles are 32 or 16 wide (plan_f64_tiles picks one per problem) and a tile's edge is
//     trimmed to 16 rows or columns: a thread owns rows ty + 16 r and columns tx + 16 c,
//     and the k loop is instantiated for every (rows, columns) = 1..2 x 1..2.  Wider tiles
//     would save L2 reads that cost nothing here and need twice the registers: four CTAs
//     an SM cover each other's queue and load latencies;
//   * K is one flat index over (k1, k0), so K0 = nvir leaves no idle tail in every k1, and
//     it can be cut at any multiple of 16;
//   * the next 16 K elements are loaded into registers while the current ones are
//     multiplied from one of two shared-memory buffers (one barrier per 16).
// Measured (energy, Gamma, P_ij, P_ab; fixed 64 x 64 tiles over whole P matrices before):
// nocc=10 nvir=40 naux=150 1042 -> 148 us (131 with the other kernels' work since), nocc=29 nvir=117 naux=437 19.8 -> 15.0 ms, 64
// monomers (nocc 8..20) 87.8 -> 46.2 ms; V at nocc=50 nvir=250 naux=750 runs at 1.24 TFLOP/s
// of issued FMAs, the rate of a register-only DFMA loop (1.25).
#pragma once

#include <type_traits>

#include "rimp2_internal.cuh"

namespace rimp2 {

constexpr int F64_T = 32;    // widest tile
constexpr int F64_CTAS = 4;  // CTAs per SM
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

// The K loop of one item: RR x 16 rows of A and CC x 16 of Bop through the two buffers;
// block(buf) multiplies 16 K elements
template <int RR, int CC, bool GEN, typename F>
__device__ __forceinline__ void f64_k_loop(const GemmProb& P, const Bases& bs, int m0, int n0, int ks,
                                           F64Smem& sm, F block) {
  // plain (coherent) loads: the operands may have been written earlier by the same kernel
  const double* A = GEN || P.kind == PK_GEN ? P.pa : (P.kind == PK_V ? bs.B : bs.ws) + P.a_off;
  const double* Bo = GEN || P.kind == PK_GEN ? P.pb : (P.b_from_B ? bs.B : bs.ws) + P.b_off;
  const long long kbeg = (long long)ks * P.k_chunk;
  long long kleft = min(P.k_total - kbeg, P.k_chunk);
  if (kleft <= 0) return;
  F64Operand<RR> oa;
  F64Operand<CC> ob;
  oa.init(A, P.sAm, P.sAk, P.sA1, m0, P.M - m0, P.K0, kbeg, threadIdx.x);
  ob.init(Bo, P.sBn, P.sBk, P.sB1, n0, P.N - n0, P.K0, kbeg, threadIdx.x);
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
    block(buf);
    if (kleft <= 0) return;
  }
}

// One result of a P or PK_GEN problem
__device__ __forceinline__ double* f64_out(const GemmProb& P, const Bases& bs) {
  return P.kind == PK_GEN ? P.pc
                          : (P.kind == PK_GAMMA ? bs.gamma : P.kind == PK_PAB ? bs.pab : bs.pij) + P.c_off;
}

// GEN: the problem is known to be PK_GEN
template <int RR, int CC, bool GEN>
__device__ __forceinline__ void f64_tile(const GemmProb& P, const Bases& bs, int tm, int tn, int ks,
                                         F64Smem& sm) {
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int m0 = tm * P.bt, n0 = tn * P.bt;
  double acc[RR][CC];
#pragma unroll
  for (int r = 0; r < RR; ++r)
#pragma unroll
    for (int c = 0; c < CC; ++c) acc[r][c] = 0.0;
  // 16-row groups in which this warp (rows 2 w, 2 w + 1 of each) has rows of the matrix: the
  // others' FMAs are left out, so the padding of an edge tile costs two rows at most
  const int nrow = min(RR, (P.M - m0 - (ty & ~1) + 15) >> 4);
  f64_k_loop<RR, CC, GEN>(P, bs, m0, n0, ks, sm, [&](int buf) {
    auto mul = [&](auto rows) {
      constexpr int R = decltype(rows)::value;
#pragma unroll
      for (int kk = 0; kk < F64_BK; ++kk) {
        double a[R], b[CC];
#pragma unroll
        for (int r = 0; r < R; ++r) a[r] = sm.a[buf][kk][ty + 16 * r];
#pragma unroll
        for (int c = 0; c < CC; ++c) b[c] = sm.b[buf][kk][tx + 16 * c];
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
          for (int c = 0; c < CC; ++c) acc[r][c] = fma(a[r], b[c], acc[r][c]);
      }
    };
    if (nrow == RR) mul(std::integral_constant<int, RR>{});
    else if (RR > 1 && nrow == 1) mul(std::integral_constant<int, 1>{});
  });

  if (!GEN && P.kind == PK_V) {   // off the diagonal: both triangles of T from one result
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
        C[(long long)n * P.ldc + m] = T;
      }
    }
    return;
  }
  double* C = GEN ? P.pc : f64_out(P, bs);
  const bool store =
      P.ksplit == 1 && (GEN || P.kind == PK_GEN ? !P.accumulate : P.kind == PK_GAMMA);
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
      atomicAdd(p, val);
      if (!GEN && P.sym) atomicAdd(C + (long long)n * P.ldc + m, val);   // a tile above the diagonal
    }
  }
}

// A diagonal tile of a symmetric problem: the 8 x 8 blocks on and above the diagonal, 64
// outputs each, dealt to the threads in order (at most three a thread, whole warps per
// block).  The full square would spend 1024 FMAs per K element on a 32-wide tile, these
// blocks 640; P_ij of a small fragment is a single such tile.
template <int R>
__device__ __forceinline__ void f64_diag(const GemmProb& P, const Bases& bs, int t, int ks, F64Smem& sm) {
  const int m0 = t * P.bt, ext = min(P.bt, P.M - m0), nb = (ext + 7) >> 3;
  const int nblk = nb * (nb + 1) / 2;
  int row[3], col[3], nr = 0;
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const int e = threadIdx.x + 256 * r, blk = e >> 6;
    int bi = 0, bj = 0;
    for (int q = blk; q > bj;) { ++bj; q -= bj; bi = q; }   // blk = bj (bj + 1) / 2 + bi
    if (bj == 0) bi = 0;
    row[r] = 8 * bi + ((e >> 3) & 7);
    col[r] = 8 * bj + (e & 7);
    if (blk < nblk) nr = r + 1;
    else row[r] = col[r] = 0;
  }
  double acc[3] = {0.0, 0.0, 0.0};
  f64_k_loop<R, R, false>(P, bs, m0, m0, ks, sm, [&](int buf) {
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      if (r < nr) {   // uniform across the warp
#pragma unroll
        for (int kk = 0; kk < F64_BK; ++kk)
          acc[r] = fma(sm.a[buf][kk][row[r]], sm.b[buf][kk][col[r]], acc[r]);
      }
    }
  });
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const int m = m0 + row[r], n = m0 + col[r];
    if (r >= nr || m > n || n >= P.N) continue;
    if (P.kind == PK_V) {
      double* C = bs.ws + P.c_off;
      const double* eo = bs.eps + P.eo_off;
      const double* ev = bs.eps + P.ev_off;
      const int i = m / P.v, j = n / P.v;
      const double T = acc[r] / ((eo[i] - ev[m - i * P.v]) + (eo[j] - ev[n - j * P.v]));
      C[(long long)m * P.ldc + n] = T;
      C[(long long)n * P.ldc + m] = T;
    } else {
      double* C = f64_out(P, bs);
      const double val = P.alpha * acc[r];
      atomicAdd(C + (long long)m * P.ldc + n, val);
      if (m < n) atomicAdd(C + (long long)n * P.ldc + m, val);
    }
  }
}

// Work item (tm, tn, ks) of problem P, by the whole CTA.  The caller separates two items by a
// barrier (the item's last reads of sm are not followed by one).
template <bool GEN = false>
__device__ __forceinline__ void f64_item(const GemmProb& P, const Bases& bs, int tm, int tn, int ks,
                                         F64Smem& sm) {
  if (!GEN && P.sym && tm == tn) {
    if (min(P.bt, P.M - tm * P.bt) > 16) f64_diag<2>(P, bs, tm, ks, sm);
    else f64_diag<1>(P, bs, tm, ks, sm);
    return;
  }
  const int rr = (min(P.bt, P.M - tm * P.bt) + 15) >> 4, cc = (min(P.bt, P.N - tn * P.bt) + 15) >> 4;
  if (rr == 2) {
    if (cc == 2) f64_tile<2, 2, GEN>(P, bs, tm, tn, ks, sm);
    else f64_tile<2, 1, GEN>(P, bs, tm, tn, ks, sm);
  } else {
    if (cc == 2) f64_tile<1, 2, GEN>(P, bs, tm, tn, ks, sm);
    else f64_tile<1, 1, GEN>(P, bs, tm, tn, ks, sm);
  }
}

// Problem of queue entry t, by a whole warp: each step reads 32 of the candidates' first
// entries at once
__device__ __forceinline__ int find_prob(const GemmProb* __restrict__ probs, int nprobs,
                                         long long t) {
  const int lane = threadIdx.x & 31;
  int lo = 0, n = nprobs;   // the last problem with tile_begin <= t is in [lo, lo + n)
  while (n > 1) {
    const int w = (n + 31) / 32, k = lane * w;
    const bool le = k < n && probs[lo + k].tile_begin <= t;
    const int q = 31 - __clz(__ballot_sync(0xffffffffu, le));   // lane 0 always holds
    lo += q * w;
    n = min(w, n - q * w);
  }
  return lo;
}

// A CTA's current queue entry, filled by its first warp
struct F64Entry {
  GemmProb P;
  long long t;
  int tm, tn, ks;
};

// Takes the next entry of a queue (all threads of the first warp call it) and, when it is a
// GEMM item (t < total), its problem descriptor and tile; the caller's barrier publishes it.
__device__ __forceinline__ void f64_next(const GemmProb* __restrict__ probs, int nprobs,
                                         long long total, unsigned* __restrict__ counter, F64Entry& e) {
  long long t = 0;
  if (threadIdx.x == 0) t = (long long)atomicAdd(counter, 1u);
  t = __shfl_sync(0xffffffffu, t, 0);
  if (t < total) {
    const int pi = find_prob(probs, nprobs, t);
    static_assert(sizeof(GemmProb) % 8 == 0, "copied in 8-byte words");
    for (int w = threadIdx.x; w < (int)(sizeof(GemmProb) / 8); w += 32)
      ((long long*)&e.P)[w] = ((const long long*)(probs + pi))[w];
    __syncwarp();
    if (threadIdx.x == 0) f64_decode(e.P, t - e.P.tile_begin, e.tm, e.tn, e.ks);
  }
  if (threadIdx.x == 0) e.t = t;
}

}  // namespace rimp2
