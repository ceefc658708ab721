// FP64 kernels of the RI-MP2 hot path: grouped persistent DFMA GEMM for the four
// contractions (Eq. MP2_ints for V; Appendix Gamma, D^MP2_ab, D^MP2_ij), the amplitude
// pass (T -> Tt = 2T - T^T and the pair energies), the compensated energy reduction,
// and input checks.  CUDA-core FP64 on sm_103a: the GEMM's work items (fp64_gemm.cuh) come
// from a device queue (an atomic counter) in the order the host sorted them (largest
// first).
#include <math.h>

#include <algorithm>

#include "energy.cuh"
#include "fp64_gemm.cuh"

namespace rimp2 {

template <typename F>
__device__ __forceinline__ int find_frag(const FragDev* __restrict__ frags, int nfrag,
                                         long long t, F key) {
  int lo = 0, hi = nfrag - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (key(frags[mid]) <= t) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// ------------------------------------------------------------------ grouped GEMM

__global__ void __launch_bounds__(256, F64_CTAS)
k_gemm_f64(const GemmProb* __restrict__ probs, int nprobs, long long total, Bases bs,
           unsigned* __restrict__ counter, int beside) {
  __shared__ F64Smem sm;
  __shared__ F64Entry e;
  for (;;) {
    if (threadIdx.x < 32) f64_next(probs, nprobs, total, counter, e);
    __syncthreads();
    if (e.t >= total) break;
    f64_item(e.P, bs, e.tm, e.tn, e.ks, sm);
    __syncthreads();  // the shared tile and descriptor are rewritten for the next item
  }
  if (beside) pdl_wait();
}

// Tile width, K pieces and queue position of every problem of one launch (sorted longest
// item first).  An item should hold about 1 / per_sm of an SM's share of the launch: large
// enough to amortise its start (queue, descriptor, first loads), small enough that the last
// items end together.  At nocc=10 nvir=40 naux=150 fixed 64 x 64 tiles put V on 28 of the
// 152 SMs and P_ij (10 x 10) into a tile with 1 / 41 of it filled: 1020 us for both GEMM
// launches.
int plan_f64_tiles(std::vector<GemmProb>& v, int grid, int per_sm, long long& total) {
  auto up16 = [](long long x) { return (x + 15) / 16 * 16; };
  auto work = [&](const GemmProb& P) {
    return (double)P.M * P.N * (double)std::max(1LL, P.k_total) * (P.sym ? 0.5 : 1.0);
  };
  double all = 0.0;
  for (const auto& P : v) all += work(P);
  const int sms = std::max(1, grid / F64_CTAS);
  const double unit = std::max(all / ((double)sms * per_sm), 1.0);
  // FMAs per K element of a symmetric problem with tiles of width bt: whole columns of tiles
  // above the diagonal (edges in 16s) and 8 x 8 blocks on it
  auto padded = [&](const GemmProb& P, int bt) {
    double s = 0.0;
    for (long long c = 0; c * bt < P.N; ++c) {
      const long long w = std::min<long long>(bt, P.N - c * bt), nb = (w + 7) / 8;
      s += (double)(c * bt) * (double)up16(w) + 64.0 * (double)(nb * (nb + 1) / 2);
    }
    return s;
  };
  for (auto& P : v) {
    const bool split = P.kind == PK_PAB || P.kind == PK_PIJ || (P.kind == PK_GEN && P.accumulate);
    // Gamma may be cut in two (P.accumulate: the caller zeroes it): 0 + x + y is the same in
    // either order, so the result stays reproducible
    const double K = (double)std::max(1LL, P.k_total);
    auto ext = [&](int bt, int n) { return (double)std::min<long long>(bt, up16(n)); };
    int bt = F64_T;
    if (split) {
      // K pieces give the balance; narrower tiles only where they save padding above the
      // diagonal or the pieces would get short
      if (P.sym)
        if (padded(P, bt) > 1.03 * padded(P, bt / 2)) bt /= 2;
      while (bt > 16 && unit / (ext(bt, P.M) * ext(bt, P.N)) < 256.0 && ext(bt, P.M) * ext(bt, P.N) > 256.0) bt /= 2;
      long long ch = up16((long long)(unit / (ext(bt, P.M) * ext(bt, P.N))) + 1);
      // P sums terms of one sign: bounded pieces also keep the rounding of their running
      // sums where it was (a single 45,000-long chain quadrupled P_ij's 1e-15 error)
      // At least 128 K elements amortise an item's start, or fewer where all pieces then still
      // run at once (a chain of 64 is half as long; 32 cost more in additions to C)
      const long long t = (P.M + bt - 1) / bt * (long long)((P.N + bt - 1) / bt);
      const long long once = up16(P.k_total * t / std::max(grid, 1) + 1);
      ch = std::max(ch, std::min<long long>(128, std::max<long long>(64, once)));
      ch = std::min<long long>(ch, 4096);
      P.k_chunk = std::min<long long>(ch, std::max<long long>(up16(P.k_total), 16));
    } else {
      while (bt > 16 && ext(bt, P.M) * ext(bt, P.N) * K > unit) bt /= 2;
      P.k_chunk = std::max<long long>(up16(P.k_total), 16);
      if (P.kind == PK_GAMMA) {
        P.accumulate = ext(bt, P.M) * ext(bt, P.N) * K > 4.0 * unit && P.k_total >= 128;
        if (P.accumulate) P.k_chunk = up16((P.k_total + 1) / 2);
      }
    }
    P.bt = bt;
    P.ksplit = (int)std::max<long long>(1, (P.k_total + P.k_chunk - 1) / P.k_chunk);
    P.tiles_m = (P.M + bt - 1) / bt;
    P.tiles_n = (P.N + bt - 1) / bt;
    P.ntiles = (P.sym ? (long long)P.tiles_m * (P.tiles_m + 1) / 2 : (long long)P.tiles_m * P.tiles_n) * P.ksplit;
  }
  auto cost = [&](const GemmProb& P) {
    return (double)std::min<long long>(P.bt, up16(P.M)) * (double)std::min<long long>(P.bt, up16(P.N)) *
           (double)std::min<long long>(P.k_chunk, std::max(1LL, P.k_total));
  };
  std::stable_sort(v.begin(), v.end(), [&](const GemmProb& a, const GemmProb& b) { return cost(a) > cost(b); });
  total = 0;
  for (auto& P : v) {
    P.tile_begin = total;
    total += P.ntiles;
  }
  // The CTAs of an SM share its FP64 unit, so short items taken beside a long one only delay
  // it: where the longest item is more than a quarter of an SM's share, fewer CTAs run
  // (Gamma and P at nocc=10 nvir=40 naux=150: 115 us with four, 78 with two)
  const double longest = v.empty() ? 0.0 : cost(v[0]), share = all / sms;
  const int ctas = longest * F64_CTAS <= share ? F64_CTAS : longest * 3 <= share ? 3 : 2;
  return sms * std::min(ctas, F64_CTAS);
}

int gemm_f64_occupancy_grid() {
  int dev = 0, sms = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_gemm_f64, 256, 0);
  if (per < 1) per = 1;
  return sms * per;
}

cudaError_t launch_gemm_f64(const GemmProb* d_probs, int nprobs, long long total_tiles,
                            Bases bs, unsigned* counter, int grid, cudaStream_t s, bool beside) {
  if (total_tiles <= 0) return cudaSuccess;
  const long long g = total_tiles < grid ? total_tiles : grid;
  return launch_pdl(k_gemm_f64, (unsigned)g, 256, 0, s, beside, d_probs, nprobs, total_tiles, bs, counter,
                    (int)beside);
}

// ------------------------------------------------------------------ amplitudes

__device__ __forceinline__ void put_pair(const FragDev& F, const Bases& bs, int a, int b, double e, double eos) {
  double* ep = bs.ws + F.ep_off;
  ep[(long long)a * F.o + b] = e;
  ep[(long long)b * F.o + a] = e;
  if (F.epos_off >= 0) {
    double* eq = bs.ws + F.epos_off;
    eq[(long long)a * F.o + b] = eos;
    eq[(long long)b * F.o + a] = eos;
  }
}

// The energies of a fragment, by one CTA of 256 threads, when its amplitude CTAs have ended:
// their shares of each pair energy (cut pairs) are added in a fixed order
__device__ __forceinline__ void sum_energies(const FragDev& F, const Bases& bs) {
  if (F.amp_split > 1) {
    const long long npair = (long long)F.o * (F.o + 1) / 2;
    for (long long p = threadIdx.x; p < npair; p += 256) {
      const double2* w = (const double2*)(bs.ws + F.part_off) + p * F.amp_split;
      double e = 0.0, eos = 0.0;
      for (int k = 0; k < F.amp_split; ++k) {
        const double2 x = __ldcg(w + k);
        e += x.x;
        eos += x.y;
      }
      int a, b;
      tri_index(p, a, b);
      put_pair(F, bs, a, b, e, eos);
    }
    __threadfence_block();
    __syncthreads();
  }
  fragment_energy(bs.ws + F.ep_off, F.epos_off >= 0 ? bs.ws + F.epos_off : nullptr, (long long)F.o * F.o,
                  F.epair_off >= 0 ? bs.epair + F.epair_off : nullptr, F.idx, bs);
}

// One CTA per pair block (i <= j) of one fragment and share of its 32 x 32 tile pairs.  Reads
// T_ij and writes Tt_ij = 2 T_ij - T_ij^T for the (i,j) block and, if i != j, Tt_ji = Tt_ij^T
// for the (j,i) block.  Pair energy e_ij = sum_ab Tt_ij(a,b) V_ij(a,b) with V = T * D, and its
// opposite-spin part sum_ab T_ij(a,b) V_ij(a,b).  FP64 operations bound it (a warp's takes the
// SM's pipe for 16 clocks): seven an element, and those of the sums, which are therefore long
// in a lane and short across lanes.  A wave of few pairs cuts them over several CTAs
// (amp_split; 55 pairs of nocc=10 nvir=40 on 55 SMs took 15 us).  Cut pairs of a narrow v are
// taken element by element: no idle lanes at tile edges, and the strided accesses of
// T_ij(b,a) and Tt_ji(b,a) stay in the lines of one block of at most 32 KB.  The energies are
// k_energy_reduce's: sums by the last CTA to finish cost every CTA a fence and the
// contractions their length (nocc=10 nvir=40 143 -> 137 us, nocc=100 nvir=20 2842 -> 2786).
__global__ void __launch_bounds__(256)
k_amplitude_f64(const FragDev* __restrict__ frags, int nfrag, Bases bs) {
  __shared__ double X[32][33];
  __shared__ double Y[32][33];
  __shared__ double red[2][256], sum[2];
  const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
  const int f = find_frag(frags, nfrag, (long long)blockIdx.x, [](const FragDev& F) { return F.cta_begin; });
  const FragDev F = frags[f];
  const long long lc = blockIdx.x - F.cta_begin, gp = lc / F.amp_split;
  const int share = (int)(lc - gp * F.amp_split);
  int i, j;
  tri_index(gp, i, j);
  const int v = F.v, o = F.o;
  const long long ov = (long long)o * v;
  const double* __restrict__ T = bs.ws + F.t_off;
  double* __restrict__ Tt = bs.ws + (F.tt_off >= 0 ? F.tt_off : 0);   // unused if < 0
  const double* eo = bs.eps + F.eo_off;
  const double* ev = bs.eps + F.ev_off;
  const double eij = eo[i] + eo[j];
  const long long rowI = (long long)i * v, rowJ = (long long)j * v;
  double e_part = 0.0, e_os = 0.0;
  const int nt = (v + 31) / 32;
  const long long ntp = (long long)nt * (nt + 1) / 2;
  const bool flat = amp_flat(F.amp_split, v);
  const long long q0 = ntp * share / F.amp_split, q1 = flat ? q0 : ntp * (share + 1) / F.amp_split;

  if (flat) {
    const int vv = v * v, end = vv * (share + 1) / F.amp_split;
    for (int e = vv * share / F.amp_split + tid; e < end; e += 256) {
      const int a = e / v, b = e - a * v;
      const double t = T[(rowI + a) * ov + rowJ + b];
      const double tt = 2.0 * t - T[(rowI + b) * ov + rowJ + a];
      if (F.tt_off >= 0) {
        Tt[(rowI + a) * ov + rowJ + b] = tt;
        if (i != j) Tt[(rowJ + b) * ov + rowI + a] = tt;
      }
      const double V = t * (eij - ev[a] - ev[b]);
      e_part += tt * V;
      e_os += t * V;
    }
  }
  for (long long q = q0; q < q1; ++q) {
    int ta, tb;
    tri_index(q, ta, tb);
    // X = T_ij[ta-rows][tb-cols], Y = T_ij[tb-rows][ta-cols]
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int l = ty + 8 * r;
      const int a = ta * 32 + l, b = tb * 32 + tx;
      X[l][tx] = (a < v && b < v) ? T[(rowI + a) * ov + rowJ + b] : 0.0;
      const int a2 = tb * 32 + l, b2 = ta * 32 + tx;
      Y[l][tx] = (a2 < v && b2 < v) ? T[(rowI + a2) * ov + rowJ + b2] : 0.0;
    }
    __syncthreads();
    // tile (ta, tb) of the (i,j) block: Tt(a,b) = 2 X[a][b] - Y[b][a]
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int l = ty + 8 * r;
      const int a = ta * 32 + l, b = tb * 32 + tx;
      if (a < v && b < v) {
        const double t = X[l][tx];
        const double tt = 2.0 * t - Y[tx][l];
        if (F.tt_off >= 0) Tt[(rowI + a) * ov + rowJ + b] = tt;
        const double D = eij - ev[a] - ev[b];
        e_part += tt * (t * D);
        e_os += t * (t * D);
      }
      if (ta != tb) {  // tile (tb, ta): Tt(a,b) = 2 Y[a][b] - X[b][a]
        const int a2 = tb * 32 + l, b2 = ta * 32 + tx;
        if (a2 < v && b2 < v) {
          const double t = Y[l][tx];
          const double tt = 2.0 * t - X[tx][l];
          if (F.tt_off >= 0) Tt[(rowI + a2) * ov + rowJ + b2] = tt;
          const double D = eij - ev[a2] - ev[b2];
          e_part += tt * (t * D);
          e_os += t * (t * D);
        }
      }
    }
    if (i != j && F.tt_off >= 0) {
      // (j,i) block: Tt_ji(a',b') = Tt_ij(b',a'); rows a' from tb, cols b' from ta
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int l = ty + 8 * r;
        const int ap = tb * 32 + l, bp = ta * 32 + tx;   // Tt_ij(bp, ap), bp in ta, ap in tb
        if (ap < v && bp < v)
          Tt[(rowJ + ap) * ov + rowI + bp] = 2.0 * X[tx][l] - Y[l][tx];
        if (ta != tb) {
          const int ap2 = ta * 32 + l, bp2 = tb * 32 + tx;  // Tt_ij(bp2, ap2), bp2 in tb
          if (ap2 < v && bp2 < v)
            Tt[(rowJ + ap2) * ov + rowI + bp2] = 2.0 * Y[tx][l] - X[l][tx];
        }
      }
    }
    __syncthreads();
  }
  // the CTA's share of the pair energy: eight values a lane, then across the lanes
  red[0][tid] = e_part;
  red[1][tid] = e_os;
  __syncthreads();
  if (ty < 2) {
    double x = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) x += red[ty][tx + 32 * w];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    if (tx == 0) sum[ty] = x;
  }
  __syncthreads();
  if (tid == 0) {
    if (F.amp_split == 1) put_pair(F, bs, i, j, sum[0], sum[1]);
    else ((double2*)(bs.ws + F.part_off))[gp * F.amp_split + share] = make_double2(sum[0], sum[1]);
  }
}

cudaError_t launch_amplitude_f64(const FragDev* d_frags, int nfrag, long long total_ctas, Bases bs,
                                 cudaStream_t s) {
  if (total_ctas <= 0) return cudaSuccess;
  k_amplitude_f64<<<(unsigned)total_ctas, 256, 0, s>>>(d_frags, nfrag, bs);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ energy reduction

// The energies, a CTA a fragment; the contractions that follow start beside it.
__global__ void __launch_bounds__(256)
k_energy_reduce(const FragDev* __restrict__ frags, Bases bs) {
  pdl_trigger();
  sum_energies(frags[blockIdx.x], bs);
}

cudaError_t launch_energy_reduce(const FragDev* d_frags, int nfrag, Bases bs, cudaStream_t s) {
  if (nfrag <= 0) return cudaSuccess;
  k_energy_reduce<<<nfrag, 256, 0, s>>>(d_frags, bs);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ prologue and input checks

// What a call's first launch prepares: the wave's queue counters (ctr, eight; may be null), zero
// P (and Gamma where it is accumulated).  check: denominators must be negative for every (i,j,a,b), i.e.
// max(eps_occ) < min(eps_vir); B and eps must be finite.  Violations set bits of the status
// word.  (Seven launches a call of nocc=10 nvir=40 had three of these few microseconds each.)
__global__ void __launch_bounds__(256)
k_prologue(const FragDev* __restrict__ frags, unsigned* ctr, int check, Bases bs) {
  const FragDev F = frags[blockIdx.y];
  const long long first = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long stride = (long long)gridDim.x * blockDim.x;
  if (ctr && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < 8) ctr[threadIdx.x] = 0u;
  if (F.pij_off >= 0)
    for (long long e = first; e < (long long)F.o * F.o; e += stride) bs.pij[F.pij_off + e] = 0.0;
  if (F.pab_off >= 0)
    for (long long e = first; e < (long long)F.v * F.v; e += stride) bs.pab[F.pab_off + e] = 0.0;
  if (F.zero_gamma)
    for (long long e = first; e < (long long)F.o * F.v * F.X; e += stride) bs.gamma[F.gamma_off + e] = 0.0;
  if (!check) return;
  bool bad_nf = false;
  const long long nb = (long long)F.o * F.v * F.X;
  const double* B = bs.B + F.b_off;
  for (long long e = first; e < nb; e += stride)
    bad_nf |= !finite_bits(B[e]);
  if (blockIdx.x == 0) {
    __shared__ double smax[256], smin[256];
    double mx = -INFINITY, mn = INFINITY;
    for (int e = threadIdx.x; e < F.o; e += blockDim.x) {
      const double x = bs.eps[F.eo_off + e];
      bad_nf |= !isfinite(x);
      mx = fmax(mx, x);
    }
    for (int e = threadIdx.x; e < F.v; e += blockDim.x) {
      const double x = bs.eps[F.ev_off + e];
      bad_nf |= !isfinite(x);
      mn = fmin(mn, x);
    }
    smax[threadIdx.x] = mx;
    smin[threadIdx.x] = mn;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
      if ((int)threadIdx.x < w) {
        smax[threadIdx.x] = fmax(smax[threadIdx.x], smax[threadIdx.x + w]);
        smin[threadIdx.x] = fmin(smin[threadIdx.x], smin[threadIdx.x + w]);
      }
      __syncthreads();
    }
    if (threadIdx.x == 0 && F.o > 0 && F.v > 0 && !(smax[0] < smin[0]))
      atomicOr(bs.status, ST_DENOM);
  }
  if (bad_nf) atomicOr(bs.status, ST_NONFINITE);
}

cudaError_t launch_prologue(const FragDev* d_frags, int nfrag, long long max_bx, unsigned* ctr, int check,
                            Bases bs, cudaStream_t s) {
  if (nfrag <= 0) return cudaSuccess;
  const unsigned bx = (unsigned)(max_bx < 1 ? 1 : (max_bx > 256 ? 256 : max_bx));
  k_prologue<<<dim3(bx, nfrag), 256, 0, s>>>(d_frags, ctr, check, bs);
  return cudaGetLastError();
}

}  // namespace rimp2
