// Split-precision path of the RI-MP2 hot path (precision RIMP2_BF16_SPLIT).
//
// Per wave of fragments:
//   1. k_split_prologue  counters and maxima slots, check of the orbital energies
//   2. k_slice_b1        B -> balanced base-512 digits with one scale per row (i,a): the
//                        operands of V (Eq. MP2_ints); d_m = e_i - e_a per row, check of B;
//                        other CTAs of the launch: max over (j,b) of |B^Q_jb| per aux index Q
//   3. split GEMM        V on the tensor cores, epilogue T = V / D kept as a double-float
//                        pair of planes, max |T| exponent
//   4. k_amp_split       Tt = 2T - T^T, digits of Tt and T with one scale per fragment, pair
//                        energies e_ij and the FP64 compensated cross-pair sums, zeroes P;
//                        other CTAs of the launch: B -> digits with one scale per aux index
//                        Q, transposed to [Q][(j,b)], the B operand of Gamma
//   5. split GEMMs for P_ab and P_ij (128 x 64 tiles, or slice-stacked for small extents),
//      then for Gamma (Appendix Gamma, D^MP2_ab, D^MP2_ij); Gamma contracts the leading s_g
//      digit planes of Tt
#include <climits>
#include <cmath>
#include <cstring>
#include <algorithm>

#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "energy.cuh"
#include "split_path.cuh"

namespace rimp2 {

namespace {

size_t al256(size_t x) { return (x + 255) / 256 * 256; }

// V tiles are walked in groups of this many rows (tile order, see decode_tile)
constexpr int kVGroupRows = 16;
// smallest K extent of a split-K piece of P_ab / P_ij
constexpr long long kMinPieceK = 4096;
// K extent of one Gamma slab (elements of the contracted (j,b) index).  Measured at
// nocc=100 nvir=500 naux=1500 (K = 51200): the Gamma/P launch takes 144.7 ms with slabs
// of 2048, 140.5 with 4096, 138.0 with 8192, 136.5 with 16384 and 138.5 without slabs.
constexpr long long kGammaSlabK = 16384;
// rows of B per CTA of the column maxima (eight loads in flight a lane)
constexpr int kColRows = 256;
int rup(int x, int m) { return (x + m - 1) / m * m; }

}  // namespace

// ------------------------------------------------------------------ device helpers

struct dfl { float h, l; };

__device__ __forceinline__ dfl d_two_sum(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  return {s, (a - (s - bb)) + (b - bb)};
}
__device__ __forceinline__ dfl d_fast(float a, float b) {
  const float s = a + b;
  return {s, b - (s - a)};
}
__device__ __forceinline__ dfl d_add(dfl a, dfl b) {
  dfl s = d_two_sum(a.h, b.h);
  s.l += a.l + b.l;
  return d_fast(s.h, s.l);
}
// (split on the integer pipes: a conversion occupies the SM's FP64 unit for 16 clocks a warp,
// however few lanes need it)
__device__ __forceinline__ dfl d_from(double x) {
  dfl d;
  split_to_df(x, d.h, d.l);
  return d;
}

__device__ __forceinline__ int find_sfd(const SplitFragDev* __restrict__ f, int n, long long t,
                                        int which) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    const long long k = which == 0 ? f[mid].row_begin : which == 1 ? f[mid].b2_tile_begin
                        : which == 2 ? f[mid].pair_begin : f[mid].qblk_begin;
    if (k <= t) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// One digit (an integer in [-2^(LB-1), 2^(LB-1)]) in the slice format: BF16 (LB = 9:
// its 8-bit significand holds every integer up to 256) or FP8 e4m3 (LB = 5); both
// represent these integers exactly.  The leading digit is HEAD bits narrower: a value x
// is sliced relative to 2^E with |x| <= 2^(E-1-HEAD) (BF16: d_0 in [-64, 64], which keeps
// the level-1 sums of a 512-long chunk within 2^24).
template <bool F8> struct Digit;
template <> struct Digit<false> {
  using T = __nv_bfloat16;
  static constexpr int LB = SG_LB_BF16;
  static constexpr int HEAD = SG_HEAD_BF16;
  __device__ static T enc(float d) { return __float2bfloat16_rn(d); }
};
template <> struct Digit<true> {
  using T = unsigned char;
  static constexpr int LB = SG_LB_FP8;
  static constexpr int HEAD = SG_HEAD_FP8;
  __device__ static T enc(float d) {
    return (T)__nv_cvt_float_to_fp8(d, __NV_SATFINITE, __NV_E4M3);
  }
};

// Four digits of one slice, packed for one store: BF16 digits are exact integers, so their
// bit patterns are the upper halves of the FP32 values; FP8 digits go through the e4m3
// conversion.
template <bool F8> struct Pack4;
template <> struct Pack4<false> {
  using T = uint2;
  __device__ static T pack(float d0, float d1, float d2, float d3) {
    return make_uint2(__byte_perm(__float_as_uint(d0), __float_as_uint(d1), 0x7632),
                      __byte_perm(__float_as_uint(d2), __float_as_uint(d3), 0x7632));
  }
};
template <> struct Pack4<true> {
  using T = uint32_t;
  __device__ static T pack(float d0, float d1, float d2, float d3) {
    return (uint32_t)Digit<true>::enc(d0) | ((uint32_t)Digit<true>::enc(d1) << 8) |
           ((uint32_t)Digit<true>::enc(d2) << 16) | ((uint32_t)Digit<true>::enc(d3) << 24);
  }
};

// One digit step of a normalised double-float (|xl| <= ulp(xh)/2) relative to the current
// scale: d = rint(xh) by the 1.5 * 2^23 shift (round to nearest even, |xh| <= 2^22);
// xh - d is exact and, when non-zero, a multiple of ulp(xh) >= 2|xl|, so Fast2Sum re-joins
// it with xl exactly; the remainder is scaled by 2^LB for the next digit.
template <int LB>
__device__ __forceinline__ float digit_step(float& xh, float& xl) {
  const float kShift = 12582912.f;
  const float d = __fsub_rn(__fadd_rn(xh, kShift), kShift);
  const float a = __fsub_rn(xh, d);
  const float s = __fadd_rn(a, xl);
  const float e = __fsub_rn(xl, __fsub_rn(s, a));
  xh = s * (float)(1 << LB);
  xl = e * (float)(1 << LB);
  return d;
}

// Two FP32 lanes in one 64-bit register for the packed f32x2 arithmetic of sm_100+
// (add/sub/mul.rn.f32x2: each lane rounds exactly like the scalar instruction).
typedef unsigned long long f2x;
__device__ __forceinline__ f2x f2_pack(float a, float b) {
  f2x r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f2_unpack(f2x r, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ f2x f2_add(f2x a, f2x b) {
  f2x d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2x f2_sub(f2x a, f2x b) {
  f2x d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2x f2_mul(f2x a, f2x b) {
  f2x d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

__device__ __forceinline__ f2x f2_fma(f2x a, f2x b, f2x c) {
  f2x d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

__device__ __forceinline__ f2x f2_neg(f2x a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ f2x f2_two(float a) { return f2_pack(a, a); }
// Double-float arithmetic on two lanes (the f32x2 forms round each lane like the scalar
// instruction and are never contracted).  s + e = a + b exactly:
__device__ __forceinline__ void f2_two_sum(f2x a, f2x b, f2x& s, f2x& e) {
  s = f2_add(a, b);
  const f2x bb = f2_sub(s, a);
  e = f2_add(f2_sub(a, f2_sub(s, bb)), f2_sub(b, bb));
}
// a - b, normalised
__device__ __forceinline__ void d_sub2(f2x ah, f2x al, f2x bh, f2x bl, f2x& h, f2x& l) {
  const f2x s = f2_sub(ah, bh);
  const f2x bb = f2_sub(ah, s);                                     // b as seen in s
  const f2x e = f2_add(f2_sub(bb, bh), f2_sub(ah, f2_add(s, bb)));   // two-difference
  const f2x t = f2_add(e, f2_sub(al, bl));
  h = f2_add(s, t);
  l = f2_sub(t, f2_sub(h, s));
}
// a b as h + l with |l| of the order of an ulp of h (not normalised); na = -ah.  al bl is
// kept: without normalisation the low part of V = T D still holds T's, and the square of it
// in every T V has one sign (E_os of 4 MBE3 trimers -6.0e-16 relative without it, on average)
__device__ __forceinline__ void d_mul2(f2x ah, f2x na, f2x al, f2x bh, f2x bl, f2x& h, f2x& l) {
  h = f2_mul(ah, bh);
  const f2x ne = f2_fma(na, bh, h);                                 // h - ah bh, exact
  l = f2_sub(f2_fma(ah, bl, f2_fma(al, bl, f2_mul(al, bh))), ne);
}
// sum (sh, sl) += (h, l): sh takes h without error, sl collects the errors and the low parts
__device__ __forceinline__ void d_acc2(f2x& sh, f2x& sl, f2x h, f2x l) {
  f2x e;
  f2_two_sum(sh, h, sh, e);
  sl = f2_add(sl, f2_add(e, l));
}

// digit_step on two elements at once, with the scaling by 2^LB folded into the Fast2Sum
// (seven packed operations instead of eight, bit-identical): with a = xh - d and
// s = a + xl as in digit_step, 2^LB s = RN(2^LB a + 2^LB xl) is one FMA; 2^LB (s - a) is
// exact, so the FMA 2^LB s - 2^LB a returns it unrounded, and 2^LB xl minus it is the
// exact error term 2^LB e
template <int LB>
__device__ __forceinline__ f2x digit_step2(f2x& xh, f2x& xl) {
  const f2x kShift = f2_pack(12582912.f, 12582912.f);
  const f2x kScale = f2_pack((float)(1 << LB), (float)(1 << LB));
  const f2x kNegScale = f2_pack(-(float)(1 << LB), -(float)(1 << LB));
  const f2x d = f2_sub(f2_add(xh, kShift), kShift);
  const f2x a = f2_sub(xh, d);
  const f2x l = f2_mul(xl, kScale);
  xh = f2_fma(a, kScale, l);
  xl = f2_sub(l, f2_fma(a, kNegScale, xh));
  return d;
}

// Digits of four consecutive elements (double-floats in element pairs, already scaled to the
// slice frame), one packed store per slice plane; the digit steps run on element pairs.  NS > 0:
// the plane count is NS, known at compile time (the loop unrolls; st is not read).
// STREAM: the stores carry the evict-first hint (the amplitude kernel's digit planes are
// far larger than L2 and are read back by later launches only).
template <bool F8, int NS = 0, bool STREAM = false>
__device__ __forceinline__ void put4(f2x h01, f2x l01, f2x h23, f2x l23, int st,
                                     typename Digit<F8>::T* out, long long plane) {
  constexpr int LB = Digit<F8>::LB;
  using PT = typename Pack4<F8>::T;
  auto one = [&](int p) {
    float d0, d1, d2, d3;
    f2_unpack(digit_step2<LB>(h01, l01), d0, d1);
    f2_unpack(digit_step2<LB>(h23, l23), d2, d3);
    if constexpr (STREAM) __stcs((PT*)(out + p * plane), Pack4<F8>::pack(d0, d1, d2, d3));
    else *(PT*)(out + p * plane) = Pack4<F8>::pack(d0, d1, d2, d3);
  };
  if constexpr (NS > 0) {
#pragma unroll
    for (int p = 0; p < NS; ++p) one(p);
  } else {
    for (int p = 0; p < st; ++p) one(p);
  }
}
template <bool F8>
__device__ __forceinline__ void put4(const dfl (&x)[4], int st, typename Digit<F8>::T* out,
                                     long long plane) {
  put4<F8>(f2_pack(x[0].h, x[1].h), f2_pack(x[0].l, x[1].l), f2_pack(x[2].h, x[3].h),
           f2_pack(x[2].l, x[3].l), st, out, plane);
}

// 2^e as two normal powers of two (e clamped to [-252, 254])
__device__ __forceinline__ void pow2_factors(int e, float& s1, float& s2) {
  e = max(-252, min(254, e));
  s1 = __int_as_float(((e / 2) + 127) << 23);
  s2 = __int_as_float(((e - e / 2) + 127) << 23);
}

// ------------------------------------------------------------------ kernels

// One CTA per fragment: the slots later kernels count or take maxima in (max |T| exponent,
// column maxima of |B|, amplitude CTA counters), the wave's work-queue counters, the check of
// the orbital energies (finite, max(eps_occ) < min(eps_vir), so that every denominator is
// negative; B is checked where it is sliced), and the energies and P_ab of a fragment without
// occupied orbitals, which has no amplitude CTAs.
__global__ void __launch_bounds__(256)
k_split_prologue(const SplitFragDev* __restrict__ f, unsigned* ctr, int check, Bases bs) {
  const SplitFragDev& F = f[blockIdx.x];
  char* ws = (char*)bs.ws;
  if (blockIdx.x == 0 && threadIdx.x < 8) ctr[threadIdx.x] = 0u;
  if (threadIdx.x == 0) {
    ((unsigned*)(ws + F.scal))[1] = 0u;
    if (F.o == 0) {
      bs.energy[F.idx] = 0.0;
      if (bs.energy_os) bs.energy_os[F.idx] = 0.0;
      if (bs.energy_scs) bs.energy_scs[F.idx] = 0.0;
    }
  }
  if (F.o == 0 && F.pab_off >= 0)
    for (long long e = threadIdx.x; e < (long long)F.v * F.v; e += blockDim.x) bs.pab[F.pab_off + e] = 0.0;
  for (int i = threadIdx.x; i <= F.o; i += blockDim.x) ((unsigned*)(ws + F.ecnt))[i] = 0u;
  if (F.sg_out > 0) {
    unsigned long long* cm = (unsigned long long*)(ws + F.ecolm);
    for (int q = threadIdx.x; q < F.X; q += blockDim.x) cm[q] = 0ull;
  }
  if (!check) return;
  // order-preserving keys of the energies (comparisons on the integer pipes; both zeros get
  // the same one)
  auto key = [](double x) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(x), top = 1ull << 63;
    return u & top ? (u == top ? top : ~u) : u | top;
  };
  auto is_nan = [](double x) { return abs_bits(x) > 0x7FF0000000000000ull; };
  __shared__ unsigned long long smax[8], smin[8];
  bool bad = false;
  unsigned long long mx = 0ull, mn = ~0ull;
  for (int e = threadIdx.x; e < F.o; e += blockDim.x) {
    const double x = bs.eps[F.eo_off + e];
    bad |= !finite_bits(x);
    if (!is_nan(x)) mx = max(mx, key(x));
  }
  for (int e = threadIdx.x; e < F.v; e += blockDim.x) {
    const double x = bs.eps[F.ev_off + e];
    bad |= !finite_bits(x);
    if (!is_nan(x)) mn = min(mn, key(x));
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, off));
  }
  if ((threadIdx.x & 31) == 0) { smax[threadIdx.x >> 5] = mx; smin[threadIdx.x >> 5] = mn; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) { mx = max(mx, smax[w]); mn = min(mn, smin[w]); }
    if (F.o > 0 && F.v > 0 && !(mx < mn)) atomicOr(bs.status, ST_DENOM);
  }
  if (bad) atomicOr(bs.status, ST_NONFINITE);
}

// One warp per row (i,a) of B: row exponent, digits of the V operand, d_m and the diagonal
// V_ii(a,a) = sum_Q (B^Q_ia)^2 in FP64.  The diagonal is the one element of V whose two operands have the same
// digits: there the truncated triangle's first dropped even level holds the square of
// the middle digit, an error of one sign that does not average out; the epilogue takes
// this FP64 value instead.
// NCH > 0: the row has at most 128 NCH elements and stays in registers between the maximum
// and the slicing, all its loads in flight at once (four consecutive elements a lane and
// chunk); 0: longer rows are read twice (the second time from L1; registers for 512 or more
// elements cost the occupancy that hides the FP64 sum of squares).  16 trimers (574 MB of B,
// 8 slices): 461 us plus 82 for a separate check of B before, now 400.
template <bool F8, int NCH>
__device__ __forceinline__ void slice_row(const SplitFragDev* __restrict__ f, int nf, long long gr,
                                          int sv, int check, const Bases& bs) {
  using DT = typename Digit<F8>::T;
  const int lane = threadIdx.x & 31;
  const SplitFragDev& F = f[find_sfd(f, nf, gr, 0)];
  const int r = (int)(gr - F.row_begin), X = F.X;
  const double* x = bs.B + F.b_off + (long long)r * X;
  const bool al = ((uintptr_t)x & 15) == 0;   // rows of odd length start on 8-byte boundaries
  auto load4 = [&](int q0, double (&v)[4]) {
    if (al && q0 + 4 <= X) {
      const double2 a = *(const double2*)(x + q0), b = *(const double2*)(x + q0 + 2);
      v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = q0 + k < X ? x[q0 + k] : 0.0;
    }
  };
  unsigned long long mx = 0;   // max |x| as bits
  double ss = 0.0;
  auto look = [&](const double (&v)[4]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      mx = max(mx, abs_bits(v[k]));
      ss = fma(v[k], v[k], ss);
    }
  };
  double row[NCH > 0 ? NCH : 1][4];
  if constexpr (NCH > 0) {
#pragma unroll
    for (int c = 0; c < NCH; ++c) load4(4 * lane + 128 * c, row[c]);
#pragma unroll
    for (int c = 0; c < NCH; ++c)
      if (128 * c < X) look(row[c]);
  } else {
#pragma unroll 4
    for (int q0 = 4 * lane; q0 < X; q0 += 128) {
      double v[4];
      load4(q0, v);
      look(v);
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    ss += __shfl_xor_sync(0xffffffffu, ss, off);
  }
  // the largest |x| as bits is that of an infinity or a NaN where the row holds one
  if (check && lane == 0 && mx >= 0x7FF0000000000000ull) atomicOr(bs.status, ST_NONFINITE);
  const int E = mx > 0 ? ilogb_bits(mx) + 2 + Digit<F8>::HEAD : -1000;
  char* ws = (char*)bs.ws;
  const long long plane = (long long)F.o * F.v * F.xpad;
  DT* out = (DT*)(ws + F.bs1) + (long long)r * F.xpad;
  float s1, s2;
  pow2_factors(Digit<F8>::LB - E, s1, s2);
  // one packed store per plane (elements in [X, xpad) get zero digits; the V operand's tensor
  // map ends at X)
  auto slice4 = [&](int q0, const double (&v)[4]) {
    dfl xs[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float h, l;
      split_to_df(v[k], h, l);
      xs[k] = {(h * s1) * s2, (l * s1) * s2};
    }
    put4<F8>(xs, sv, out + q0, plane);
  };
  if constexpr (NCH > 0) {
#pragma unroll
    for (int c = 0; c < NCH; ++c)
      if (4 * lane + 128 * c < X) slice4(4 * lane + 128 * c, row[c]);
  } else {
    for (int q0 = 4 * lane; q0 < X; q0 += 128) {
      double v[4];
      load4(q0, v);
      slice4(q0, v);
    }
  }
  const int i = r / F.v, a = r - i * F.v;
  if (lane == 0) {
    ((int*)(ws + F.erow))[r] = E;
    const dfl d = d_from(bs.eps[F.eo_off + i] - bs.eps[F.ev_off + a]);
    ((float2*)(ws + F.drow))[r] = make_float2(d.h, d.l);
    // the same terms by padded j blocks for the amplitude kernel's 16-byte loads
    ((float*)(ws + F.dnh))[(long long)i * F.vpadt + a] = d.h;
    ((float*)(ws + F.dnl))[(long long)i * F.vpadt + a] = d.l;
    const dfl vd = d_from(ss);
    ((float2*)(ws + F.vdrow))[r] = make_float2(vd.h, vd.l);
  }
  if (a == F.v - 1 && F.v + lane < F.vpadt) {
    ((float*)(ws + F.dnh))[(long long)i * F.vpadt + F.v + lane] = 0.f;
    ((float*)(ws + F.dnl))[(long long)i * F.vpadt + F.v + lane] = 0.f;
  }
}

// Column maxima of B for Gamma's B operand: max over rows (j,b) of |B^Q_jb| for every aux
// index Q.  One CTA per 32 aux indices x kColRows rows (lane: Q, warp: every 8th row), FP64
// bits combined by atomicMax (non-negative doubles order like their bit patterns).
__device__ __forceinline__ void column_maxima(const SplitFragDev* __restrict__ f, int nf, long long gb,
                                              const Bases& bs) {
  __shared__ unsigned long long red[8][32];   // |B| maxima as bits
  const SplitFragDev& F = f[find_sfd(f, nf, gb, 3)];
  const long long lb = gb - F.qblk_begin;
  const int nqb = (F.X + 31) / 32;
  const int qb = (int)(lb % nqb), rc = (int)(lb / nqb);
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int Q = qb * 32 + lane;
  const int r0 = rc * kColRows, r1 = min(F.o * F.v, r0 + kColRows);
  unsigned long long mx = 0;
  if (Q < F.X) {
    const double* x = bs.B + F.b_off + Q;
#pragma unroll 8
    for (int r = r0 + g; r < r1; r += 8) mx = max(mx, abs_bits(x[(long long)r * F.X]));
  }
  red[g][lane] = mx;
  __syncthreads();
  if (g == 0) {
    for (int k = 1; k < 8; ++k) mx = max(mx, red[k][lane]);
    if (Q < F.X && mx > 0) atomicMax((unsigned long long*)((char*)bs.ws + F.ecolm) + Q, mx);
  }
}

// Both passes over B in one launch: CTAs below row_blocks slice eight rows each, the others take
// the column maxima
template <bool F8, int NCH>
__global__ void __launch_bounds__(256, 6)
k_slice_b1(const SplitFragDev* __restrict__ f, int nf, long long rows, unsigned row_blocks, int sv,
           int check, Bases bs) {
  if (blockIdx.x < row_blocks) {
    const long long gr = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (gr < rows) slice_row<F8, NCH>(f, nf, gr, sv, check, bs);
  } else {
    column_maxima(f, nf, (long long)(blockIdx.x - row_blocks), bs);
  }
}

// Gamma's B operand: Bs2[p][Q][c], c = j*vpad + b (zero for b >= nvir), one scale
// 2^E_Q per aux index, E_Q = ilogb(max_(j,b) |B^Q_jb|) + 2 + HEAD (also stored for the GEMM
// epilogue).  Tiles of B2Q aux indices x B2C columns c (128 bytes of digits), loaded with
// every element in flight and transposed through shared memory; each thread then writes four
// consecutive c of one Q, one packed store per plane, the lanes of a row covering whole lines.
template <bool F8> constexpr int B2Q = F8 ? 16 : 32;
template <bool F8> constexpr int B2C = F8 ? 128 : 64;

template <bool F8>
__device__ __forceinline__ void slice_b2(const SplitFragDev* __restrict__ f, int nf, long long gt, int st,
                                         double (*tile)[B2C<F8> + 2], const Bases& bs) {
  using DT = typename Digit<F8>::T;
  constexpr int NQ = B2Q<F8>, NC = B2C<F8>, RS = 256 / NQ;   // RS: columns c per load pass
  const SplitFragDev& F = f[find_sfd(f, nf, gt, 1)];
  const long long lt = gt - F.b2_tile_begin;
  const int RL = F.o * F.vpad;
  const int ntc = (RL + NC - 1) / NC;
  const int tq = (int)(lt / ntc), tc = (int)(lt % ntc);
  {
    const int tx = threadIdx.x % NQ, ty = threadIdx.x / NQ, Q = tq * NQ + tx;
    const double* B = bs.B + F.b_off + Q;
    int c = tc * NC + ty, j = c / F.vpad, b = c - j * F.vpad;
    double val[NC / RS];
#pragma unroll
    for (int k = 0; k < NC / RS; ++k) {
      val[k] = c < RL && b < F.v && Q < F.X ? B[((long long)j * F.v + b) * F.X] : 0.0;
      c += RS;
      b += RS;
      while (b >= F.vpad) { b -= F.vpad; ++j; }
    }
#pragma unroll
    for (int k = 0; k < NC / RS; ++k) tile[tx][ty + RS * k] = val[k];
  }
  __syncthreads();
  char* ws = (char*)bs.ws;
  const unsigned long long* cm = (const unsigned long long*)(ws + F.ecolm);
  int* ec = (int*)(ws + F.ecol);
  const long long plane = (long long)F.X * F.ldd;
  DT* out = (DT*)(ws + F.bs2);
  const int cl = 4 * (threadIdx.x % (NC / 4)), c = tc * NC + cl;   // RL is a multiple of 4
#pragma unroll 1
  for (int qi = threadIdx.x / (NC / 4); qi < NQ; qi += 1024 / NC) {
    const int Q = tq * NQ + qi;
    if (Q >= F.X || c >= RL) break;
    const int E = cm[Q] > 0 ? ilogb_bits(cm[Q]) + 2 + Digit<F8>::HEAD : -1000;
    if (c == 0) ec[Q] = E;
    float s1, s2;
    pow2_factors(Digit<F8>::LB - E, s1, s2);
    const double2 u = *(const double2*)&tile[qi][cl], w = *(const double2*)&tile[qi][cl + 2];
    const double v4[4] = {u.x, u.y, w.x, w.y};
    dfl xs[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float h, l;
      split_to_df(v4[k], h, l);
      xs[k] = {(h * s1) * s2, (l * s1) * s2};
    }
    put4<F8>(xs, st, out + (long long)Q * F.ldd + c, plane);
  }
}

// Exponent of T's scale from the largest |T|'s
template <bool F8>
__device__ __forceinline__ int t_scale(unsigned emax) {
  return Digit<F8>::LB - ((int)emax - 124 + Digit<F8>::HEAD);
}

// Pair energies e_ij, j >= i, and their opposite-spin parts: the amplitude warps' shares of row
// i summed in a fixed order (FP64) by warp w of nw; strips: row strips of the fragment, kt: the
// exponent of T's scale
__device__ __forceinline__ void row_energies(const SplitFragDev& F, char* ws, int i, int w, int nw, int strips,
                                             int kt) {
  const int o = F.o, lane = threadIdx.x & 31;
  double* ep = (double*)(ws + F.ep);
  const int parts = F.v > 0 ? strips * 8 : 0;
  for (int j0 = i + 4 * w; j0 < o; j0 += 4 * nw) {   // eight lanes a pair
    const int jj = j0 + (lane >> 3);
    double e = 0.0, eo = 0.0;
    if (jj < o) {
      const float4* p = (const float4*)(ws + F.epart) + ((long long)i * o + jj) * (strips * 8);
#pragma unroll 4
      for (int k = lane & 7; k < parts; k += 8) {
        const float4 x = __ldcg(p + k);
        e += (double)x.x + (double)x.y;
        eo += (double)x.z + (double)x.w;
      }
    }
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) {
      e += __shfl_xor_sync(0xffffffffu, e, off);
      eo += __shfl_xor_sync(0xffffffffu, eo, off);
    }
    if (jj < o && (lane & 7) == 0) {
      e = ldexp(e, 1 - 2 * kt);   // the scales of T and Tt
      eo = ldexp(eo, -2 * kt);
      ep[(long long)i * o + jj] = e;
      ep[(long long)jj * o + i] = e;
      double* eq = ep + (long long)o * o;   // opposite-spin pair energies
      eq[(long long)i * o + jj] = eo;
      eq[(long long)jj * o + i] = eo;
    }
  }
}

// Amplitude stage: Tt = 2T - T^T, digits of T and Tt (one scale per fragment each), pair
// energies e_ij = sum_ab Tt_ij(a,b) V_ij(a,b) (V = T D) and their opposite-spin part
// sum_ab T_ij(a,b) V_ij(a,b) for i <= j.
//
// A CTA takes a strip of ROWS rows (i, a0 ..) and a range of j; per step it forms C = 4 LPR
// columns of one j block, a group of LPR lanes per row, four columns a lane.  The stored block
// (min(i,j), max(i,j)) of the double-float T planes (rows (i,a), columns j*vpadt + b;
// T_ij(a,b) = T_ji(b,a)) gives both operands: a direct tile (rows a, columns b) the lanes read
// for themselves, and a transposed tile (rows b, columns a) that goes through shared memory.
// For i <= j the direct tile is T and the other its partner T_ij(b,a), for i > j the reverse.
//
// The write pattern bounds this kernel: 24 (BF16) or 20 (FP8) bytes an element in 12 or 20
// planes.  HBM and L2 take full rate only when a warp's store covers whole 128-byte lines of a
// row, and neighbouring lines follow soon: as pairs of 32 x 32 tiles (64 or 32 bytes a row and
// store) the same bytes moved at 3.1 TB/s (BF16) and 1.3 TB/s (FP8), in these strips at 6.2
// and 4.8 (copies of both patterns without the arithmetic, nocc=40 nvir=400), although the
// strips read T twice.
// LPR: lanes per row, 32, or fewer where the rows are short (amp_lanes).
template <bool F8, int LPR>
__global__ void __launch_bounds__(256, 3)
k_amp_split(const SplitFragDev* __restrict__ f, int nf, unsigned amp_ctas, int sg, int sums, Bases bs) {
  using DT = typename Digit<F8>::T;
  constexpr int LB = Digit<F8>::LB;
  constexpr int GROUPS = 32 / LPR, ROWS = 8 * GROUPS, C = 4 * LPR;
  constexpr int LDY = C + 4;   // 16-byte rows; the transposing writes of a warp then hit all banks
  union Smem {
    float y[2][2][ROWS * LDY];    // [hi / lo][buffer]
    double tile[B2Q<F8>][B2C<F8> + 2];
  };
  __shared__ __align__(16) Smem sm;
  __shared__ int s_last;
  if (blockIdx.x >= amp_ctas) {   // Gamma's B operand, needed only after this launch
    slice_b2<F8>(f, nf, (long long)(blockIdx.x - amp_ctas), sg, sm.tile, bs);
    return;
  }
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const SplitFragDev& F = f[find_sfd(f, nf, blockIdx.x, 2)];
  const int v = F.v, o = F.o, vpad = F.vpad, vpadt = F.vpadt;
  const int strips = max(1, (v + ROWS - 1) / ROWS);
  // CTA -> (i, j range, strip): neighbouring CTAs take neighbouring strips of the same i
  int q = (int)(blockIdx.x - F.pair_begin);
  const int strip = q % strips;
  q /= strips;
  const int jranges = (o + F.amp_jchunk - 1) / F.amp_jchunk;
  const int i = q / jranges;
  const int st = F.st_out, stt = F.st_t;   // digit planes of Tt (0: energies only) and T (0: no P)
  const int jb0 = (q % jranges) * F.amp_jchunk, je = min(o, jb0 + F.amp_jchunk);
  const int jb = st == 0 ? max(jb0, i) : jb0;   // energies only: the pairs i <= j
  // BF16: the usual plane count (6) unrolled; FP8's ten planes stay a loop (unrolled, they
  // cost more registers than the loop saves)
  constexpr int NS = F8 ? 0 : 6;
  const bool ns = NS > 0 && st == NS && stt == NS;
  char* ws = (char*)bs.ws;
  const float* Th = (const float*)(ws + F.thi);
  const float* Tl = (const float*)(ws + F.tlo);
  const float* __restrict__ Dh = (const float*)(ws + F.dnh);   // e_j - e_b at j*vpadt + b
  const float* __restrict__ Dl = (const float*)(ws + F.dnl);
  const unsigned emax = *(const unsigned*)(ws + F.scal + 4);
  // |T| < 2^(emax - 126) and |Tt| <= 3 max |T| < 2^(emax - 124): the scales 2^kt of T and
  // 2^(kt - 1) of Tt keep both within 2^(E - 2 - HEAD) and 2^(E - 1 - HEAD).  T_ij(b,a) is
  // scaled by the latter, so that Tt = 2T - T^T is a plain difference of scaled values, and the
  // energies are formed from the scaled T and Tt (all exact powers of two).
  const int kt = t_scale<F8>(emax);
  const bool one = kt <= 126 && kt >= -125;   // 2^kt is a normal float (unless |T| < 2^-121)
  float sa, sb;
  pow2_factors(kt, sa, sb);
  if (one) { sa = __int_as_float((kt + 127) << 23); sb = 1.f; }
  const f2x sc_t = f2_two(sa), sc_y = f2_two(0.5f * sa), sc_2 = f2_two(sb);
  DT* tts = (DT*)(ws + F.tts);
  DT* ts = (DT*)(ws + F.ts);
  const long long ldd = F.ldd, ldt = F.ldt, plane = (long long)o * v * ldd;
  const int nb = (vpad + C - 1) / C, steps = max(0, je - jb) * nb;
  const int a0 = strip * ROWS;
  // this lane's row and columns of the direct tile, and its float4 of the transposed one
  const int row = warp * GROUPS + lane / LPR, a = a0 + row, c0 = 4 * (lane % LPR);
  const int yq = 4 * (tid % (ROWS / 4)), yb = tid / (ROWS / 4);

  // this CTA's share of the outputs that the contractions accumulate into
  {
    const long long ctas = (long long)strips * jranges * o, me = (long long)(blockIdx.x - F.pair_begin);
    const long long no = F.pij_off >= 0 ? (long long)o * o : 0, nv = F.pab_off >= 0 ? (long long)v * v : 0;
    const long long ng = F.zero_gamma ? (long long)o * v * F.X : 0;
    for (long long e = me * 256 + tid; e < no; e += ctas * 256) bs.pij[F.pij_off + e] = 0.0;
    for (long long e = me * 256 + tid; e < nv; e += ctas * 256) bs.pab[F.pab_off + e] = 0.0;
    for (long long e = me * 256 + tid; e < ng; e += ctas * 256) __stcs(bs.gamma + F.gamma_off + e, 0.0);
  }
  // the next step's direct and transposed elements; their offsets advance within a j block
  float4 dh, dl, xh, xl;
  long long id = 0, ix = 0;
  const long long xstep = (long long)C * ldt;
  auto load = [&](int j, int b0) {
    if (b0 == 0) {
      const long long rows = (long long)min(i, j) * v, cols = (long long)max(i, j) * vpadt;
      id = (rows + a) * ldt + cols + c0;
      ix = (rows + yb) * ldt + cols + a0 + yq;
    }
    dh = dl = xh = xl = make_float4(0.f, 0.f, 0.f, 0.f);
    if (a < v && b0 + c0 < vpadt) {
      dh = __ldg((const float4*)(Th + id));
      dl = __ldg((const float4*)(Tl + id));
    }
    if (b0 + yb < v && a0 + yq < vpadt) {
      xh = __ldg((const float4*)(Th + ix));
      xl = __ldg((const float4*)(Tl + ix));
    }
    id += C;
    ix += xstep;
  };

  // pair energy and its opposite-spin part, two running sums each (even and odd columns)
  f2x e_h = 0ull, e_l = 0ull, o_h = 0ull, o_l = 0ull;
  const float dmh1 = a < v ? Dh[(long long)i * vpadt + a] : 0.f, dml1 = a < v ? Dl[(long long)i * vpadt + a] : 0.f;
  const f2x dmh = f2_two(dmh1), dml = f2_two(dml1);
  int j = jb, b0 = 0;
  if (steps > 0) load(j, 0);
  for (int s = 0; s < steps; ++s) {
    float* const Sh = sm.y[0][s & 1];
    float* const Sl = sm.y[1][s & 1];
    Sh[(yq + 0) * LDY + yb] = xh.x; Sh[(yq + 1) * LDY + yb] = xh.y;
    Sh[(yq + 2) * LDY + yb] = xh.z; Sh[(yq + 3) * LDY + yb] = xh.w;
    Sl[(yq + 0) * LDY + yb] = xl.x; Sl[(yq + 1) * LDY + yb] = xl.y;
    Sl[(yq + 2) * LDY + yb] = xl.z; Sl[(yq + 3) * LDY + yb] = xl.w;
    f2x th[2] = {f2_pack(dh.x, dh.y), f2_pack(dh.z, dh.w)};
    f2x tl[2] = {f2_pack(dl.x, dl.y), f2_pack(dl.z, dl.w)};
    __syncthreads();   // the other buffer's readers are past it: two buffers, one barrier a step
    const int cj = j, b = b0 + c0;
    b0 += C;
    if (b0 >= vpad) { b0 = 0; ++j; }
    if (s + 1 < steps) load(j, b0);   // in flight while this step is processed
    if (a < v && b < vpad) {
      const float4 ph = *(const float4*)(Sh + row * LDY + c0), pl = *(const float4*)(Sl + row * LDY + c0);
      f2x yh[2] = {f2_pack(ph.x, ph.y), f2_pack(ph.z, ph.w)};
      f2x yl[2] = {f2_pack(pl.x, pl.y), f2_pack(pl.z, pl.w)};
      if (i > cj) {
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          f2x t = th[g]; th[g] = yh[g]; yh[g] = t;
          t = tl[g]; tl[g] = yl[g]; yl[g] = t;
        }
      }
      if (b + 4 > v) {   // columns in [nvir, vpad) get zero digits
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          const f2x m = (b + 2 * g < v ? 0xffffffffull : 0ull) |
                        (b + 2 * g + 1 < v ? 0xffffffff00000000ull : 0ull);
          th[g] &= m; tl[g] &= m; yh[g] &= m; yl[g] &= m;
        }
      }
      f2x uh[2], ul[2];   // Tt
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        th[g] = f2_mul(th[g], sc_t);
        tl[g] = f2_mul(tl[g], sc_t);
        yh[g] = f2_mul(yh[g], sc_y);
        yl[g] = f2_mul(yl[g], sc_y);
        if (!one) {
          th[g] = f2_mul(th[g], sc_2);
          tl[g] = f2_mul(tl[g], sc_2);
          yh[g] = f2_mul(yh[g], sc_2);
          yl[g] = f2_mul(yl[g], sc_2);
        }
        d_sub2(th[g], tl[g], yh[g], yl[g], uh[g], ul[g]);
      }
      if (i <= cj && b < v) {
        const float4 nh = __ldg((const float4*)(Dh + (long long)cj * vpadt + b));
        const float4 nl = __ldg((const float4*)(Dl + (long long)cj * vpadt + b));
        const f2x dnh[2] = {f2_pack(nh.x, nh.y), f2_pack(nh.z, nh.w)};
        const f2x dnl[2] = {f2_pack(nl.x, nl.y), f2_pack(nl.z, nl.w)};
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          const f2x nt = f2_neg(th[g]);
          f2x dh2, dl2, vh, vl, qh, ql;
          f2_two_sum(dmh, dnh[g], dh2, dl2);
          dl2 = f2_add(dl2, f2_add(dml, dnl[g]));
          d_mul2(th[g], nt, tl[g], dh2, dl2, vh, vl);
          d_mul2(uh[g], f2_neg(uh[g]), ul[g], vh, vl, qh, ql);
          d_acc2(e_h, e_l, qh, ql);
          d_mul2(th[g], nt, tl[g], vh, vl, qh, ql);
          d_acc2(o_h, o_l, qh, ql);
        }
      }
      if (st > 0) {
        const long long out = ((long long)i * v + a) * ldd + (long long)cj * vpad + b;
        if (ns) {
          put4<F8, NS, true>(th[0], tl[0], th[1], tl[1], stt, ts + out, plane);
          put4<F8, NS, true>(uh[0], ul[0], uh[1], ul[1], st, tts + out, plane);
        } else {
          put4<F8, 0, true>(th[0], tl[0], th[1], tl[1], stt, ts + out, plane);
          put4<F8, 0, true>(uh[0], ul[0], uh[1], ul[1], st, tts + out, plane);
        }
      }
    }
    if (i <= cj && b0 == 0) {   // the block (i, cj) is done: this warp's share of its energy
      auto join = [](f2x h, f2x l) {
        float h0, h1, l0, l1;
        f2_unpack(h, h0, h1);
        f2_unpack(l, l0, l1);
        return d_add({h0, l0}, {h1, l1});
      };
      // lanes 0..15 go on with the energy, 16..31 with its opposite-spin part
      const dfl e = join(e_h, e_l), eo = join(o_h, o_l);
      const bool up = lane >= 16;
      const dfl give = up ? e : eo, keep = up ? eo : e;
      dfl w = d_add(keep, {__shfl_xor_sync(0xffffffffu, give.h, 16), __shfl_xor_sync(0xffffffffu, give.l, 16)});
#pragma unroll
      for (int off = 8; off > 0; off >>= 1)
        w = d_add(w, {__shfl_xor_sync(0xffffffffu, w.h, off), __shfl_xor_sync(0xffffffffu, w.l, off)});
      if ((lane & 15) == 0)
        ((float2*)(ws + F.epart))[2 * (((long long)i * o + cj) * (strips * 8) + strip * 8 + warp) + up] =
            make_float2(w.h, w.l);
      e_h = e_l = o_h = o_l = 0ull;
    }
  }
  if (!sums) return;   // k_split_energy's
  // the last CTA of row i sums the warps' shares of e_ij, j >= i
  __threadfence();
  __syncthreads();
  if (tid == 0)
    s_last = atomicAdd((unsigned*)(ws + F.ecnt) + i, 1u) + 1u == (unsigned)(strips * jranges);
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  row_energies(F, ws, i, warp, 8, strips, kt);
  // the last row's CTA sums the fragment's energies
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd((unsigned*)(ws + F.ecnt) + o, 1u) + 1u == (unsigned)o;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const double* ep = (const double*)(ws + F.ep);
  fragment_energy(ep, ep + (long long)o * o, (long long)o * o,
                  F.epair_off >= 0 ? bs.epair + F.epair_off : nullptr, F.idx, bs);
}

// The energies of small fragments, a CTA each, beside the contractions that follow (they start
// as soon as this kernel's CTAs have).  Counted down by the amplitude CTAs, row by row and then
// for the fragment, the sums are a chain of fences and FP64 latencies that P and Gamma would
// wait for.  A call (BF16) at nocc=4 65 -> 59 us, nocc=10 nvir=40 naux=150 88 -> 78, nocc=24
// nvir=96 naux=360 343 -> 328; from nocc=32 on nothing is left of it, and one CTA is too few for
// many pairs of a short call (nocc=100 nvir=20 naux=200 342 -> 581 us): up to kSepOcc.
constexpr int kSepOcc = 24;

template <bool F8>
__global__ void __launch_bounds__(256)
k_split_energy(const SplitFragDev* __restrict__ f, int lpr, Bases bs) {
  pdl_trigger();
  const SplitFragDev& F = f[blockIdx.x];
  if (F.o == 0) return;   // the prologue's
  char* ws = (char*)bs.ws;
  const int warp = threadIdx.x >> 5, rows = 8 * 32 / lpr, strips = max(1, (F.v + rows - 1) / rows);
  const int kt = t_scale<F8>(*(const unsigned*)(ws + F.scal + 4));
  for (int i = warp; i < F.o; i += 8) row_energies(F, ws, i, 0, 1, strips, kt);
  __threadfence_block();
  __syncthreads();
  const double* ep = (const double*)(ws + F.ep);
  fragment_energy(ep, ep + (long long)F.o * F.o, (long long)F.o * F.o,
                  F.epair_off >= 0 ? bs.epair + F.epair_off : nullptr, F.idx, bs);
}

// ------------------------------------------------------------------ host

namespace {

// Tile shapes a launch of `slices` digit planes can take: the default one (n_tile_first,
// 0: the kernel's default width) first, then every other (n_tile, K per stage) the kernel
// is built for whose level accumulators fit the 512 TMEM columns (BF16: 48..96 columns x
// K 32 or 16; FP8: 32..64 columns); non-zero n_tile / stage_k options pin that dimension.
std::vector<SplitLaunch> shape_candidates(int slices, bool fp8, int n_tile_first, int stage_k,
                                          int n_tile) {
  std::vector<SplitLaunch> c;
  c.push_back(split_launch_config(slices, stage_k ? stage_k : 32, n_tile_first, fp8));
  auto add = [&](const SplitLaunch& x) {
    for (const auto& y : c)
      if (y.n_tile_max == x.n_tile_max && y.bk == x.bk) return;
    c.push_back(x);
  };
  if (fp8) {
    for (int nt : {64, 48, 32})
      if ((n_tile == 0 || n_tile == nt) && slices * nt <= 512) {
        const SplitLaunch x = split_launch_config(slices, 64, nt, true);
        if (x.n_tile_max == nt) add(x);
      }
  } else {
    for (int bk : {32, 16})
      for (int nt : {64, 48, 80, 96})
        if ((stage_k == 0 || stage_k == bk) && (n_tile == 0 || n_tile == nt)) {
          const SplitLaunch x = split_launch_config(slices, bk, nt, false);
          if (x.n_tile_max == nt && slices * nt <= 512) add(x);
        }
  }
  return c;
}

}  // namespace

void split_set_shapes(SplitPlan& sp, int iv, int it, int ig) {
  auto pick = [](const std::vector<SplitLaunch>& c, int i) {
    return std::max(0, std::min(i, (int)c.size() - 1));
  };
  sp.shape_v = pick(sp.cand_v, iv);
  sp.shape_t = pick(sp.cand_t, it);
  // Gamma with P's slice count runs in P's launch: it must take that launch's shape
  sp.shape_g = sp.slices_g == sp.slices_t ? sp.shape_t : pick(sp.cand_g, ig);
  sp.cfg_t = sp.cand_t[sp.shape_t];
  sp.cfg_g = sp.cand_g[sp.shape_g];
  sp.v_by_wave = false;
}

int split_plan_init(SplitPlan& sp, int precision, const rimp2_options& opt) {
  sp.precision = precision;
  sp.slices_v = opt.slices_v;
  sp.slices_t = opt.slices_t;
  sp.slices_g = opt.slices_g;
  sp.fp8 = precision == RIMP2_FP8_SPLIT;
  // First tile widths per launch (BF16; an n_tile option overrides them): Gamma, with K =
  // nocc x nvir, takes 80 columns, whose wider B tiles cut its operand traffic (nocc=100
  // nvir=500 naux=1500: 74 ms against 80 at 64); P_ab / P_ij keep 64; V: split_shape_v.
  int nv = opt.n_tile, ng = opt.n_tile;
  if (!sp.fp8 && opt.n_tile == 0) {
    nv = 2 * sp.slices_v * 48 <= 512 ? 48 : 0;
    ng = sp.slices_g * 80 <= 512 && sp.slices_g != sp.slices_t ? 80 : 0;
  }
  sp.cand_v = shape_candidates(sp.slices_v, sp.fp8, nv, opt.stage_k, opt.n_tile);
  sp.cand_t = shape_candidates(sp.slices_t, sp.fp8, opt.n_tile, opt.stage_k, opt.n_tile);
  sp.cand_g = shape_candidates(sp.slices_g, sp.fp8, ng, opt.stage_k, opt.n_tile);
  split_set_shapes(sp, 0, 0, 0);
  sp.v_by_wave = opt.n_tile == 0;
  sp.grid = split_gemm_grid();
  if (split_gemm_prepare() != cudaSuccess) { cudaGetLastError(); return RIMP2_ERR_CUDA; }
  sp.ready = true;
  return RIMP2_OK;
}

// V's tile width before any tuning, by the work of one launch (of each wave: 64 monomers, nocc
// 8..20, in 64 waves 4.04 ms with the whole batch's 64 columns, 3.99 with a wave's 48). Its
// operands come from L2, (128 + n_tile) rows for 128 x n_tile results, and bound a launch of
// many tiles; wider tiles need less of them, but leave SMs idle where the tiles are few and,
// with 5 slices, spend longer in the epilogue of a short K (48 columns leave TMEM for a second
// accumulator set, which hides it). Measured, BF16 with 5 slices at 48 / 64 / 80 columns:
// nocc=10 nvir=40 naux=150 31 / 33 / 43 us, nocc=20 nvir=80 naux=300 46 / 49 / 57 us, nocc=29
// nvir=117 naux=437 111 / 110 / 125 us, 40 MBE3 dimers (naux about 420) 3.58 / 3.21 / 3.22 ms,
// nocc=42 nvir=168 naux=630 453 / 442 / 428 us, nocc=50 nvir=250 naux=750 1.46 / 1.38 / 1.30
// ms, nocc=100 nvir=500 naux=1500 38.9 / 37.2 / 34.3 ms (96 columns: 35.6). 8 slices at 48 /
// 64: nocc=20 55 / 66 us, nocc=29 174 / 162, nocc=42 854 / 768 us; FP8 with 8 slices: nocc=20
// 47 / 57 us, nocc=29 119 / 121, nocc=42 480 / 442 us.
int split_shape_v(const SplitPlan& sp, const rimp2_frag* frags, const std::vector<int>& members) {
  if (!sp.v_by_wave) return sp.shape_v;
  double tiles = 0.0, blocks = 0.0;   // tiles of 128 x 48 with results; times naux
  for (int f : members) {
    const double ov = (double)frags[f].nocc * frags[f].nvir, t = ov * (ov + SG_BM) / (2.0 * SG_BM * 48);
    tiles += t;
    blocks += t * frags[f].naux;
  }
  const bool two = !sp.fp8 && 2 * sp.slices_v * 48 <= 512;
  const int want = tiles < 4.0 * sp.grid ? 48 : two && blocks >= 576.0 * tiles ? 80 : 64;
  for (int nt : {want, 64, 48})
    for (size_t i = 0; i < sp.cand_v.size(); ++i)
      if (sp.cand_v[i].n_tile_max == nt && sp.cand_v[i].bk == sp.cand_v[0].bk) return (int)i;
  return sp.shape_v;
}

void split_plan_release(SplitPlan&) {}

namespace {

struct Layout {
  size_t bs1, bs2, erow, drow, vdrow, dnh, dnl, thi, tlo, tts, ts, ecolm, ecol, ep, epart, ecnt, scal, total;
};

// element size of the digit planes and the padding that keeps every row 16-byte aligned
size_t esz_of(const SplitPlan& sp) { return sp.fp8 ? 1 : 2; }
int padg(const SplitPlan& sp) { return sp.fp8 ? 16 : 8; }

// Padded extent of a digit-row segment of n elements: the widest alignment up to 128 bytes
// of digits that costs under 3 % of padding (so that row segments start on L2 line or
// sector boundaries), at least the 16-byte TMA stride rule.
int pad_extent(const SplitPlan& sp, int n) {
  const int esz = (int)esz_of(sp);
  for (int a = 128 / esz; a > padg(sp); a /= 2) {
    const int r = rup(n, a);
    if ((long long)(r - n) * 100 < 3LL * n) return r;
  }
  return rup(n, padg(sp));
}

// Row stride of a plane whose rows hold n elements of esz bytes: the smallest odd multiple of
// 128 bytes that holds them.  Tiles that run side by side read rows a fixed number of rows
// apart; with strides that are multiples of large powers of two their addresses coincide
// modulo 4 KB and crowd the same L2 slices.
long long row_stride(long long n, long long esz) {
  long long lines = (n * esz + 127) / 128;
  if ((lines & 1) == 0) ++lines;
  return lines * 128 / esz;
}

Layout frag_layout(const SplitPlan& sp, const rimp2_frag& f) {
  const size_t o = f.nocc, v = f.nvir, X = f.naux;
  const size_t esz = esz_of(sp);
  const size_t ov = o * v, vpad = pad_extent(sp, (int)v), xpad = pad_extent(sp, (int)X), RL = o * vpad;
  // digit planes exist only when an output needs them: T and Tt for P_ab and P_ij; Tt
  // (its leading s_g planes) and B^T with one scale per aux index for Gamma
  const bool want_p = f.pij_off >= 0 || f.pab_off >= 0;
  const size_t st_g = f.gamma_off >= 0 ? (size_t)sp.slices_g : 0;
  const size_t st_t = want_p ? (size_t)sp.slices_t : 0;
  const size_t st_tt = std::max(st_t, st_g);
  Layout L{};
  size_t off = 0;
  L.bs1 = off; off += al256((size_t)sp.slices_v * ov * xpad * esz);
  const size_t ldd = (size_t)row_stride((long long)RL, (long long)esz);
  const size_t ldt = (size_t)row_stride((long long)o * rup((int)v, 32), 4);
  L.bs2 = off; off += al256(st_g * X * ldd * esz);
  L.erow = off; off += al256(ov * 4);
  L.drow = off; off += al256(ov * 8);
  L.vdrow = off; off += al256(ov * 8);
  L.dnh = off; off += al256(o * rup((int)v, 32) * 4);
  L.dnl = off; off += al256(o * rup((int)v, 32) * 4);
  L.thi = off; off += al256(ov * ldt * 4);   // T planes: rows (i,a), columns j*vpadt + b
  L.tlo = off; off += al256(ov * ldt * 4);
  L.tts = off; off += al256(st_tt * ov * ldd * esz);
  L.ts = off; off += al256(st_t * ov * ldd * esz);
  L.ecolm = off; off += al256(X * 8);
  L.ecol = off; off += al256(X * 4);
  L.ep = off; off += al256(2 * o * o * 8);   // pair energies, opposite-spin pair energies
  L.epart = off; off += al256(o * o * 8 * ((v + 7) / 8) * 16);   // warps' shares, at most
  L.ecnt = off; off += al256((o + 1) * 4);
  L.scal = off; off += 256;
  L.total = off;
  return L;
}

void choose_split_k(SplitProb& P, int grid, int mul) {
  const long long tiles = (long long)P.tiles_m * P.tiles_n;
  long long want = std::max(1LL, ((long long)mul * grid + tiles - 1) / tiles);
  want = std::min<long long>(want, std::max(1, P.k1_count));
  int chunk = (int)((P.k1_count + want - 1) / want);
  if (chunk < 1) chunk = 1;
  P.k1_chunk = chunk;
  P.ksplit = std::max(1, (P.k1_count + chunk - 1) / chunk);
}

// Tensor-core FLOPs one problem issues: 2 x 128 x n_tile x K per computed tile (the
// skip rules of the kernel's tile decoder: V keeps tiles with some row >= some column,
// symmetric accumulations tiles with some row <= some column) x the digit products.
double prob_mma_flops(const SplitProb& P, int slices, int bk) {
  long long tiles = 0;
  for (int tm = 0; tm < P.tiles_m; ++tm)
    for (int tn = 0; tn < P.tiles_n; ++tn) {
      bool skip = P.kind == PK_V && tm * SG_BM + SG_BM - 1 < tn * P.n_tile;
      if (P.sym) skip = tm * SG_BM > tn * P.n_tile + P.n_tile - 1;
      tiles += !skip;
    }
  const double K = (double)P.k1_count * P.k0_blocks * bk;
  return (double)tiles * 2.0 * SG_BM * P.n_tile * K * (slices * (slices + 1) / 2);
}

// Lanes per row of the amplitude kernel: a step takes 1024 element slots whatever the width,
// so the width that wastes fewest on rows and columns past nvir, weighted by what a full step
// costs.  Measured per step relative to 16 lanes (nocc=100 nvir=500, MBE3 dimers, nocc=42
// nvir=168 in FP8): BF16 1.06 with 32 lanes (its 64 columns already fill 128-byte lines with
// 16), 1.05 with 8 (64-byte runs); FP8 0.96 and 1.25 (32 lanes are what fills its lines).
int amp_lanes(const std::vector<SplitFragDev>& fr, bool fp8) {
  int best = 0;
  double cost = 0.0;
  for (int lpr : {16, 32, 8}) {
    double c = 0.0;
    for (const auto& s : fr)
      c += (double)s.o * s.o * ((s.v + 256 / lpr - 1) / (256 / lpr)) * ((s.vpad + 4 * lpr - 1) / (4 * lpr));
    c *= lpr == 16 ? 1.0 : lpr == 32 ? (fp8 ? 0.96 : 1.06) : (fp8 ? 1.25 : 1.05);
    if (best == 0 || c < cost) { best = lpr; cost = c; }
  }
  return best;
}

void finish(std::vector<SplitProb>& v, long long& total) {
  std::stable_sort(v.begin(), v.end(), [](const SplitProb& a, const SplitProb& b) {
    return (double)a.k0_blocks * a.k1_chunk > (double)b.k0_blocks * b.k1_chunk;
  });
  total = 0;
  for (auto& P : v) {
    P.tile_begin = total;
    total += P.ntiles;
  }
}

}  // namespace

size_t split_frag_ws_bytes(const SplitPlan& sp, const rimp2_frag& f) {
  return frag_layout(sp, f).total;
}

int split_build_wave(SplitPlan& sp, const rimp2_frag* frags, const std::vector<int>& members,
                     const double* B, void* ws, SplitWave& w, long long& total_pairs) {
  (void)B;
  char* wsb = (char*)ws;
  size_t off = 0;
  long long pairs = 0, rows = 0, b2t = 0, qbl = 0;
  const int sv = sp.slices_v, st = sp.slices_t, sgl = sp.slices_g;
  // Gamma with P's slice count joins P's launch and so takes its tile shape
  const SplitLaunch& cg = sgl == st ? sp.cfg_t : sp.cfg_g;
  w.cfg_v = sp.cand_v[split_shape_v(sp, frags, members)];
  const int NTv = w.cfg_v.n_tile_max, NTt = sp.cfg_t.n_tile_max, NTg = cg.n_tile_max;
  const int BKv = w.cfg_v.bk, BKt = sp.cfg_t.bk, BKg = cg.bk;
  const int BKs = sp.fp8 ? 64 : 32;   // K per stage of the slice-stacked kernel
  // split-K target of P_ab / P_ij in multiples of the grid: finer pieces keep the tiles of
  // one occupied-index range closer together in time (their operand rows stay in L2);
  // measured at nocc=100 nvir=500 naux=1500: the P launch 33.3 ms at 2x, 32.2 at 8x, 31.6
  // at 16x; at nocc=42 nvir=168 naux=630: 0.73, 0.65, 0.68 ms
  const int split_mul = sp.variant == 2 ? 16 : 8;
  const bool pij_direct = sp.variant == 1;
  // exponents of the Tt and T digit planes: the stored max |T| exponent plus these (the
  // amplitude kernel's scales)
  const int head = sp.fp8 ? SG_HEAD_FP8 : SG_HEAD_BF16;
  const int kTtAdd = -123 + head, kTAdd = -124 + head;
  for (int idx : members) {
    const rimp2_frag& f = frags[idx];
    const Layout L = frag_layout(sp, f);
    const int o = f.nocc, v = f.nvir, X = f.naux;
    const int ov = o * v, vpad = pad_extent(sp, v), xpad = pad_extent(sp, X), RL = o * vpad;
    const uint64_t E2 = esz_of(sp);
    const int vpadt = rup(v, 32);
    const long long ldd = row_stride(RL, (long long)E2), ldt = row_stride((long long)o * vpadt, 4);
    SplitFragDev s{};
    s.o = o; s.v = v; s.X = X; s.idx = idx; s.vpad = vpad; s.xpad = xpad;
    s.ldd = ldd; s.ldt = ldt; s.vpadt = vpadt;
    const bool g = f.gamma_off >= 0 && X > 0 && ov > 0;
    const bool want_p = f.pij_off >= 0 || f.pab_off >= 0;
    s.st_t = want_p ? st : 0;
    s.sg_out = g ? sgl : 0;
    s.st_out = std::max(s.st_t, s.sg_out);
    s.b_off = f.b_off; s.eo_off = f.eo_off; s.ev_off = f.ev_off;
    s.gamma_off = f.gamma_off; s.pij_off = f.pij_off; s.pab_off = f.pab_off; s.epair_off = f.epair_off;
    s.bs1 = off + L.bs1; s.bs2 = off + L.bs2; s.erow = off + L.erow; s.drow = off + L.drow;
    s.vdrow = off + L.vdrow; s.dnh = off + L.dnh; s.dnl = off + L.dnl;
    s.thi = off + L.thi; s.tlo = off + L.tlo; s.tts = off + L.tts; s.ts = off + L.ts;
    s.ecolm = off + L.ecolm; s.ecol = off + L.ecol;
    s.ep = off + L.ep; s.epart = off + L.epart; s.ecnt = off + L.ecnt; s.scal = off + L.scal;
    s.row_begin = rows; s.b2_tile_begin = b2t; s.qblk_begin = qbl;
    rows += ov;
    if (g) {
      const int nq = sp.fp8 ? B2Q<true> : B2Q<false>, nc = sp.fp8 ? B2C<true> : B2C<false>;
      b2t += (long long)((X + nq - 1) / nq) * ((RL + nc - 1) / nc);
      qbl += (long long)((X + 31) / 32) * ((ov + kColRows - 1) / kColRows);
    }
    w.sfd.push_back(s);
    off += L.total;
    if (ov == 0) continue;

    // V over rows (i,a) x (j,b), K = Q
    {
      SplitProb P{};
      P.kind = PK_V; P.frag = idx;
      P.M = P.N = ov; P.n_tile = NTv;
      P.tiles_m = (ov + SG_BM - 1) / SG_BM; P.tiles_n = (ov + NTv - 1) / NTv;
      P.ksplit = 1; P.k0_blocks = (X + BKv - 1) / BKv; P.k1_count = 1; P.k1_chunk = 1;
      P.a_mode = P.b_mode = TM_3D; P.div5 = 1;
      P.ea_rows = P.eb_rows = 1; P.ea_off = P.eb_off = s.erow;
      P.c_off = s.thi; P.c2_off = s.tlo; P.ldc = ldt; P.alpha = 1.0; P.vpad = vpadt;
      P.d_off = s.drow; P.vd_off = s.vdrow; P.et_off = s.scal + 4; P.v = v;
      P.group_m = kVGroupRows;
      P.ntiles = (long long)P.tiles_m * P.tiles_n;
      const uint64_t dims[3] = {(uint64_t)std::max(X, 1), (uint64_t)ov, (uint64_t)sv};
      const uint64_t str[2] = {(uint64_t)xpad * E2, (uint64_t)ov * xpad * E2};
      const uint32_t boxA[3] = {(uint32_t)BKv, SG_BM, (uint32_t)sv}, boxB[3] = {(uint32_t)BKv, (uint32_t)NTv, (uint32_t)sv};
      if (encode_tmap(&P.tmA, wsb + s.bs1, 3, dims, str, boxA, (int)E2) != RIMP2_OK ||
          encode_tmap(&P.tmB, wsb + s.bs1, 3, dims, str, boxB, (int)E2) != RIMP2_OK)
        return RIMP2_ERR_UNSUPPORTED;
      w.probs_v.push_back(P);
    }
    const uint64_t plane_b = (uint64_t)ov * ldd * E2;
    // P_ij / P_ab of small extents: slice-stacked tiles, one a side, or two in BF16 (up to 80
    // rows with 6 slices; three tiles of 40 x 40 rows then read less than a 128 x 64 tile or
    // two; FP8 at nocc = 42: 1.73 ms either way, so it stays in the launch it shares with
    // Gamma).  The contraction runs over k = (k1, k0) of 4-D views {k0, row, k1, slice}.
    auto stacked = [&](int kind, int n, const uint64_t* d4, const uint64_t* s4, int k0, int k1) -> int {
      const int most = sp.fp8 ? 1 : 2;
      int nb = 1;
      while (nb <= most && split_stack_rows(st, (n + nb - 1) / nb) == 0) ++nb;
      if (nb > most) return 0;
      SplitProb P{};
      P.kind = kind; P.frag = idx;
      P.M = P.N = n; P.n_tile = split_stack_rows(st, (n + nb - 1) / nb);
      P.tiles_m = P.tiles_n = nb;
      P.k0_blocks = (k0 + BKs - 1) / BKs; P.k1_count = k1;
      P.a_mode = P.b_mode = TM_4D; P.div5 = 1;
      P.ea_off = P.eb_off = s.scal + 4;
      P.ea_add = kTtAdd; P.eb_add = kTAdd;
      P.c_off = kind == PK_PAB ? f.pab_off : f.pij_off;
      P.ldc = n; P.alpha = kind == PK_PAB ? 1.0 : -1.0; P.sym = 1; P.ks_outer = 1;
      const uint32_t box[4] = {(uint32_t)BKs, (uint32_t)P.n_tile, 1, (uint32_t)st};
      if (encode_tmap(&P.tmA, wsb + s.tts, 4, d4, s4, box, (int)E2) != RIMP2_OK ||
          encode_tmap(&P.tmB, wsb + s.ts, 4, d4, s4, box, (int)E2) != RIMP2_OK)
        return -1;
      w.probs_s.push_back(P);
      return 1;
    };
    if (g) {  // Gamma[(i,a)][Q] = sum_(j,b) Tt[(i,a)][(j,b)] B[(j,b)][Q]
      SplitProb P{};
      P.kind = PK_GAMMA; P.frag = idx;
      P.M = ov; P.N = X; P.n_tile = NTg;
      P.tiles_m = (ov + SG_BM - 1) / SG_BM; P.tiles_n = (X + NTg - 1) / NTg;
      P.ksplit = 1; P.k0_blocks = (RL + BKg - 1) / BKg; P.k1_count = 1; P.k1_chunk = 1;
      P.a_mode = P.b_mode = TM_3D; P.div5 = 1;
      // K = (j,b) cut into slabs of about kGammaSlabK elements (split-K for large
      // fragments), slab index outermost: the tiles in flight share one slab, and the
      // tiles of a row start close together, which keeps their Tt rows in L2; the slabs
      // meet in Gamma by FP64 atomics.  Fewer, longer slabs mean fewer atomics and tile
      // switches, which measured faster down to two or three slabs.
      const int kb = P.k0_blocks;
      int slabs = sp.variant == 3 ? 1 : (int)(((long long)kb * BKg + kGammaSlabK / 2) / kGammaSlabK);
      if (slabs > 1) {
        const int per = (kb + slabs - 1) / slabs;
        slabs = (kb + per - 1) / per;
        P.k0_blocks = per; P.k1_count = slabs; P.ksplit = slabs;
        P.a_mode = P.b_mode = TM_3DK; P.div5 = per * BKg; P.ks_outer = 1;
        w.sfd.back().zero_gamma = 1;
      }
      // the leading s_g planes of Tt (one scale per fragment) and B with one scale per aux
      // index Q
      P.ea_rows = 0; P.ea_off = s.scal + 4; P.ea_add = kTtAdd;
      P.eb_rows = 1; P.eb_off = s.ecol; P.eb_add = 0;
      P.c_off = f.gamma_off; P.ldc = X; P.alpha = 1.0;
      P.ntiles = (long long)P.tiles_m * P.tiles_n * P.ksplit;
      const uint64_t dA[3] = {(uint64_t)RL, (uint64_t)ov, (uint64_t)s.st_out};
      const uint64_t sA[2] = {(uint64_t)ldd * E2, plane_b};
      const uint64_t dB[3] = {(uint64_t)RL, (uint64_t)X, (uint64_t)sgl};
      const uint64_t sB[2] = {(uint64_t)ldd * E2, (uint64_t)X * ldd * E2};
      const uint32_t boxA[3] = {(uint32_t)BKg, SG_BM, (uint32_t)sgl}, boxB[3] = {(uint32_t)BKg, (uint32_t)NTg, (uint32_t)sgl};
      if (encode_tmap(&P.tmA, wsb + s.tts, 3, dA, sA, boxA, (int)E2) != RIMP2_OK ||
          encode_tmap(&P.tmB, wsb + s.bs2, 3, dB, sB, boxB, (int)E2) != RIMP2_OK)
        return RIMP2_ERR_UNSUPPORTED;
      // with the slice count of P, Gamma joins P's launch
      (sgl == st ? w.probs_c : w.probs_g).push_back(P);
    }
    const uint64_t d4ab[4] = {(uint64_t)RL, (uint64_t)v, (uint64_t)o, (uint64_t)st};
    const uint64_t s4ab[3] = {(uint64_t)ldd * E2, (uint64_t)v * ldd * E2, plane_b};
    const int st_ab = f.pab_off >= 0 ? stacked(PK_PAB, v, d4ab, s4ab, RL, o) : 0;
    const uint64_t d4ij[4] = {(uint64_t)vpad, (uint64_t)o, (uint64_t)ov, (uint64_t)st};
    const uint64_t s4ij[3] = {(uint64_t)vpad * E2, (uint64_t)ldd * E2, plane_b};
    const int st_ij = f.pij_off >= 0 ? stacked(PK_PIJ, o, d4ij, s4ij, vpad, ov) : 0;
    if (st_ab < 0 || st_ij < 0) return RIMP2_ERR_UNSUPPORTED;
    if (f.pab_off >= 0 && !st_ab) {  // P_ab = sum_i sum_(j,c) Tt[(i,a)][(j,c)] T[(i,b)][(j,c)]
      SplitProb P{};
      P.kind = PK_PAB; P.frag = idx;
      P.M = P.N = v; P.n_tile = NTt;
      P.tiles_m = (v + SG_BM - 1) / SG_BM; P.tiles_n = (v + NTt - 1) / NTt;
      P.k0_blocks = (RL + BKt - 1) / BKt; P.k1_count = o;
      P.a_mode = P.b_mode = TM_4D; P.div5 = 1;
      P.ea_rows = P.eb_rows = 0; P.ea_off = P.eb_off = s.scal + 4;
      P.ea_add = kTtAdd; P.eb_add = kTAdd;
      P.c_off = f.pab_off; P.ldc = v; P.alpha = 1.0; P.sym = 1;
      choose_split_k(P, sp.grid, split_mul);
      // split index outermost: the tiles in flight share one range of i and so read the
      // same Tt_i / T_i rows; with it innermost, neighbours worked on different i and the
      // launch re-read its operands from DRAM (226 GB at nocc=100 nvir=500, 0.92 of HBM)
      P.ks_outer = 1;
      P.ntiles = (long long)P.tiles_m * P.tiles_n * P.ksplit;
      const uint32_t boxA[4] = {(uint32_t)BKt, SG_BM, 1, (uint32_t)st}, boxB[4] = {(uint32_t)BKt, (uint32_t)NTt, 1, (uint32_t)st};
      if (encode_tmap(&P.tmA, wsb + s.tts, 4, d4ab, s4ab, boxA, (int)E2) != RIMP2_OK ||
          encode_tmap(&P.tmB, wsb + s.ts, 4, d4ab, s4ab, boxB, (int)E2) != RIMP2_OK)
        return RIMP2_ERR_UNSUPPORTED;
      w.probs_c.push_back(P);
    }
    if (f.pij_off >= 0 && !st_ij && pij_direct) {  // P_ij = -sum_(k,a) sum_b Tt[(i,a)][(k,b)] T[(j,a)][(k,b)]
      SplitProb P{};
      P.kind = PK_PIJ; P.frag = idx;
      P.M = P.N = o; P.n_tile = NTt;
      P.tiles_m = (o + SG_BM - 1) / SG_BM; P.tiles_n = (o + NTt - 1) / NTt;
      P.k0_blocks = (vpad + BKt - 1) / BKt; P.k1_count = o * v;
      P.a_mode = P.b_mode = TM_5D; P.div5 = v;
      P.ea_rows = P.eb_rows = 0; P.ea_off = P.eb_off = s.scal + 4;
      P.ea_add = kTtAdd; P.eb_add = kTAdd;
      P.c_off = f.pij_off; P.ldc = o; P.alpha = -1.0; P.sym = 1;
      choose_split_k(P, sp.grid, split_mul);
      P.ks_outer = 1;   // as for P_ab: the tiles in flight share one (k,b) range
      P.ntiles = (long long)P.tiles_m * P.tiles_n * P.ksplit;
      const uint64_t d5[5] = {(uint64_t)vpad, (uint64_t)o, (uint64_t)v, (uint64_t)o, (uint64_t)st};
      const uint64_t s5[4] = {(uint64_t)vpad * E2, (uint64_t)ldd * E2, (uint64_t)v * ldd * E2, plane_b};
      const uint32_t boxA[5] = {(uint32_t)BKt, 1, 1, SG_BM, (uint32_t)st}, boxB[5] = {(uint32_t)BKt, 1, 1, (uint32_t)NTt, (uint32_t)st};
      if (encode_tmap(&P.tmA, wsb + s.tts, 5, d5, s5, boxA, (int)E2) != RIMP2_OK ||
          encode_tmap(&P.tmB, wsb + s.ts, 5, d5, s5, boxB, (int)E2) != RIMP2_OK)
        return RIMP2_ERR_UNSUPPORTED;
      w.probs_c.push_back(P);
    } else if (f.pij_off >= 0 && !st_ij) {
      // P_ij through the pair symmetry Tt_ik(a,b) = Tt_ki(b,a):
      // P_ij = -sum_(k,b) sum_a Tt[(k,b)][(i,a)] T[(k,b)][(j,a)]; the rows i of one
      // (k,b) row are vpad elements apart, so a 128-row TMA box reads one contiguous span
      SplitProb P{};
      P.kind = PK_PIJ; P.frag = idx;
      P.M = P.N = o; P.n_tile = NTt;
      P.tiles_m = (o + SG_BM - 1) / SG_BM; P.tiles_n = (o + NTt - 1) / NTt;
      P.k0_blocks = (vpad + BKt - 1) / BKt; P.k1_count = o * v;
      P.a_mode = P.b_mode = TM_4D; P.div5 = 1;
      P.ea_rows = P.eb_rows = 0; P.ea_off = P.eb_off = s.scal + 4;
      P.ea_add = kTtAdd; P.eb_add = kTAdd;
      P.c_off = f.pij_off; P.ldc = o; P.alpha = -1.0; P.sym = 1;
      choose_split_k(P, sp.grid, split_mul);
      P.ks_outer = 1;   // as for P_ab: the tiles in flight share one (k,b) range
      P.ntiles = (long long)P.tiles_m * P.tiles_n * P.ksplit;
      const uint32_t boxA[4] = {(uint32_t)BKt, SG_BM, 1, (uint32_t)st}, boxB[4] = {(uint32_t)BKt, (uint32_t)NTt, 1, (uint32_t)st};
      if (encode_tmap(&P.tmA, wsb + s.tts, 4, d4ij, s4ij, boxA, (int)E2) != RIMP2_OK ||
          encode_tmap(&P.tmB, wsb + s.ts, 4, d4ij, s4ij, boxB, (int)E2) != RIMP2_OK)
        return RIMP2_ERR_UNSUPPORTED;
      w.probs_c.push_back(P);
    }
  }
  // A split-K piece of P_ab / P_ij spans at least kMinPieceK elements of K: the per-problem
  // target (a multiple of the grid, for locality at large sizes) would otherwise cut the
  // P_ij of small fragments, K0 = nvir per outer index, into pieces whose drain, epilogue
  // and atomics cost as much as their MMAs.  A launch whose pieces would not fill the grid
  // twice takes shorter ones, down to one accumulation chunk.
  {
    double work = 0.0;
    for (const auto& P : w.probs_c) work += (double)P.tiles_m * P.tiles_n * P.k1_count * P.k0_blocks * BKt;
    const long long least = std::max<long long>(512, std::min<long long>(kMinPieceK, (long long)(work / (2.0 * sp.grid))));
    for (auto& P : w.probs_c)
      if (P.kind == PK_PAB || P.kind == PK_PIJ) {
        const long long per = (long long)P.k0_blocks * BKt;   // K elements per outer index
        const int chunk = (int)std::min<long long>(P.k1_count, (least + per - 1) / per);
        if (P.k1_chunk < chunk) {
          P.k1_chunk = chunk;
          P.ksplit = std::max(1, (P.k1_count + chunk - 1) / chunk);
          P.ntiles = (long long)P.tiles_m * P.tiles_n * P.ksplit;
        }
      }
  }
  // Slice-stacked pieces: eight per SM over the launch, at least eight stages each
  {
    double stages = 0.0;
    auto tri = [](const SplitProb& P) { return (long long)P.tiles_m * (P.tiles_m + 1) / 2; };
    for (const auto& P : w.probs_s) stages += (double)tri(P) * P.k1_count * P.k0_blocks;
    const double piece = std::max(8.0, stages / (8.0 * sp.grid));
    w.stack_rows = 0;
    for (auto& P : w.probs_s) {
      P.k1_chunk = (int)std::min<double>(P.k1_count, std::max(1.0, std::ceil(piece / P.k0_blocks)));
      P.ksplit = std::max(1, (P.k1_count + P.k1_chunk - 1) / P.k1_chunk);
      P.ntiles = tri(P) * P.ksplit;
      w.stack_rows = std::max(w.stack_rows, P.n_tile);
    }
  }
  // A Gamma launch of few tiles is cut along K as well, in two (at least four stages a slab):
  // 0 + x + y is the same in either order, so Gamma's bits do not depend on which slab ends
  // first, which three slabs would not give
  {
    long long tiles = 0;
    for (const auto& P : w.probs_g) tiles += P.ntiles;
    const int want = tiles > 0 && sp.variant != 3 ? (int)std::min<long long>(2, sp.grid / tiles) : 1;
    for (auto& P : w.probs_g) {
      const int slabs = std::min(want, P.k0_blocks / 4);
      if (P.k1_count != 1 || slabs < 2) continue;
      const int per = (P.k0_blocks + slabs - 1) / slabs;
      P.k1_count = P.ksplit = (P.k0_blocks + per - 1) / per;
      P.k0_blocks = per;
      P.a_mode = P.b_mode = TM_3DK; P.div5 = per * BKg; P.ks_outer = 1;
      P.ntiles *= P.ksplit;
      for (auto& d : w.sfd)
        if (d.idx == P.frag) d.zero_gamma = 1;
    }
  }
  w.max_x = 0;
  for (const auto& f : w.sfd) w.max_x = std::max(w.max_x, f.X);
  // Amplitude stage: CTAs (i, j range, strip).  One range of all j where the strips alone make
  // eight rounds of three CTAs per SM (a shorter last round costs less of the whole); shorter
  // ranges, down to one j, for smaller waves
  w.amp_lpr = amp_lanes(w.sfd, sp.fp8);
  {
    const int R = 8 * (32 / w.amp_lpr);
    auto strips = [&](const SplitFragDev& s) { return (long long)std::max(1, (s.v + R - 1) / R); };
    long long ctas = 0;
    for (const auto& s : w.sfd) ctas += s.o * strips(s);
    const long long split = ctas > 0 ? (24LL * sp.grid + ctas - 1) / ctas : 1;
    for (auto& s : w.sfd) {
      s.amp_jchunk = std::max(1, (int)((s.o + split - 1) / split));
      s.pair_begin = pairs;
      pairs += (long long)s.o * strips(s) * ((s.o + s.amp_jchunk - 1) / s.amp_jchunk);
    }
  }
  total_pairs = pairs;
  w.rows = rows;
  w.b2_tiles = b2t;
  w.qblks = qbl;
  w.sep_energy = !w.probs_c.empty() || !w.probs_s.empty() || !w.probs_g.empty();
  for (const auto& d : w.sfd) w.sep_energy = w.sep_energy && d.o <= kSepOcc;
  finish(w.probs_v, w.tiles_v);
  finish(w.probs_c, w.tiles_c);
  finish(w.probs_g, w.tiles_g);
  finish(w.probs_s, w.tiles_s);
  // every problem's tiles and TMA boxes must match the kernel instance of its launch
  auto same_shape = [](const std::vector<SplitProb>& v, const SplitLaunch& c) {
    for (const auto& P : v)
      if (P.n_tile != c.n_tile_max) return false;
    return true;
  };
  if (!same_shape(w.probs_v, w.cfg_v) || !same_shape(w.probs_c, sp.cfg_t) ||
      !same_shape(w.probs_g, sp.cfg_g))
    return RIMP2_ERR_UNSUPPORTED;
  w.mma_v = w.mma_c = w.mma_g = 0.0;
  for (const auto& P : w.probs_v) w.mma_v += prob_mma_flops(P, sv, BKv);
  for (const auto& P : w.probs_c) w.mma_c += prob_mma_flops(P, st, BKt);
  for (const auto& P : w.probs_g) w.mma_g += prob_mma_flops(P, sgl, BKg);
  for (const auto& P : w.probs_s) {   // 128 rows x the accumulator columns of both row groups
    const int R = P.n_tile, n0 = (st * R + 15) / 16 * 16;
    const int n1 = st * R <= 128 ? 0 : ((st - 128 / R) * R + 15) / 16 * 16;
    w.mma_c += 2.0 * SG_BM * (n0 + n1) * (double)P.k1_count * P.k0_blocks * BKs * (P.tiles_m * (P.tiles_m + 1) / 2);
  }
  return RIMP2_OK;
}

size_t split_layout_wave(SplitWave& w, size_t off) {
  off = al256(off);
  w.off_sfd = off; off = al256(off + w.sfd.size() * sizeof(SplitFragDev));
  w.off_pv = off; off = al256(off + w.probs_v.size() * sizeof(SplitProb));
  w.off_pc = off; off = al256(off + w.probs_c.size() * sizeof(SplitProb));
  w.off_pg = off; off = al256(off + w.probs_g.size() * sizeof(SplitProb));
  w.off_ps = off; off = al256(off + w.probs_s.size() * sizeof(SplitProb));
  w.off_bv = off; off = al256(off + w.probs_v.size() * sizeof(long long));
  w.off_bc = off; off = al256(off + w.probs_c.size() * sizeof(long long));
  w.off_bg = off; off = al256(off + w.probs_g.size() * sizeof(long long));
  w.off_bs = off; off = al256(off + w.probs_s.size() * sizeof(long long));
  return off;
}

void split_fill_wave(const SplitWave& w, char* host) {
  if (!w.sfd.empty()) memcpy(host + w.off_sfd, w.sfd.data(), w.sfd.size() * sizeof(SplitFragDev));
  if (!w.probs_v.empty()) memcpy(host + w.off_pv, w.probs_v.data(), w.probs_v.size() * sizeof(SplitProb));
  if (!w.probs_c.empty()) memcpy(host + w.off_pc, w.probs_c.data(), w.probs_c.size() * sizeof(SplitProb));
  if (!w.probs_g.empty()) memcpy(host + w.off_pg, w.probs_g.data(), w.probs_g.size() * sizeof(SplitProb));
  if (!w.probs_s.empty()) memcpy(host + w.off_ps, w.probs_s.data(), w.probs_s.size() * sizeof(SplitProb));
  auto begins = [&](const std::vector<SplitProb>& v, size_t off) {
    for (size_t k = 0; k < v.size(); ++k) {
      const long long b = v[k].tile_begin;
      memcpy(host + off + k * sizeof(long long), &b, sizeof(b));
    }
  };
  begins(w.probs_v, w.off_bv);
  begins(w.probs_c, w.off_bc);
  begins(w.probs_g, w.off_bg);
  begins(w.probs_s, w.off_bs);
}

int split_enqueue_wave(SplitPlan& sp, SplitWave& w, char* dblk, int nf, long long total_pairs,
                       Bases bs, int check, unsigned* ctr, cudaStream_t s, int* launches,
                       long long* tiles, cudaEvent_t* ev) {
  const SplitFragDev* sfd = (const SplitFragDev*)(dblk + w.off_sfd);
  int nl = 0;
  cudaError_t e = cudaSuccess;
  if (nf > 0) {
    k_split_prologue<<<(unsigned)nf, 256, 0, s>>>(sfd, ctr, check, bs);
    ++nl;
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && w.rows > 0) {
    const unsigned rb = (unsigned)((w.rows + 7) / 8), blocks = rb + (unsigned)w.qblks;
    auto b1 = [&](auto kernel) { kernel<<<blocks, 256, 0, s>>>(sfd, nf, w.rows, rb, sp.slices_v, check, bs); };
    if (w.max_x <= 256) sp.fp8 ? b1(k_slice_b1<true, 2>) : b1(k_slice_b1<false, 2>);
    else sp.fp8 ? b1(k_slice_b1<true, 0>) : b1(k_slice_b1<false, 0>);
    ++nl;
    e = cudaGetLastError();
  }
  if (ev) cudaEventRecordWithFlags(ev[1], s, cudaEventRecordExternal);
  if (e == cudaSuccess && w.tiles_v > 0) {
    e = launch_split_gemm((const SplitProb*)(dblk + w.off_pv), (const long long*)(dblk + w.off_bv),
                          (int)w.probs_v.size(), w.tiles_v, bs,
                          ctr + 0, w.cfg_v, sp.grid, s);
    ++nl;
  }
  if (ev) cudaEventRecordWithFlags(ev[2], s, cudaEventRecordExternal);
  if (e == cudaSuccess && total_pairs > 0) {
    const unsigned ctas = (unsigned)total_pairs;
    auto amp = [&](auto kernel) {
      kernel<<<ctas + (unsigned)w.b2_tiles, 256, 0, s>>>(sfd, nf, ctas, sp.slices_g, !w.sep_energy, bs);
    };
    switch (w.amp_lpr) {
      case 8: sp.fp8 ? amp(k_amp_split<true, 8>) : amp(k_amp_split<false, 8>); break;
      case 16: sp.fp8 ? amp(k_amp_split<true, 16>) : amp(k_amp_split<false, 16>); break;
      default: sp.fp8 ? amp(k_amp_split<true, 32>) : amp(k_amp_split<false, 32>); break;
    }
    ++nl;
    e = cudaGetLastError();
    if (e == cudaSuccess && w.sep_energy) {
      if (sp.fp8) k_split_energy<true><<<(unsigned)nf, 256, 0, s>>>(sfd, w.amp_lpr, bs);
      else k_split_energy<false><<<(unsigned)nf, 256, 0, s>>>(sfd, w.amp_lpr, bs);
      ++nl;
      e = cudaGetLastError();
    }
  }
  if (ev) cudaEventRecordWithFlags(ev[3], s, cudaEventRecordExternal);
  // The P launches and Gamma's read what the amplitude launch wrote and nothing of each other:
  // the next one's CTAs take the SMs that the one before leaves (at nocc=10 nvir=40 all 134 CTAs
  // of both run at once).  Events between the launches keep them apart.
  bool beside = !ev && w.sep_energy;
  if (e == cudaSuccess && w.tiles_c > 0) {
    SplitLaunch cfg = sp.cfg_t;
    cfg.beside = beside;
    e = launch_split_gemm((const SplitProb*)(dblk + w.off_pc), (const long long*)(dblk + w.off_bc),
                          (int)w.probs_c.size(), w.tiles_c, bs,
                          ctr + 1, cfg, sp.grid, s);
    beside = !ev;
    ++nl;
  }
  if (e == cudaSuccess && w.tiles_s > 0) {
    e = launch_split_stack((const SplitProb*)(dblk + w.off_ps), (const long long*)(dblk + w.off_bs),
                           (int)w.probs_s.size(), w.tiles_s, bs, ctr + 3, sp.slices_t, w.stack_rows,
                           sp.fp8, sp.grid, beside, s);
    beside = !ev;
    ++nl;
  }
  if (ev) cudaEventRecordWithFlags(ev[4], s, cudaEventRecordExternal);
  if (e == cudaSuccess && w.tiles_g > 0) {
    SplitLaunch cfg = sp.cfg_g;
    cfg.beside = beside;
    e = launch_split_gemm((const SplitProb*)(dblk + w.off_pg), (const long long*)(dblk + w.off_bg),
                          (int)w.probs_g.size(), w.tiles_g, bs,
                          ctr + 2, cfg, sp.grid, s);
    ++nl;
  }
  if (ev) cudaEventRecordWithFlags(ev[5], s, cudaEventRecordExternal);
  *launches = nl;
  *tiles = w.tiles_v + w.tiles_c + w.tiles_g + w.tiles_s;
  return e == cudaSuccess ? RIMP2_OK : RIMP2_ERR_CUDA;
}

}  // namespace rimp2
