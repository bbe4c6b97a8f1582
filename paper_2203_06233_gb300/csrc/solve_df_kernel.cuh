// The weight solve in double-float arithmetic: the same steps as solve.cu's
// FP64 kernels (load, Rl = Lu Dg Lu^H, solve, refine, normalise),
//   delta = lf Re tr(R) / D,  Rl = R + delta I,  u = Rl^{-1} v,
//   u += Rl^{-1} (v - Rl u)  refine_steps times,  w = u / sqrt(Re v^H u),
// with every FP64 value replaced by an unevaluated sum of two floats and
// every sum compensated, on the FP32 pipe.
//
// Why.  GB300 runs FP64 at 1/62 of the FP32 rate: a complex multiply-add of a
// warp holds the SM's FP64 pipe for 64 cycles, while the 48 FP32
// instructions of its double-float form take the four schedulers 12.  The
// FP64 kernels were at 65-80% of that FP64 bound, i.e. at their floor, and the
// solve was 95% of a D = 64 or D = 128 CPI.
//
// Arithmetic.  A real multiply-add is the Dot2 step of Ogita, Rump and Oishi
// ("Accurate sum and dot product", SISC 2005) with double-float factors: the
// product of the high parts split exactly by an FMA, the running sum by
// Knuth's TwoSum, every rounding error and the cross terms collected in a
// second float; the pair is renormalised every LR columns, so the collected
// errors stay small against the sum.  Relative to the terms' running sums
// that is about 2^-44, against FP64's 2^-50 over as many terms.  Where a bound
// on the partial sums is known and close, the sum runs on a fixed grid at half
// the instructions (gmac): from D = 33 on, the factorisation (an entry's sums
// stay below sqrt(Rl_ii Rl_ll)) and the substitutions' blocks off the diagonal
// (|x| + max |l| sum |y|, formed per row and block).  Not the residual: its only
// cheap bound, sqrt(Rl_ii) sum sqrt(Rl_jj) |u_j|, is far above the sums where
// the solutions of the separable basis cancel (measured: one system in eight
// 3.6e-6 off instead of 2.9e-8), though it would be a third faster.
//
// Where it may stand in for FP64.  The weights are stored as complex64
// (2^-25), and the error of a right-hand side's solution is at most kappa(Rl)
// times the arithmetic's.  For a covariance (R positive semidefinite) the load
// bounds kappa <= D / lf + 1, so launch_solve takes these kernels when that bound
// is at most kDfMaxKappa = 2^19 (the default load 1e-3 gives 1.28e5 at D = 128;
// see solve_df_eligible for plans without refinement) and the FP64 kernels for
// weaker loads, where nothing bounds kappa.  Two things are outside of that
// argument and are looked at per system: a combination of basis solutions that
// cancels (combine) and, in stap_solve_weights, a matrix that is no covariance
// (kAnyMatrix).  The measured weights are then as far from the 64-bit ones as
// their complex64 rounding, 2.5e-8 normwise, at the default and at the weakest
// accepted load, for 0 to 80 dB of interference, along beams or not.
//
// Range.  Floats span 2^+-126 only, so each system is scaled by the even
// power of two 2^-e that brings Rl's trace into [1, 4): the conversion from
// FP64 adds -e to the exponent field (no instruction more), and the weights
// take 2^(-e/2) back with their normalisation.  Entries below 2^-73 of the
// trace become zero; an infinity or NaN becomes a NaN, which no pivot test
// passes.
//
// Layout.  A system belongs to a team of TEAM threads: half a warp, a warp or, of
// few, 128 threads (D <= 16), a CTA of 64, 128 (D <= 32), 256 (D <= 64) or 512 (D <=
// 128) threads.
// LR lanes hold one right-hand side, row li + LR q in register q < RPL.  The
// factor (column-major packed) and the solutions stay in shared memory, the
// column's entry is broadcast by shuffles, so a 16-byte read feeds one complex
// multiply-add of 48 FP32 instructions.  The residual's Rl comes from the
// input again, in chunks of KC columns that the team converts once for all its
// right-hand sides (the FP64 kernel read each entry from global memory for
// every right-hand side).  Sixteen warps of 128 registers per SM at D = 128
// issued 74% of the slots against 62% for eight warps of 255 with two
// right-hand sides per thread; packed FP32 pairs (FFMA2) of two right-hand
// sides, or of real and imaginary part, needed so many moves to form the pairs
// that they were no faster.  With the grids a warp per right-hand side is the
// faster split at D > 96 (2048 systems of 128 rows: half a warp 10230 us, a warp
// 9470; without grids 10820, 10890), half a warp below (96 rows: 4958, 5540).
//
// Measured (GB300; the FP64 kernels, double-float without grids, with them, as it
// is: with the look at combinations that cancel and, being the step, the check
// of any matrix and its second launch of 3.5 us), us:
//   D = 128, 16384 systems, C 32 S 64    266533, 82470, 71420, 74020
//   D =  64, 8192 systems,  C 16 S 32     15859,  5403,  5234,  5410
//   D =  15, 3840 systems,  C 5  S 11       258,   117 (no grids), 124
//   D =  12, 16384 systems, C 4  S 16       324,   160 (no grids), 164
//   D =  12, 256 systems,   C 4  S 4      103.5,    21 (no grids),  23
// What bounds it at D = 128: issue, 72% of the slots in use by four warps per
// scheduler (shared memory holds one system per SM), the sums' own
// instructions a third of all slots; masked lanes of the diagonal blocks,
// renormalisations, the shuffles that broadcast a column's entry and the loads
// take the rest.
//
// kMixedIr (STAP_SOLVE_MIXED_IR): the factor and the substitutions in FP32, the
// residual and the solution in double-float as above.
#pragma once

#include "df64.cuh"
#include "batch.cuh"
#include "checked.cuh"
#include "snapshots.cuh"
#include "solve_df.cuh"

namespace stap {
namespace {

constexpr int KC = 8;   // columns of Rl per residual chunk

// Which solve a kernel is: double-float throughout of a covariance; the same of
// any Hermitian matrix, marking what it cannot answer for (kernels of their own,
// as the marking costs the others 2 to 3%); the refinement option.
constexpr int kCovariance = 0, kAnyMatrix = 1, kMixedIr = 2;
__host__ __device__ constexpr bool f32f(int mode) { return mode == kMixedIr; }   // FP32 factor

// Whether the factorisation and the substitutions' off-diagonal blocks run on
// grids: from D = 33 on.
template <int TEAM, int MODE>
__host__ __device__ constexpr bool grids() { return !f32f(MODE) && TEAM >= 256; }

// One complex value: running sums (rs, is) and the errors collected beside
// them (re, ie); in shared memory (re hi, im hi, re lo, im lo).
struct Cdf {
  float rs, re, is, ie;
};
__device__ __forceinline__ float4 pack(const Cdf& x) { return make_float4(x.rs, x.is, x.re, x.ie); }
__device__ __forceinline__ Cdf unpack(float4 v) { return Cdf{v.x, v.z, v.y, v.w}; }
__device__ __forceinline__ float4 conj4(float4 v) { return make_float4(v.x, -v.y, v.z, -v.w); }

// s + e += (ah + al) (bh + bl), dropping al bl (below 2^-48 of the product)
__device__ __forceinline__ void mac(float& s, float& e, float ah, float al, float bh, float bl) {
  const float p = __fmul_rn(ah, bh);
  float pe = __fmaf_rn(ah, bh, -p);
  pe = __fmaf_rn(ah, bl, pe);
  pe = __fmaf_rn(al, bh, pe);
  const float t = __fadd_rn(s, p);
  const float z = __fsub_rn(t, s);
  const float te = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z));
  s = t;
  e = __fadd_rn(e, __fadd_rn(te, pe));
}

// renormalise: |lo| <= ulp(hi) / 2 (the collected errors are smaller than the sum)
__device__ __forceinline__ void norm2(float& s, float& e) {
  const ff::F2 t = ff::fast_two_sum(s, e);
  s = t.hi;
  e = t.lo;
}
__device__ __forceinline__ void norm(Cdf& x) {
  norm2(x.rs, x.re);
  norm2(x.is, x.ie);
}
// x -= l y
__device__ __forceinline__ void cms(Cdf& x, float4 l, float4 y) {
  mac(x.rs, x.re, -l.x, -l.z, y.x, y.z);
  mac(x.is, x.ie, -l.x, -l.z, y.y, y.w);
  mac(x.rs, x.re, l.y, l.w, y.y, y.w);
  mac(x.is, x.ie, -l.y, -l.w, y.x, y.z);
}

// A sum whose partial sums a bound M is known for runs from sig = 3 P, P the
// power of two above M, instead of from zero: it stays in (2 P, 4 P), where
// floats have one spacing, 2^-22 P, so that t - s is exact and no TwoSum is
// needed: 6 instructions instead of 12 per real product.  What rounds: the rest
// a b - (t - s), at most half a spacing, to 24 bits of itself (2^-47 P), the two
// cross terms on top of it likewise, and the sum e of the rests, which after n
// terms may have grown to n half spacings.  That is below n (3 + n / 2) 2^-47 P,
// and as the roundings are independent about 2^-46 M for the n in question --
// of the bound M, where the TwoSum form is about 2^-47 of the running sums:
// the grid is for sums whose bound is close.
__device__ __forceinline__ void gmac(float& s, float& e, float ah, float al, float bh, float bl) {
  const float t = __fmaf_rn(ah, bh, s);
  float q = __fmaf_rn(ah, bh, __fsub_rn(s, t));
  q = __fmaf_rn(ah, bl, q);
  q = __fmaf_rn(al, bh, q);
  s = t;
  e = __fadd_rn(e, q);
}
__device__ __forceinline__ void gcms(Cdf& x, float4 l, float4 y) {
  gmac(x.rs, x.re, -l.x, -l.z, y.x, y.z);
  gmac(x.is, x.ie, -l.x, -l.z, y.y, y.w);
  gmac(x.rs, x.re, l.y, l.w, y.y, y.w);
  gmac(x.is, x.ie, -l.y, -l.w, y.x, y.z);
}
__device__ __forceinline__ float sigma(float m) {
  return __fmul_rn(__uint_as_float(__float_as_uint(m) & 0x7F800000u), 6.f);
}
// onto sig's grid, the rest of s to e; and back (normalised)
__device__ __forceinline__ void bias2(float& s, float& e, float sig) {
  const float t = __fadd_rn(s, sig);
  e = __fadd_rn(e, __fsub_rn(s, __fsub_rn(t, sig)));
  s = t;
}
__device__ __forceinline__ void unbias2(float& s, float& e, float sig) {
  norm2(s, e);                       // |e| <= spacing / 2: the difference is 0 or larger
  s = __fsub_rn(s, sig);
  norm2(s, e);
}
__device__ __forceinline__ void bias(Cdf& x, float sig) {
  bias2(x.rs, x.re, sig);
  bias2(x.is, x.ie, sig);
}
__device__ __forceinline__ void unbias(Cdf& x, float sig) {
  unbias2(x.rs, x.re, sig);
  unbias2(x.is, x.ie, sig);
}

// a b of two normalised double-floats
__device__ __forceinline__ ff::F2 mul2(float ah, float al, float bh, float bl) {
  const float p = __fmul_rn(ah, bh);
  float e = __fmaf_rn(ah, bh, -p);
  e = __fmaf_rn(ah, bl, e);
  e = __fmaf_rn(al, bh, e);
  return ff::fast_two_sum(p, e);
}
__device__ __forceinline__ Cdf scale(const Cdf& x, ff::F2 r) {
  const ff::F2 a = mul2(x.rs, x.re, r.hi, r.lo), b = mul2(x.is, x.ie, r.hi, r.lo);
  return Cdf{a.hi, a.lo, b.hi, b.lo};
}
// u + v, normalised
__device__ __forceinline__ Cdf add(const Cdf& u, const Cdf& v) {
  const ff::F2 a = ff::add2({u.rs, u.re}, {v.rs, v.re}), b = ff::add2({u.is, u.ie}, {v.is, v.ie});
  return Cdf{a.hi, a.lo, b.hi, b.lo};
}

// 1 / d: from the hardware's approximate reciprocal r of the high part, with
// e = 1 - d r (about 2^-23) the series r (1 + e + e^2) leaves e^3
__device__ __forceinline__ ff::F2 recip(ff::F2 d) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d.hi));
  float e = __fmaf_rn(-d.hi, r, 1.f);
  e = __fmaf_rn(-d.lo, r, e);
  return ff::fast_two_sum(r, __fmul_rn(r, __fmaf_rn(e, e, e)));
}

// x 2^-e as hi + lo by its IEEE fields (integer instructions: a conversion
// instruction would hold the FP64 pipe): hi = the top 24 bits, lo = the other
// 29 rounded to a float, both with x's sign.  `base` = 896 + e.  Below 2^-73:
// zero; beyond float range or not finite: NaN.
__device__ __forceinline__ ff::F2 split(double x, int base) {
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
  const int E = (int)((h >> 20) & 0x7FF) - base;   // biased float exponent
  const uint32_t sign = h & 0x80000000u;
  if (E <= 53) return {0.f, 0.f};
  if (E >= 255 || (h & 0x7FF00000u) == 0x7FF00000u) return {__int_as_float(0x7FC00000), 0.f};
  const float hi = __uint_as_float(sign | ((uint32_t)E << 23) | ((h & 0xFFFFFu) << 3) | (l >> 29));
  const float lo = __fmul_rn((float)(l & 0x1FFFFFFFu), __uint_as_float((uint32_t)(E - 52) << 23));
  return {hi, __uint_as_float(__float_as_uint(lo) | sign)};
}
__device__ __forceinline__ float4 split(double2 a, int base) {
  const ff::F2 r = split(a.x, base), i = split(a.y, base);
  return make_float4(r.hi, i.hi, r.lo, i.lo);
}

__device__ __forceinline__ int cstart(int l, int D) { return l * D - l * (l - 1) / 2; }

// The weights' factor 2^h / sqrt(q) (h = -e/2 undoes the system's scale): the
// double-float 1 / sqrt(q), from the approximate r by r (1 + (1 - q r^2) / 2),
// times the part of 2^h that floats hold surely; `rest` the exponent left
// over (zero but for traces beyond 2^+-200).
struct Gain {
  float hi, lo;
  int rest;
};
__device__ __forceinline__ Gain gain(ff::F2 q, int h) {
  const float r = rsqrtf(q.hi);
  const float p = __fmul_rn(r, r), pl = __fmaf_rn(r, r, -p);
  float e = __fmaf_rn(-q.hi, p, 1.f);
  e = __fmaf_rn(-q.hi, pl, e);
  e = __fmaf_rn(-q.lo, p, e);
  const ff::F2 g = ff::fast_two_sum(r, __fmul_rn(r, __fmul_rn(0.5f, e)));
  const int hc = max(-100, min(100, h));
  const float sc = __uint_as_float((uint32_t)(127 + hc) << 23);
  return {__fmul_rn(g.hi, sc), __fmul_rn(g.lo, sc), h - hc};
}
// (re, im) times that, rounded once
__device__ __forceinline__ float2 weight(ff::F2 re, ff::F2 im, const Gain& g, bool good) {
  if (!good) return make_float2(0.f, 0.f);
  float2 w = make_float2(mul2(re.hi, re.lo, g.hi, g.lo).hi, mul2(im.hi, im.lo, g.hi, g.lo).hi);
  if (g.rest != 0) w = make_float2(ldexpf(w.x, g.rest), ldexpf(w.y, g.rest));
  return w;
}
// sum of s + e over W lanes, the same in all of them
template <int W>
__device__ __forceinline__ ff::F2 lanes_sum2(float s, float e) {
  for (int o = W / 2; o > 0; o >>= 1) {
    const ff::F2 t = ff::two_sum(s, __shfl_xor_sync(0xffffffffu, s, o));
    e = __fadd_rn(__fadd_rn(e, __shfl_xor_sync(0xffffffffu, e, o)), t.lo);
    s = t.hi;
  }
  return ff::fast_two_sum(s, e);
}
__device__ __forceinline__ bool usable(ff::F2 q) { return q.hi > 0.f && isfinite(q.hi); }

template <int W>
__device__ __forceinline__ float lanes_max(float v) {
  for (int o = W / 2; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

template <int W>
__device__ __forceinline__ double lanes_sum(double v) {
  for (int o = W / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// In-place forward (Lu z = x) or back (Lu^H z = x) substitution of the vector
// that the LR lanes of a group hold (row li + LR q in x[q]).  The columns go
// in blocks of LR (block qb's columns live in x[qb], a shuffle broadcasts the
// column's entry), and only the row blocks that a block's columns update are
// visited, with the block indices compile-time constants.  Only the diagonal
// block decides per lane; rows past D read whatever lies after their column
// (inside the team's shared memory) into registers that nothing reads.
template <int LR, int RPL, bool BACK, bool GRID>
__device__ __forceinline__ void subst(Cdf (&x)[RPL], const float4* L, const float* lmax, int D, int li, int gbase) {
#pragma unroll
  for (int bb = 0; bb < RPL; ++bb) {
    const int qb = BACK ? RPL - 1 - bb : bb;
    if (LR * qb >= D) continue;                           // team-uniform
    const int jn = min(LR, D - LR * qb);
    // forward: column j's entries start at cstart(j) - j + i; back: row j of
    // column i = li + LR q lies at cstart(i) - i + j, which is b0 + b1 q -
    // q^2 LR^2 / 2 + j
    const int b0 = li * D - li * (li - 1) / 2 - li, b1 = LR * D - LR * li - LR / 2;
#pragma unroll (LR >= 16 ? 2 : 1)
    for (int jj = 0; jj < jn; ++jj) {
      const int jo = BACK ? jn - 1 - jj : jj;
      const int j = LR * qb + jo;
      norm(x[qb]);
      const Cdf y{__shfl_sync(0xffffffffu, x[qb].rs, gbase + jo), __shfl_sync(0xffffffffu, x[qb].re, gbase + jo),
                  __shfl_sync(0xffffffffu, x[qb].is, gbase + jo), __shfl_sync(0xffffffffu, x[qb].ie, gbase + jo)};
      const float4* cj = L + cstart(j, D) - j + li;
#pragma unroll
      for (int q = 0; q < RPL; ++q) {
        if (GRID ? q != qb : (BACK ? (q > qb) : (q < qb))) continue;   // compile-time
        if (LR * q >= D) continue;                        // team-uniform
        float4 l = make_float4(0.f, 0.f, 0.f, 0.f);
        if (q != qb || (BACK ? li < jo : (li > jo && li + LR * q < D)))
          l = BACK ? conj4(L[b0 + j + b1 * q - q * q * (LR * LR / 2)]) : cj[LR * q];
        cms(x[q], l, pack(y));
      }
    }
    if constexpr (!GRID) {
#pragma unroll
      for (int q = 0; q < RPL; ++q)
        if (BACK ? q < qb : q > qb) norm(x[q]);
    } else if (BACK ? qb > 0 : LR * (qb + 1) < D) {
      // the block's entries are final: the other rows on a grid whose bound is
      // |x| + max |l| sum |y|
      norm(x[qb]);
      float ys = li < jn ? fabsf(x[qb].rs) + fabsf(x[qb].is) : 0.f;
#pragma unroll
      for (int o = LR / 2; o > 0; o >>= 1) ys += __shfl_xor_sync(0xffffffffu, ys, o);
      ys *= 1.001f;
      float sig[RPL];
#pragma unroll
      for (int q = 0; q < RPL; ++q) {
        if (BACK ? q >= qb : q <= qb) continue;
        if (LR * q >= D) continue;
        const int i = min(li + LR * q, D - 1);
        sig[q] = sigma(fmaf(lmax[(BACK ? RPL + qb : qb) * D + i], ys, fmaxf(fabsf(x[q].rs), fabsf(x[q].is))));
        bias(x[q], sig[q]);
      }
#pragma unroll (LR * RPL > 64 ? 2 : 1)
      for (int jo = 0; jo < jn; ++jo) {
        const int j = LR * qb + jo;
        const Cdf y{__shfl_sync(0xffffffffu, x[qb].rs, gbase + jo), __shfl_sync(0xffffffffu, x[qb].re, gbase + jo),
                    __shfl_sync(0xffffffffu, x[qb].is, gbase + jo), __shfl_sync(0xffffffffu, x[qb].ie, gbase + jo)};
        const float4* cj = L + cstart(j, D) - j + li;
#pragma unroll
        for (int q = 0; q < RPL; ++q) {
          if (BACK ? q >= qb : q <= qb) continue;
          if (LR * q >= D) continue;
          gcms(x[q], BACK ? conj4(L[b0 + j + b1 * q - q * q * (LR * LR / 2)]) : cj[LR * q], pack(y));
        }
      }
#pragma unroll
      for (int q = 0; q < RPL; ++q) {
        if (BACK ? q >= qb : q <= qb) continue;
        if (LR * q >= D) continue;
        unbias(x[q], sig[q]);
      }
    }
  }
}

// x <- Rl^{-1} x with Rl = Lu Dg Lu^H (rd: the pivot reciprocals).
template <int LR, int RPL, bool GRID>
__device__ __forceinline__ void ldl_solve(Cdf (&x)[RPL], const float4* L, const float* lmax, const float2* rd, int D,
                                          int li, int gbase) {
  subst<LR, RPL, false, GRID>(x, L, lmax, D, li, gbase);
#pragma unroll
  for (int q = 0; q < RPL; ++q) {
    const int i = li + LR * q;
    const float2 r = rd[i < D ? i : D - 1];
    x[q] = i < D ? scale(x[q], ff::F2{r.x, r.y}) : Cdf{0.f, 0.f, 0.f, 0.f};
  }
  subst<LR, RPL, true, GRID>(x, L, lmax, D, li, gbase);
#pragma unroll
  for (int q = 0; q < RPL; ++q) norm(x[q]);
}

// The same in FP32 with the FP32 factor (kMixedIr).
template <int LR, int RPL, bool BACK>
__device__ __forceinline__ void subst_f32(float2 (&x)[RPL], const float2* L, int D, int li, int gbase) {
#pragma unroll
  for (int bb = 0; bb < RPL; ++bb) {
    const int qb = BACK ? RPL - 1 - bb : bb;
    if (LR * qb >= D) continue;
    const int jn = min(LR, D - LR * qb);
    const int b0 = li * D - li * (li - 1) / 2 - li, b1 = LR * D - LR * li - LR / 2;
#pragma unroll 2
    for (int jj = 0; jj < jn; ++jj) {
      const int jo = BACK ? jn - 1 - jj : jj;
      const int j = LR * qb + jo;
      const float yr = __shfl_sync(0xffffffffu, x[qb].x, gbase + jo);
      const float yi = __shfl_sync(0xffffffffu, x[qb].y, gbase + jo);
      const float2* cj = L + cstart(j, D) - j + li;
#pragma unroll
      for (int q = 0; q < RPL; ++q) {
        if (BACK ? (q > qb) : (q < qb)) continue;
        if (LR * q >= D) continue;
        float2 l = make_float2(0.f, 0.f);
        if (q != qb || (BACK ? li < jo : (li > jo && li + LR * q < D))) l = BACK ? L[b0 + j + b1 * q - q * q * (LR * LR / 2)] : cj[LR * q];
        if (BACK) l.y = -l.y;
        x[q].x = fmaf(-l.x, yr, x[q].x);
        x[q].y = fmaf(-l.x, yi, x[q].y);
        x[q].x = fmaf(l.y, yi, x[q].x);
        x[q].y = fmaf(-l.y, yr, x[q].y);
      }
    }
  }
}

template <int LR, int RPL>
__device__ __forceinline__ void ldl_solve_f32(Cdf (&x)[RPL], const float2* L, const float2* rd, int D, int li,
                                              int gbase) {
  float2 xf[RPL];
#pragma unroll
  for (int q = 0; q < RPL; ++q) xf[q] = make_float2(__fadd_rn(x[q].rs, x[q].re), __fadd_rn(x[q].is, x[q].ie));
  subst_f32<LR, RPL, false>(xf, L, D, li, gbase);
#pragma unroll
  for (int q = 0; q < RPL; ++q) {
    const int i = li + LR * q;
    const float r = i < D ? rd[i].x : 0.f;
    xf[q] = i < D ? make_float2(xf[q].x * r, xf[q].y * r) : make_float2(0.f, 0.f);
  }
  subst_f32<LR, RPL, true>(xf, L, D, li, gbase);
#pragma unroll
  for (int q = 0; q < RPL; ++q) x[q] = Cdf{xf[q].x, 0.f, xf[q].y, 0.f};
}

// Shared memory of one team: the solutions U [nu][D], Rl in As (a chunk of
// columns [KC][D + 1], or where the team is part of a warp the whole matrix:
// small systems convert it once -- as columns [D][D + 1] (SQUARE), or for more
// than 12 rows, where that would cost a third of the resident warps (D = 15:
// 197 -> 160 us per 3840 systems), as the lower triangle packed like the factor), the two pivot columns before division
// [2][D] (in the chunk's place: the factorisation is over before the first
// residual), the factor
// [Dp] (column-major packed), the pivot reciprocals [D], the pivot flag and
// three words of bits for passes with a vector whose combination cancels.
template <int LR, int RPL>
__host__ __device__ constexpr bool square() { return LR * RPL <= 12; }

template <int TEAM, int MODE, bool SQUARE>
struct Shared {
  static constexpr bool FULL = TEAM <= 32;
  using LT = typename std::conditional<f32f(MODE), float2, float4>::type;   // factor entries
  int u, as, col, l, rd, ok, bytes;                // byte offsets, all multiples of 16
  __host__ __device__ Shared(int D, int nu) {
    const int Dp = D * (D + 1) / 2;
    u = 0;
    as = u + nu * D * 16;
    col = FULL ? as + (SQUARE ? D * (D + 1) : Dp) * 16 : as;
    l = FULL ? col + 2 * D * 16 : as + KC * (D + 1) * 16;
    rd = l + (Dp * (int)sizeof(LT) + 15) / 16 * 16;
    ok = rd + (D * 8 + 15) / 16 * 16;
    bytes = ok + 16;
  }
};

// A team's system, as its phases need it.
struct System {
  int off;              // the team's shared memory, in bytes
  int nu;               // rows of U
  int sbase;            // split()'s exponent offset
  double delta;         // the load
  const double2* A;     // the covariance
  long long a0, aext;   // its first entry's index and the extent of the array
};

template <int TEAM>
__device__ __forceinline__ void team_sync() {
  if constexpr (TEAM > 32) __syncthreads();
  else __syncwarp();
}
template <int TEAM>
__device__ __forceinline__ int team_thread() {
  return TEAM > 32 ? threadIdx.x : threadIdx.x % TEAM;
}

// Rl[i][l], i >= l
__device__ __forceinline__ float4 entry(const System& y, int D, int i, int l) {
  double2 a = in_bounds(y.a0 + (long long)i * D + l, y.aext, kSiteSolveIn) ? __ldg(y.A + (size_t)i * D + l)
                                                                           : make_double2(0.0, 0.0);
  if (i == l) {
    a.x += y.delta;
    a.y = 0.0;
  }
  return split(a, y.sbase);
}

template <bool F32F>
__device__ __forceinline__ ff::F2 pivot(ff::F2 d, int* okf) {
  if (!(d.hi > 0.f) || !isfinite(d.hi)) {
    *okf = 0;
    return {1.f, 0.f};   // keep going; this system's weights become zero
  }
  if constexpr (F32F) return {1.0f / d.hi, 0.f};
  return recip(d);
}

// Copy Rl's lower triangle into shared memory and factor it: Rl = Lu Dg Lu^H,
// right-looking, two columns per round.  Phase 1: the thread of row i scales
// column j, brings its entry of column j+1 up to date and scales that; each
// thread forms the two pivots' reciprocals itself.  Phase 2: the rank-2 update
// of the trailing triangle, its columns spread over groups of RW threads, a
// group's threads over a column's rows.  On grids every other phase 2 updates
// the next two columns only and the one after it takes four columns at once,
// half the passes over the triangle in shared memory (128 rows: 410k cycles
// without grids, 325k with, 287k by four columns).
template <int TEAM, int MODE, bool SQUARE>
__device__ __forceinline__ void factor(const System y, int D) {
  extern __shared__ float4 smdf[];
  using SH = Shared<TEAM, MODE, SQUARE>;
  const SH sh(D, y.nu);
  using LT = typename SH::LT;
  char* base = reinterpret_cast<char*>(smdf) + y.off;
  LT* L = reinterpret_cast<LT*>(base + sh.l);
  float2* rd = reinterpret_cast<float2*>(base + sh.rd);
  int* okf = reinterpret_cast<int*>(base + sh.ok);
  const int tt = team_thread<TEAM>();
  // On grids: h_i = sqrt(Rl_ii); |Rl_il| and every partial sum of the entry's
  // updates are at most h_i h_l where Rl is positive definite (h_i in rd[i]
  // until the pivot's reciprocal comes)
  constexpr bool GRID = grids<TEAM, MODE>();
  if constexpr (GRID) {
    for (int i = tt; i < D; i += TEAM) rd[i].x = 1.0001f * sqrtf(fmaxf(entry(y, D, i, i).x, 0.f));
    team_sync<TEAM>();
  }
  auto take = [](Cdf& x, float hh) {               // an entry's finished sum
    if constexpr (GRID) unbias(x, sigma(hh));
    else norm(x);
  };
  auto less = [](Cdf& x, float4 l, float4 v) {
    if constexpr (GRID) gcms(x, l, v);
    else cms(x, l, v);
  };
  auto put = [&](int i, int l, float4 v) {
    if constexpr (f32f(MODE)) {
      L[cstart(l, D) + i - l] = make_float2(__fadd_rn(v.x, v.z), __fadd_rn(v.y, v.w));
    } else if constexpr (GRID) {
      Cdf b = unpack(v);
      bias(b, sigma(rd[i].x * rd[l].x));
      L[cstart(l, D) + i - l] = pack(b);
    } else {
      L[cstart(l, D) + i - l] = v;
    }
    if constexpr (SH::FULL) {
      float4* As = reinterpret_cast<float4*>(base + sh.as);
      if constexpr (!SQUARE) {
        As[cstart(l, D) + i - l] = v;
      } else {
        As[l * (D + 1) + i] = v;                   // column l, row i
        As[i * (D + 1) + l] = conj4(v);
      }
    }
  };
  if constexpr (TEAM > 32) {                       // rows coalesced
    for (int i = tt >> 5; i < D; i += TEAM / 32)
      for (int l = tt & 31; l <= i; l += 32) put(i, l, entry(y, D, i, l));
  } else {
    int i = 0, l = tt;
    while (l > i) l -= ++i;
    for (int q = tt; q < D * (D + 1) / 2; q += TEAM) {
      put(i, l, entry(y, D, i, l));
      l += TEAM;
      while (l > i) l -= ++i;
    }
  }
  if (tt < 4) okf[tt] = tt == 0;
  team_sync<TEAM>();

  for (int j = 0; j < D; j += 2) {
    const int j1 = j + 1;
    const bool pair = j1 < D, second = GRID && (j & 2) != 0;
    LT* colb = reinterpret_cast<LT*>(base + sh.col) + (second ? 2 * D : 0);
    LT* colb2 = colb + D;
    const int cj = cstart(j, D), c1 = pair ? cstart(j1, D) : cj;
    if constexpr (f32f(MODE)) {
      const float rj = pivot<f32f(MODE)>({L[cj].x, 0.f}, okf).hi;
      float2 a1j = make_float2(0.f, 0.f);
      float r1 = 1.f;
      if (pair) {
        a1j = L[cj + 1];
        float d1 = L[c1].x;
        d1 = fmaf(-a1j.x * rj, a1j.x, d1);
        d1 = fmaf(-a1j.y * rj, a1j.y, d1);
        r1 = pivot<f32f(MODE)>({d1, 0.f}, okf).hi;
      }
      float2 own = make_float2(0.f, 0.f);
      bool own1 = false;
      for (int i = j1 + tt; i < D; i += TEAM) {
        const float2 v = L[cj + i - j];
        colb[i] = v;
        const float2 lij = make_float2(v.x * rj, v.y * rj);
        if (i == j1) {
          own = lij;
          own1 = true;
        } else {
          L[cj + i - j] = lij;
          float2 w = L[c1 + i - j1];
          w.x = fmaf(-lij.x, a1j.x, w.x);
          w.y = fmaf(-lij.y, a1j.x, w.y);
          w.x = fmaf(-lij.y, a1j.y, w.x);
          w.y = fmaf(lij.x, a1j.y, w.y);
          colb2[i] = w;
          L[c1 + i - j1] = make_float2(w.x * r1, w.y * r1);
        }
      }
      if (tt == 0) {
        rd[j] = make_float2(rj, 0.f);
        if (pair) rd[j1] = make_float2(r1, 0.f);
      }
      team_sync<TEAM>();
      if (own1) L[cj + 1] = own;
    } else {
      const float hj = GRID ? rd[j].x : 0.f, h1 = GRID && pair ? rd[j1].x : 0.f;
      Cdf dj = unpack(L[cj]);
      take(dj, hj * hj);
      const ff::F2 rj = pivot<f32f(MODE)>({dj.rs, dj.re}, okf);
      Cdf a1j{0.f, 0.f, 0.f, 0.f};
      ff::F2 r1{1.f, 0.f};
      if (pair) {
        a1j = unpack(L[cj + 1]);
        take(a1j, hj * h1);
        Cdf d1 = unpack(L[c1]);
        less(d1, pack(scale(a1j, rj)), conj4(pack(a1j)));
        take(d1, h1 * h1);
        r1 = pivot<f32f(MODE)>({d1.rs, d1.re}, okf);
      }
      const float4 a1c = conj4(pack(a1j));
      float4 own = make_float4(0.f, 0.f, 0.f, 0.f);
      bool own1 = false;
      for (int i = j1 + tt; i < D; i += TEAM) {
        const float hi = GRID ? rd[i].x : 0.f;
        Cdf v = unpack(L[cj + i - j]);
        take(v, hi * hj);
        colb[i] = conj4(pack(v));                // stored conjugated
        const float4 lij = pack(scale(v, rj));
        if (i == j1) {
          own = lij;
          own1 = true;
        } else {
          L[cj + i - j] = lij;
          Cdf w = unpack(L[c1 + i - j1]);
          less(w, lij, a1c);
          take(w, hi * h1);
          colb2[i] = conj4(pack(w));
          L[c1 + i - j1] = pack(scale(w, r1));
        }
      }
      team_sync<TEAM>();
      if (tt == 0) {
        rd[j] = make_float2(rj.hi, rj.lo);
        if (pair) rd[j1] = make_float2(r1.hi, r1.lo);
      }
      if (own1) L[cj + 1] = own;
    }
    if constexpr (GRID) {
      if (!second) {                               // the next pair of columns only
        const int l = j + 2 + tt / (TEAM / 2), i = l + tt % (TEAM / 2);
        if (i < D) {
          LT* e = L + cstart(l, D) + i - l;
          Cdf acc = unpack(*e);
          gcms(acc, L[cj + i - j], colb[l]);
          gcms(acc, L[c1 + i - j1], colb2[l]);
          norm(acc);
          *e = pack(acc);
        }
      } else {                                     // the rest, by both pairs
        constexpr int RW = TEAM == 512 ? 32 : 16;
        const LT* la = L + cstart(j - 2, D) + 2 - j;
        const LT* lb = L + cstart(j - 1, D) + 1 - j;
        for (int l = j + 2 + tt / RW; l < D; l += TEAM / RW) {
          const LT ya = colb[l - 2 * D], yb = colb[l - D], yc = colb[l], yd = colb2[l];
          LT* cl = L + cstart(l, D) - l;
          for (int i = l + tt % RW; i < D; i += RW) {
            Cdf acc = unpack(cl[i]);
            gcms(acc, la[i], ya);
            gcms(acc, lb[i], yb);
            gcms(acc, L[cj + i - j], yc);
            gcms(acc, L[c1 + i - j1], yd);
            norm(acc);
            cl[i] = pack(acc);
          }
        }
      }
      team_sync<TEAM>();
      continue;
    }
    constexpr int RW = TEAM == 512 ? 32 : (TEAM >= 128 ? 16 : (TEAM >= 32 ? 8 : 4));
    for (int l = j + 2 + tt / RW; l < D; l += TEAM / RW) {
      const LT alj = colb[l], blj = colb2[l];
      LT* cl = L + cstart(l, D) - l;
      for (int i = l + tt % RW; i < D; i += RW) {
        const LT lij = L[cj + i - j], mij = L[c1 + i - j1];
        if constexpr (f32f(MODE)) {
          float2 acc = cl[i];
          acc.x = fmaf(-lij.x, alj.x, acc.x);
          acc.y = fmaf(-lij.y, alj.x, acc.y);
          acc.x = fmaf(-lij.y, alj.y, acc.x);
          acc.y = fmaf(lij.x, alj.y, acc.y);
          acc.x = fmaf(-mij.x, blj.x, acc.x);
          acc.y = fmaf(-mij.y, blj.x, acc.y);
          acc.x = fmaf(-mij.y, blj.y, acc.x);
          acc.y = fmaf(mij.x, blj.y, acc.y);
          cl[i] = acc;
        } else {
          Cdf acc = unpack(cl[i]);
          less(acc, lij, alj);
          less(acc, mij, blj);
          norm(acc);
          cl[i] = pack(acc);
        }
      }
    }
    team_sync<TEAM>();
  }
}

// What a group of LR lanes solves in a pass: steering vector rhs itself
// (direct) or basis vector rhs, into row `row` of U; a group without one of its
// own (!live) computes a copy that is never stored.
struct Rhs {
  int rhs, row;
  bool live, direct;
  bool work;   // a CTA team's warps without right-hand sides only help convert
};

// Solve and refine a pass of right-hand sides, one per group of LR lanes.
//
// kAnyMatrix: what the first refinement step corrects is the solution's error up
// to then, kappa(Rl) times the arithmetic's for this right-hand side.  Above
// max_correction of the solution, 2^-43 of the bound on a covariance's kappa, and
// above 2^-36 / delta (entries of the right-hand side are about 1: a solution much
// smaller than 1 / delta, of a vector along strong interference, has an error
// of up to 2^-40 / delta), the system gets the second bit of the pivot flag.
// Without refinement steps the correction is formed all the same, but not
// applied.
// Refinement steps: a vector whose combination cancels takes one at least, its
// small solution loses up to kappa(Rl) 2^-46 to the unrefined solve.
template <int MODE>
__device__ __forceinline__ int steps(const Rhs& z, const SolveDfParams& prm) {
  return !f32f(MODE) && z.direct && prm.sep != 0 ? max(prm.refine_steps, 1) : prm.refine_steps;
}

template <int LR, int RPL, int TEAM, int MODE>
__device__ __forceinline__ void solve_rhs(const SolveDfParams& prm, const System y, const Rhs z) {
  constexpr int EPT = (KC * LR * RPL + TEAM - 1) / TEAM;   // chunk entries per thread
  using SH = Shared<TEAM, MODE, square<LR, RPL>()>;
  extern __shared__ float4 smdf[];
  const int D = prm.D, C = prm.C;
  const SH sh(D, y.nu);
  char* base = reinterpret_cast<char*>(smdf) + y.off;
  float4* U = reinterpret_cast<float4*>(base + sh.u);
  float4* As = reinterpret_cast<float4*>(base + sh.as);
  const typename SH::LT* L = reinterpret_cast<const typename SH::LT*>(base + sh.l);
  const float2* rd = reinterpret_cast<const float2*>(base + sh.rd);
  constexpr bool GRID = grids<TEAM, MODE>();
  const int tt = team_thread<TEAM>(), li = tt % LR;
  const int gbase = (threadIdx.x & 31) - li;       // first lane of this thread's group
  const bool work = z.work, live = z.live;
  const int rhs = z.rhs;
  float4* Ur = U + (size_t)z.row * D;              // its solution
  auto b_at = [&](int i) -> Cdf {              // right-hand side entry
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);   // tables: (re hi, re lo, im hi, im lo)
    if (i < D) {
      if (z.direct) {
        v = __ldg(prm.steer_ff + (size_t)rhs * D + i);
      } else {
        const int t = i / C;
        if (i - t * C == rhs) v = __ldg(prm.g_ff + t);
      }
    }
    return Cdf{v.x, v.y, v.z, v.w};
  };
  Cdf x[RPL];
#pragma unroll
  for (int q = 0; q < RPL; ++q) x[q] = b_at(li + LR * q);
  for (int it = 0;; ++it) {
    // the largest entry of each row block of a column and column block of a
    // row, in the chunk's place
    float* lmax = reinterpret_cast<float*>(As);
    if constexpr (GRID) {
      __syncthreads();
      for (int f = tt; f < 2 * RPL * D; f += TEAM) {
        const int b = f / D, i = f - b * D, j0 = LR * (b < RPL ? b : b - RPL);
        const int j1 = min(j0 + LR, D);
        float m = 0.f;
        if (b < RPL ? i >= j1 : i < j0)
          for (int j = j0; j < j1; ++j) {
            const float4 l = L[b < RPL ? cstart(j, D) - j + i : cstart(i, D) - i + j];
            m = fmaxf(m, fmaxf(fabsf(l.x), fabsf(l.y)));
          }
        lmax[f] = m;
      }
      __syncthreads();
    }
    if (work) {
      if constexpr (f32f(MODE)) ldl_solve_f32<LR, RPL>(x, L, rd, D, li, gbase);
      else ldl_solve<LR, RPL, GRID>(x, L, lmax, rd, D, li, gbase);
      if (MODE == kAnyMatrix && it == 1) {
        float c = 0.f, u = 0.f;
#pragma unroll
        for (int q = 0; q < RPL; ++q) {
          const int i = li + LR * q;
          if (i < D) {
            const float4 v = Ur[i];
            const float a = fabsf(x[q].rs) + fabsf(x[q].is);
            c = a < INFINITY ? fmaxf(c, a) : INFINITY;   // (a NaN too)
            u = fmaxf(u, fabsf(v.x) + fabsf(v.y));
          }
        }
        c = lanes_max<LR>(c);
        u = lanes_max<LR>(u);
        const float some = __fdividef(1.5e-11f, split(y.delta, y.sbase).hi);
        if (live && li == 0 && !(c <= fmaf(prm.max_correction, u, some))) atomicOr(reinterpret_cast<int*>(base + sh.ok), 2);
      }
      if (MODE != kAnyMatrix || it <= steps<MODE>(z, prm))
#pragma unroll
        for (int q = 0; q < RPL; ++q) {
          const int i = li + LR * q;
          if (i < D) {
            if (it > 0) x[q] = add(unpack(Ur[i]), x[q]);   // u += c
            if (live) Ur[i] = pack(x[q]);
          }
        }
    }
    if (it == (MODE == kAnyMatrix ? max(steps<MODE>(z, prm), 1) : steps<MODE>(z, prm))) break;
    // x = b - Rl u
#pragma unroll
    for (int q = 0; q < RPL; ++q) x[q] = b_at(li + LR * q);
    // columns l0 .. l0 + n - 1 at a, pitch D + 1; rows past D: never read
    auto columns = [&](const float4* a, int l0, int n) {
      for (int ll = 0; ll < n; ++ll) {
        const float4 u = Ur[l0 + ll];
        const float4* al = a + ll * (D + 1) + li;
#pragma unroll
        for (int q = 0; q < RPL; ++q)
          if (LR * q < D) cms(x[q], al[LR * q], u);
      }
#pragma unroll
      for (int q = 0; q < RPL; ++q) norm(x[q]);
    };
    if constexpr (SH::FULL && square<LR, RPL>()) {
      __syncwarp();                                // the U rows are written
      for (int l0 = 0; l0 < D; l0 += KC) columns(As + l0 * (D + 1), l0, min(KC, D - l0));
    } else if constexpr (SH::FULL) {
      __syncwarp();
      // column l: rows i >= l lie at cstart(l) - l + i, above the diagonal the
      // conjugates of row l at cstart(i) - i + l
      for (int l = 0; l < D; ++l) {
        const float4 u = Ur[l];
        const int below = cstart(l, D) - l;
#pragma unroll
        for (int q = 0; q < RPL; ++q) {
          const int i = min(li + LR * q, D - 1);
          const bool low = i >= l;
          const float4 a = As[low ? below + i : cstart(i, D) - i + l];
          cms(x[q], low ? a : conj4(a), u);
        }
        if (l % KC == KC - 1 || l == D - 1)
#pragma unroll
          for (int q = 0; q < RPL; ++q) norm(x[q]);
      }
    } else {
      // entry f of the chunk at column l0: column l0 + f % KC, row f / KC; the
      // next chunk's entries wait in registers
      auto chunk_entry = [&](int l0, int f) -> float4 {
        const int l = l0 + f % KC, i = f / KC;
        if (l >= D || i >= D) return make_float4(0.f, 0.f, 0.f, 0.f);
        return i >= l ? entry(y, D, i, l) : conj4(entry(y, D, l, i));
      };
      float4 pre[EPT];
#pragma unroll
      for (int k = 0; k < EPT; ++k) pre[k] = chunk_entry(0, tt + k * TEAM);
      for (int l0 = 0; l0 < D; l0 += KC) {
        __syncthreads();                           // the last chunk (and the U rows) are done with
#pragma unroll
        for (int k = 0; k < EPT; ++k) {
          const int f = tt + k * TEAM;
          if (f / KC < D) As[(f % KC) * (D + 1) + f / KC] = pre[k];
        }
        __syncthreads();
        if (l0 + KC < D)
#pragma unroll
          for (int k = 0; k < EPT; ++k) pre[k] = chunk_entry(l0 + KC, tt + k * TEAM);
        if (work) columns(As, l0, min(KC, D - l0));
      }
    }
  }
}

// The weights of a pass's steering vectors from their solutions in U.  (This
// and combine() are calls: inlined, their registers cost the substitutions
// theirs; 3% on a D = 128 system.)
template <int LR, int RPL, int TEAM>
__device__ __noinline__ void emit(const SolveDfParams& prm, int off, long long sys, bool store, bool ok, int e,
                                  int rhs, int row) {
  extern __shared__ float4 smdf[];
  const int D = prm.D, S = prm.S;
  const long long nsys = prm.nsys;
  float2* __restrict__ wts = prm.wts;
  const int tt = team_thread<TEAM>(), li = tt % LR;
  const float4* Ur = smdf + off / 16 + (size_t)row * D;
  float qs = 0.f, qe = 0.f;
#pragma unroll
  for (int q = 0; q < RPL; ++q) {
    const int i = li + LR * q;
    if (i < D) {
      const float4 v = __ldg(prm.steer_ff + (size_t)rhs * D + i), u = Ur[i];
      mac(qs, qe, v.x, v.y, u.x, u.z);
      mac(qs, qe, v.z, v.w, u.y, u.w);
    }
  }
  const ff::F2 qd = lanes_sum2<LR>(qs, qe);
  const bool good = ok && usable(qd);
  const Gain sf = gain(qd, -e / 2);
  if (store) {
    const long long w0 = (sys * S + rhs) * D;
#pragma unroll
    for (int q = 0; q < RPL; ++q) {
      const int i = li + LR * q;
      if (i < D && in_bounds(w0 + i, nsys * S * D, kSiteSolveOut)) {
        const float4 u = Ur[i];
        wts[w0 + i] = weight({u.x, u.z}, {u.y, u.w}, sf, good);
      }
    }
  }
}

// Separable steering: u_s = sum_c a_s[c] U_c from the team's basis solutions U
// (at byte `off` of shared memory) and the normalised weights.
//
// Where v_s lies along strong interference, u_s is up to kappa(Rl) times smaller
// than the terms of that sum and keeps their errors.  Unrefined basis solutions
// belong to one slightly other matrix, and so does their combination; but a
// refinement step rounds every residual by itself, 2^-48 of |Rl| |U_c|, which
// the smallest eigenvalue, the load, turns into about 2^-47 / lf of U_c: measured
// 6e-15 / lf of sum max |U_c| (spatial factors of magnitude 1) for D = 12 to 128, loads 1e-3 to 2.3e-5 and
// one or two steps.  (Rank one along v_s, 60 dB and more: errors of 2.5e-7 at D =
// 12 to 1.8e-5 at D = 128 for load 1e-3, up to 5e-4 for the weakest loads; a solve
// of v_s itself is below the complex64 rounding.)  A vector whose ratio is 2^21
// lf or more (SolveDfParams::cancel), i.e. half a complex64 rounding, is solved
// by itself, with the others of its pass.  A clutter ridge seldom gets there
// (whole CPIs, 40 dB, load 1e-3: median ratio 3 to 30; 77 of 16384 systems of
// 128 rows have such a vector, none of up to 64 rows).  (The refinement option
// keeps the combination.)
// Most vectors need no look at the sums: |U_c| <= |g| / delta and Re v^H u <= max
// |u| sum |v|, so that a q of cancel_q / delta or more rules the ratio out (or, once
// the sum over the basis is there, of steer_sum times that; a caller's matrix need
// not keep the first bound).
// The sum over the basis of max |U_c|.  (A call: inlined it costs the combination
// its registers, for a look that few vectors need.)
template <int LR>
__device__ __noinline__ float sum_of_largest(const float4* U, int C, int D) {
  const int li = (threadIdx.x & 31) % LR;
  float sum = 0.f;
  for (int c = 0; c < C; ++c) {
    float m = 0.f;
    for (int i = li; i < D; i += LR)
      m = fmaxf(m, fmaxf(fabsf(U[(size_t)c * D + i].x), fabsf(U[(size_t)c * D + i].y)));
    sum += lanes_max<LR>(m);
  }
  return sum;
}

// Which passes solve steering vectors by themselves, PASS or (the rows of U) C of
// them at a time: all, or of 512 threads, whose passes are long, those with a
// marked vector -- a bit each beside the pivot flag, the last one for all from
// the 96th on (D = 120, 191 of 4096 systems marked: 10% of the solve's time, with
// the bits 5%; for smaller systems the bits cost 1 to 2% and save little).
template <int TEAM>
__host__ __device__ constexpr bool pass_bits() { return TEAM == 512; }
template <int LR, int TEAM>
__device__ __forceinline__ int direct_step(int C) { return min(TEAM / LR, C); }
template <int LR, int TEAM>
__device__ __forceinline__ void mark(int* bits, int s, int C) {
  const int b = pass_bits<TEAM>() ? min(s / direct_step<LR, TEAM>(C), 95) : 0;
  atomicOr(bits + b / 32, 1 << (b & 31));
}

template <int LR, int RPL, int TEAM, int MODE>
__device__ __noinline__ void combine(const SolveDfParams& prm, int off, long long sys, bool valid, bool ok, int e,
                                     float delta) {
  constexpr int NG = TEAM / LR;
  extern __shared__ float4 smdf[];
  const float4* U = smdf + off / 16;
  const int D = prm.D, S = prm.S, C = prm.C;
  const long long nsys = prm.nsys;
  float2* __restrict__ wts = prm.wts;
  const int tt = team_thread<TEAM>(), li = tt % LR, g = tt / LR;
  const Shared<TEAM, MODE, square<LR, RPL>()> sh(D, C);
  char* base = reinterpret_cast<char*>(smdf) + off;
  int* cancels = reinterpret_cast<int*>(base + sh.ok) + 1;
  float least_q = MODE == kAnyMatrix ? INFINITY : __fdividef(prm.cancel_q, delta), least = -1.f;
  // u_s = sum_c a_s[c] U_c: a group takes a steering vector s1 -- with
  // conjugate-symmetric factors (a_{S-1-s} = conj(a_s)) the pair s1,
  // S-1-s1 from the four real sums P = sum ar Ur, Q = sum ai Ui,
  // R = sum ar Ui, T = sum ai Ur: u_s1 = (P - Q) + j (R + T),
  // u_s2 = (P + Q) + j (R - T)
  const bool sym = prm.sym != 0;
  const int n1 = sym ? (S + 1) / 2 : S;
  for (int p0 = 0; p0 < n1; p0 += NG) {
    const int s1 = min(p0 + g, n1 - 1), s2 = S - 1 - s1;
    const bool st1 = valid && p0 + g < n1, st2 = st1 && sym && s2 != s1;
    const float4* as = prm.sep_a_ff + (size_t)s1 * C;
    const float4* v1 = prm.steer_ff + (size_t)s1 * D;
    const float4* v2 = prm.steer_ff + (size_t)s2 * D;
    ff::F2 w1r[RPL], w1i[RPL], w2r[RPL], w2i[RPL];
    float q1s = 0.f, q1e = 0.f, q2s = 0.f, q2e = 0.f;
    constexpr int QB = RPL % 4 == 0 ? 4 : (RPL % 3 == 0 ? 3 : 2);   // rows per pass over the basis
#pragma unroll
    for (int q0 = 0; q0 < RPL; q0 += QB) {
      if (LR * q0 >= D) continue;
      Cdf PR[QB], TQ[QB];                        // (P, R) and (T, Q) of each row
#pragma unroll
      for (int q = 0; q < QB; ++q) PR[q] = TQ[q] = Cdf{0.f, 0.f, 0.f, 0.f};
      for (int c = 0; c < C; ++c) {
        const float4 a = __ldg(as + c);
#pragma unroll
        for (int q = 0; q < QB; ++q) {
          const int i = li + LR * (q0 + q);
          const float4 u = U[(size_t)c * D + (i < D ? i : D - 1)];
          mac(PR[q].rs, PR[q].re, a.x, a.y, u.x, u.z);
          mac(TQ[q].is, TQ[q].ie, a.z, a.w, u.y, u.w);
          mac(PR[q].is, PR[q].ie, a.x, a.y, u.y, u.w);
          mac(TQ[q].rs, TQ[q].re, a.z, a.w, u.x, u.z);
        }
      }
#pragma unroll
      for (int q = q0; q < q0 + QB; ++q) {
        const int i = li + LR * q;
        norm(PR[q - q0]);
        norm(TQ[q - q0]);
        const ff::F2 P{PR[q - q0].rs, PR[q - q0].re}, R{PR[q - q0].is, PR[q - q0].ie};
        const ff::F2 T{TQ[q - q0].rs, TQ[q - q0].re}, Q{TQ[q - q0].is, TQ[q - q0].ie};
        const ff::F2 ur1 = ff::sub2(P, Q), ui1 = ff::add2(R, T);
        const ff::F2 ur2 = ff::add2(P, Q), ui2 = ff::sub2(R, T);
        if (i < D) {
          const float4 b1 = __ldg(v1 + i), b2 = __ldg(v2 + i);
          mac(q1s, q1e, b1.x, b1.y, ur1.hi, ur1.lo);
          mac(q1s, q1e, b1.z, b1.w, ui1.hi, ui1.lo);
          mac(q2s, q2e, b2.x, b2.y, ur2.hi, ur2.lo);
          mac(q2s, q2e, b2.z, b2.w, ui2.hi, ui2.lo);
        }
        w1r[q] = ur1;
        w1i[q] = ui1;
        w2r[q] = ur2;
        w2i[q] = ui2;
      }
    }
    const ff::F2 d1 = lanes_sum2<LR>(q1s, q1e), d2 = lanes_sum2<LR>(q2s, q2e);
    if (!f32f(MODE) && __any_sync(0xffffffffu, !(d1.hi >= least_q) || (sym && !(d2.hi >= least_q)))) {
      float m1 = 0.f, m2 = 0.f;                    // max |u_s1|, max |u_s2|
#pragma unroll
      for (int q = 0; q < RPL; ++q)
        if (li + LR * q < D) {
          m1 = fmaxf(m1, fmaxf(fabsf(w1r[q].hi), fabsf(w1i[q].hi)));
          m2 = fmaxf(m2, fmaxf(fabsf(w2r[q].hi), fabsf(w2i[q].hi)));
        }
      m1 = lanes_max<LR>(m1);
      m2 = lanes_max<LR>(m2);
      if (least < 0.f) {                           // the system's sum of max |U_c|, once
        least = sum_of_largest<LR>(U, C, D);
        least *= prm.cancel;
        least_q = fminf(least_q, least * prm.steer_sum);
      }
      if (ok && li == 0 && p0 + g < n1) {
        if (!(m1 >= least)) mark<LR, TEAM>(cancels, s1, C);
        if (sym && !(m2 >= least)) mark<LR, TEAM>(cancels, s2, C);
      }
    }
    const bool good1 = ok && usable(d1), good2 = ok && usable(d2);
    const Gain f1 = gain(d1, -e / 2), f2 = gain(d2, -e / 2);
#pragma unroll
    for (int q = 0; q < RPL; ++q) {
      const int i = li + LR * q;
      if (i < D) {
        const long long o1 = (sys * S + s1) * D + i, o2 = (sys * S + s2) * D + i, ext = nsys * S * D;
        if (st1 && in_bounds(o1, ext, kSiteSolveOut))
          wts[o1] = weight(w1r[q], w1i[q], f1, good1);
        if (st2 && in_bounds(o2, ext, kSiteSolveOut))
          wts[o2] = weight(w2r[q], w2i[q], f2, good2);
      }
    }
  }
}

template <int LR, int RPL, int TEAM, int MODE>
__device__ __forceinline__ void solve_df_body(const SolveDfParams& prm, long long bx, long long gx) {
  constexpr int PASS = TEAM / LR;                  // right-hand sides per pass, one per group
  const long long nsys = prm.nsys;
  const int D = prm.D;
  const bool sep = prm.sep != 0;
  extern __shared__ float4 smdf[];
  const int team = TEAM > 32 ? 0 : threadIdx.x / TEAM;   // team in CTA
  const int teams = TEAM > 32 ? 1 : blockDim.x / TEAM;
  const int tt = team_thread<TEAM>();
  System y;
  y.nu = sep ? prm.C : PASS;
  const Shared<TEAM, MODE, square<LR, RPL>()> sh(D, y.nu);
  y.off = team * sh.bytes;
  y.aext = nsys * (long long)D * D;
  const int* okf = reinterpret_cast<const int*>(reinterpret_cast<char*>(smdf) + y.off + sh.ok);

  for (long long base_sys = bx * teams; base_sys < nsys; base_sys += gx * teams) {
    const long long sys = base_sys + team;
    const bool valid = sys < nsys;                 // the last CTA's spare teams repeat the last system
    y.a0 = (valid ? sys : nsys - 1) * (long long)D * D;
    y.A = prm.cov + y.a0;
    // trace: lanes over the diagonal (every warp of a CTA team its own sum)
    constexpr int TW = TEAM > 32 ? 32 : TEAM;
    double tr = 0.0;
    for (int j = threadIdx.x % TW; j < D; j += TW)
      if (in_bounds(y.a0 + (long long)j * D + j, y.aext, kSiteSolveIn)) tr += __ldg(&y.A[(size_t)j * D + j].x);
    tr = lanes_sum<TW>(tr);
    y.delta = prm.load_factor * tr * (1.0 / D);
    // scale 2^-e, e even, trace of Rl 2^-e in [1, 4)
    const int et = (int)(((uint32_t)__double2hiint(fma(prm.load_factor, tr, tr)) >> 20) & 0x7FF);
    const int e = et == 0 || et == 0x7FF ? 0 : (et - 1023) & ~1;
    y.sbase = 896 + e;
    factor<TEAM, MODE, square<LR, RPL>()>(y, D);
    const bool ok = *okf != 0;
    // the basis and its combinations, and the passes with a vector whose
    // combination cancelled; or all the vectors
    bool direct = !sep;
    for (;;) {
      const int nrhs = direct ? prm.S : prm.C;
      const int step = direct && sep ? direct_step<LR, TEAM>(prm.C) : PASS;   // the rows of U
      for (int r0 = 0; r0 < nrhs; r0 += step) {
        if constexpr (pass_bits<TEAM>() && !f32f(MODE)) {
          const int b = min(r0 / step, 95);
          if (direct && sep && (okf[1 + b / 32] >> (b & 31) & 1) == 0) continue;
        }
        const int g = tt / LR, w0 = (tt >> 5) * (32 / LR);        // group in team, its warp's first
        Rhs z;
        z.direct = direct;
        z.live = g < step && r0 + g < nrhs;
        z.work = TEAM <= 32 || (w0 < step && r0 + w0 < nrhs);
        z.rhs = z.live ? r0 + g : nrhs - 1;
        z.row = direct ? min(g, step - 1) : z.rhs;
        solve_rhs<LR, RPL, TEAM, MODE>(prm, y, z);
        if (direct)
          emit<LR, RPL, TEAM>(prm, y.off, sys, valid && z.live && (pass_bits<TEAM>() || !sep || okf[1] != 0), ok, e, z.rhs,
                              z.row);
        team_sync<TEAM>();   // the next pass reuses U's rows, the combination reads them all
      }
      if (direct) break;
      combine<LR, RPL, TEAM, MODE>(prm, y.off, sys, valid, ok, e, split(y.delta, y.sbase).hi);
      team_sync<TEAM>();
      if (f32f(MODE)) break;
      if (!pass_bits<TEAM>() && (TEAM > 32 ? okf[1] == 0 : !__any_sync(0xffffffffu, okf[1] != 0))) break;   // alike in a warp
      direct = true;
    }
    if constexpr (MODE == kAnyMatrix) {            // (the pass and the combination ended with a barrier)
      if (valid && *okf != 1 && tt == 0) prm.wts[sys * prm.S * D] = make_float2(__uint_as_float(kUnsolved), 0.f);
    } else {
      if (valid && !ok && tt == 0) atomicAdd(&prm.status->n_failed, 1ULL);
    }
    team_sync<TEAM>();     // the next system reuses the team's shared memory
  }
}

constexpr int cta_threads(int team) { return team > 32 ? team : 128; }
// CTAs per SM that the registers must allow (shared memory allows about as many;
// five of 128 threads for teams within a warp: 96 registers instead of 80, 1 to 4%
// for D <= 16)
constexpr int min_ctas(int team, int mode) {
  return team == 512 ? 1 : (team == 256 ? 3 : (team == 128 ? 6 : (team == 64 ? 12 : (f32f(mode) ? 6 : 5))));
}

template <int LR, int RPL, int TEAM, int MODE>
__global__ void __launch_bounds__(cta_threads(TEAM), min_ctas(TEAM, MODE))
solve_df_kernel(SolveDfParams p) {
  solve_df_body<LR, RPL, TEAM, MODE>(p, blockIdx.x, gridDim.x);
}

// the same solves as a persistent launch over the CPIs of a batch
template <int LR, int RPL, int TEAM, int MODE>
__global__ void __launch_bounds__(cta_threads(TEAM), min_ctas(TEAM, MODE))
solve_df_batched(BatchCtl ctl) {
  batched_loop<SolveDfParams>(ctl, [&](const SolveDfParams& p, int bx, int, int gx) {
    solve_df_body<LR, RPL, TEAM, MODE>(p, bx, gx);
  });
}

template <int LR, int RPL, int TEAM, int MODE>
cudaError_t launch_df(SolveDfParams p, cudaStream_t s) {
  constexpr int PASS = TEAM / LR;
  constexpr size_t kMaxSmem = 227 * 1024;
  // the basis form keeps all C solutions in shared memory
  if (p.sep && Shared<TEAM, MODE, square<LR, RPL>()>(p.D, p.C).bytes > (int)kMaxSmem) p.sep = p.sym = 0;
  const size_t tb = Shared<TEAM, MODE, square<LR, RPL>()>(p.D, p.sep ? p.C : PASS).bytes;
  int threads = TEAM;
  if (TEAM <= 32) {
    // several teams per CTA; with few systems one warp per CTA, so that they
    // spread over the SMs
    threads = p.nsys * TEAM <= 152LL * 4 * 32 ? 32 : 128;
    while (threads > 32 && tb * (threads / TEAM) > 64 * 1024) threads >>= 1;
  }
  const int teams = TEAM > 32 ? 1 : threads / TEAM;
  const size_t smem = tb * teams;
  if (smem > kMaxSmem) return cudaErrorInvalidValue;
  static int set_bytes[64] = {0}, set_bytes_b[64] = {0};
  cudaError_t err = ensure_smem(solve_df_kernel<LR, RPL, TEAM, MODE>, smem, set_bytes);
  const long long units = (p.nsys + teams - 1) / teams;
  const long long blocks = units < (1LL << 30) ? units : (1LL << 30);
  p.gx = (int)blocks;
  if constexpr (MODE == kAnyMatrix) {              // one call's launch: no persistent form
    if (err != cudaSuccess) return err;
    solve_df_kernel<LR, RPL, TEAM, MODE><<<(unsigned)blocks, threads, smem, s>>>(p);
    return cudaGetLastError();
  } else {
    if (err == cudaSuccess) err = ensure_smem(solve_df_batched<LR, RPL, TEAM, MODE>, smem, set_bytes_b);
    if (err != cudaSuccess) return err;
    return launch_params(reinterpret_cast<const void*>(solve_df_kernel<LR, RPL, TEAM, MODE>),
                         reinterpret_cast<const void*>(solve_df_batched<LR, RPL, TEAM, MODE>),
                         dim3((unsigned)blocks), threads, smem, s, p, blocks);
  }
}

// The splits of the double-float solves: D <= 32, and above.
template <int MODE>
cudaError_t launch_small(const SolveDfParams& p, cudaStream_t s) {
  const int D = p.D;
  // Few systems with more right-hand sides than a warp's four groups take at
  // once, or many combinations: 128 threads per system, all of its right-hand
  // sides in one or two passes (us with a warp / with 128 threads, arbitrary
  // tables: D = 8 S = 64, 128 systems 100 / 21, 1024 102 / 60; D = 15 S = 16, 128
  // systems 51 / 22, 512 52 / 38, 1024 68 / 64; D = 16 S = 64, 1024 systems 233 / 185,
  // 2048 381 / 336; separable: C = 5 S = 16, D = 15, 512 systems 40 / 35, 1024 49 /
  // 64; C = 4 S = 64, D = 12, 512 systems 38 / 30, 1024 44 / 54)
  const int nrhs = p.sep ? p.C : p.S;
  const bool wide = (nrhs > 4 || p.S > 16) && p.cpi_sys <= (nrhs > 16 ? 1024 : 512);
  // D <= 12: half a warp per system, or a whole one where the systems are too
  // few to fill the SMs and the latency of one counts (C 4 S 16, D = 12, half /
  // whole: 256 systems 34.4 / 26.3 us, 1024 36.5 / 30.3, 4096 58.0 / 65.9).  D = 16:
  // a warp (1024: half 55.5, whole 36.4; 16384: 299, 277).  D = 32: 128 threads
  // (256: 64 threads 82.1, 128 58.0; 16384: 1875, 1817)
  if (D <= 8) return wide ? launch_df<4, 2, 128, MODE>(p, s) : launch_df<4, 2, 16, MODE>(p, s);
  if (D <= 12 && p.cpi_sys >= 2048) return launch_df<4, 3, 16, MODE>(p, s);
  if (D <= 16) return wide ? launch_df<8, 2, 128, MODE>(p, s) : launch_df<8, 2, 32, MODE>(p, s);
  if (D <= 24) return launch_df<8, 3, 64, MODE>(p, s);
  return launch_df<16, 2, 128, MODE>(p, s);
}

template <int MODE>
cudaError_t launch_large(const SolveDfParams& p, cudaStream_t s) {
  const int D = p.D;
  if (D <= 48) return launch_df<16, 3, 256, MODE>(p, s);
  if (D <= 64) return launch_df<16, 4, 256, MODE>(p, s);
  if (D <= 96) return launch_df<16, 6, 512, MODE>(p, s);
  return launch_df<32, 4, 512, MODE>(p, s);
}

}  // namespace
}  // namespace stap
