// Covariance per (Doppler bin, range training block) (statement U of the STAP
// kernel, arXiv 2203.06233 Sec. 4.2, read as the sample covariance):
//   cov[k][b] = (1/B) sum_{r in block b} x_{k,r} x_{k,r}^H
// with x_{k,r} the D = C*T snapshot of T adjacent Doppler bins.
//
// Precision: the solve downstream sees covariances whose condition number is
// bounded only by the diagonal load (about 1e3 * D), so rounding R to FP32
// would dominate the weight error.  Each entry is therefore accumulated
// error-free in FP32 pairs on the FP32 pipe and written as FP64; only the final
// conversion touches FP64.  The bin-pair form below, which serves nearly every
// shape, sums on a fixed grid (four FP32 instructions per real product, see
// there).  The general form splits every product a*b exactly into p + e by one
// FMA (TwoProduct), adds p to the running sum with Knuth's TwoSum and collects
// all rounding errors in a second FP32 accumulator (about 10 instructions): the
// result is accurate to about n^2 u^2 times the sum of |terms| (Ogita, Rump &
// Oishi, "Accurate sum and dot product", SISC 2005, Dot2).
//
// Mapping of the general form: a CTA owns NS consecutive blocks of one Doppler bin, stages their
// D x B snapshot tiles in shared memory (chunks of BC cells if B is large) and
// gives each thread whole entries (i >= l) of the lower triangle; the upper
// triangle is written as the conjugate mirror.
#include <algorithm>
#include <cmath>

#include "df64.cuh"
#include "batch.cuh"
#include "checked.cuh"
#include "snapshots.cuh"

namespace stap {
namespace {

struct FF {
  float s, e;  // value = s + e (e collects every rounding error)
};

__device__ __forceinline__ void ff_add_prod(FF& acc, float a, float b) {
  const float p = __fmul_rn(a, b);
  const float pe = __fmaf_rn(a, b, -p);        // a*b = p + pe exactly
  const float t = __fadd_rn(acc.s, p);         // TwoSum(acc.s, p) = t + te exactly
  const float z = __fsub_rn(t, acc.s);
  const float te = __fadd_rn(__fsub_rn(acc.s, __fsub_rn(t, z)), __fsub_rn(p, z));
  acc.s = t;
  acc.e = __fadd_rn(acc.e, __fadd_rn(te, pe));
}

__device__ __forceinline__ void unpack_lower(int q, int& i, int& l) {
  int r = (int)((sqrtf(8.0f * (float)q + 1.0f) - 1.0f) * 0.5f);
  while (r * (r + 1) / 2 > q) --r;
  while ((r + 1) * (r + 2) / 2 <= q) ++r;
  i = r;
  l = q - r * (r + 1) / 2;
}

__global__ void __launch_bounds__(256)
covariance_ff_kernel(const float2* __restrict__ dop, double2* __restrict__ cov, int C, int K, int ldr,
                     int T, int B, int NB, int NS, int BC, double invB) {
  extern __shared__ float2 xs[];  // [NS][D][BC + 1]
  const int k = blockIdx.y;
  const int b0 = blockIdx.x * NS;
  const int D = C * T;
  const int E = D * (D + 1) / 2;
  const int ld = BC + 1;
  const int ns = min(NS, NB - b0);

  for (int c0 = 0; c0 < B; c0 += BC) {
    const int bc = min(BC, B - c0);
    __syncthreads();
    for (int j = 0; j < ns; ++j)
      stage_snapshots(xs + (size_t)j * D * ld, ld, dop, C, K, ldr, T, k, (b0 + j) * B + c0, bc);
    __syncthreads();
    for (int it = threadIdx.x; it < ns * E; it += blockDim.x) {
      const int j = it / E;
      int i, l;
      unpack_lower(it - j * E, i, l);
      const float2* xi = xs + ((size_t)j * D + i) * ld;
      const float2* xl = xs + ((size_t)j * D + l) * ld;
      FF re{0.f, 0.f}, im{0.f, 0.f};
      for (int rr = 0; rr < bc; ++rr) {
        const float2 a = xi[rr], b = xl[rr];
        // a * conj(b) = (a.x b.x + a.y b.y) + i (a.y b.x - a.x b.y)
        ff_add_prod(re, a.x, b.x);
        ff_add_prod(re, a.y, b.y);
        ff_add_prod(im, a.y, b.x);
        ff_add_prod(im, -a.x, b.y);
      }
      double vr = (ff::f2d_exact(re.s) + ff::f2d_exact(re.e)) * invB;
      double vi = (ff::f2d_exact(im.s) + ff::f2d_exact(im.e)) * invB;
      double2* out = cov + ((size_t)k * NB + b0 + j) * (size_t)D * D;
      if (c0 > 0) {  // later chunks add to what earlier chunks wrote (same thread owns the entry)
        const double2 prev = out[(size_t)i * D + l];
        vr += prev.x;
        vi += prev.y;
      }
      if (i == l) vi = 0.0;
      out[(size_t)i * D + l] = make_double2(vr, vi);
      if (i != l) out[(size_t)l * D + i] = make_double2(vr, ff::dneg(vi));
    }
  }
}

// ---------------------------------------------------------------------------
// Bin-pair form.  Block (t, t') of R_k is the cross-covariance of bins
// k + m_t and k + m_t' (m_t = t - floor(T/2)):
//   R_k[(t,c),(t',c')] = Q(k + m_t, k + m_t')[c][c'],
//   Q(k1, k2)[c][c'] = (1/B) sum_r X_c(k1, r) conj(X_c'(k2, r)),
// and Q(k2, k1) = Q(k1, k2)^H.  Neighbouring bins share these blocks, so a CTA
// that owns KT consecutive bins of one range block computes every Q(k1, k1+d),
// d < T, once (C(C+1)/2 entries for d = 0, C^2 otherwise) and assembles its KT
// covariances from them: T C^2 - C(C-1)/2 products per bin instead of
// D(D+1)/2.
//
// Accumulation on a fixed grid (error-free transformation in the manner of
// Rump, Ogita & Oishi, "Accurate floating-point summation part I", SISC 2008,
// ExtractScalar).  An entry's partial sums, and the products in them, are at
// most n1 n2 in magnitude, the product of its two rows' 2-norms over the cells
// (Cauchy and Schwarz, for any subset of the terms), so with a power of two
// sig >= 2 n1 n2 a running sum that starts at 1.5 sig stays inside [sig, 2 sig),
// where floats are the multiples of ulp(sig).  Each product is added by
// t = fma(a, b, s), which rounds the product onto that grid; q = t - s is
// exact, and what the grid left out, fma(a, b, -q) (|.| <= ulp(sig) / 2), goes
// to a second FP32 accumulator: four FP32 instructions per real product.  At
// the end s - 1.5 sig is exact, and the pair is combined in FP64.  (Bounding
// the sums by 4 B m1 m2 with the rows' maxima, as before, takes a fifth
// instruction -- the sums then start at zero beside the grid constant -- on a
// grid about eight times coarser for noise-like rows.)
//
// A thread computes one entry, two cells per pair of 16-byte reads of shared
// memory for 32 FP32 instructions.  The row pitch is an odd number of 16-byte
// units, so eight lanes reading eight consecutive rows touch all the banks
// once.  (Two by two entries per thread halve the reads but leave a quarter
// of the warps: slower but for D = 64, 5% there.)
// Measured, before and after: C16 K256 R4096 T4 B128 (D = 64) 1387 -> 1036 us;
// C8 K256 R8192 T3 B64 (D = 24) 577 -> 433; C4 K256 R4096 T3 B64 (D = 12) 79.1 ->
// 69; error against 64 bits at D = 64 5.6e-12 -> 7.6e-13.
constexpr float kFar = 0x1p40f;         // see the rows' norms
constexpr int kPairMaxThreads = 1024;   // one thread per entry, up to this

__device__ __forceinline__ float pow2_ceil(float x) {  // smallest power of two >= x, at most 2^126
  if (!(x > 0.f)) return 1.0f;
  unsigned u = __float_as_uint(x);
  unsigned e = u >> 23;
  if (u & 0x7fffffu) e += 1;
  if (e < 1) e = 1;
  if (e > 253) e = 253;
  return __uint_as_float(e << 23);
}

// s += a b on the grid, the remainder to lo
__device__ __forceinline__ void grid_add(float& s, float& lo, float a, float b) {
  const float t = __fmaf_rn(a, b, s);
  const float q = __fsub_rn(t, s);
  lo = __fadd_rn(lo, __fmaf_rn(a, b, -q));
  s = t;
}

// Parameters of one bin-pair launch (one CPI): grid gx = NB blocks by K / KT
// bin groups.
struct CovPairsParams {
  const float2* dop;
  double2* cov;
  int C, K, ldr, T, B, NB, KT, CB;
  int lower;       // write only the lower triangle
  double invB;
  int gx;
};

// row pitch in cells: at least cb, and an odd number of 16-byte units
__host__ __device__ constexpr int pair_ld(int cb) { return (cb + 1) / 4 * 4 + 2; }

// SHORT: blocks of up to kShort cells, where an entry's few cells do not hide its
// latency and the matrices' stores are most of the work: 32 registers, i.e. 64
// warps per SM instead of 51, without the unrolling.  (D = 15 K64 R8192 B4: 494
// -> 385 us; B 32: 3% better, B 50: 2% worse)
constexpr int kShort = 32;

template <bool SHORT>
__device__ __forceinline__ void covariance_pairs_body(const CovPairsParams& prm, int bx, int by) {
  const float2* __restrict__ dop = prm.dop;
  double2* __restrict__ cov = prm.cov;
  const int C = prm.C, K = prm.K, ldr = prm.ldr, T = prm.T, B = prm.B, NB = prm.NB, KT = prm.KT,
            CB = prm.CB;
  const double invB = prm.invB;
  extern __shared__ double2 smd[];
  const int b = bx;
  const int k0 = by * KT;
  const int h = T / 2;
  const int NBIN = KT + T - 1;                    // staged bins k0-h .. k0+KT-1+(T-1-h)
  const int nrows = NBIN * C;
  const int ld = pair_ld(CB);
  const int Ediag = C * (C + 1) / 2, Eoff = C * C;
  // entries: d-major; d = 0 has NBIN * Ediag, d > 0 has (NBIN - d) * Eoff
  const int nitems = NBIN * Ediag + (T - 1) * (2 * NBIN - T) / 2 * Eoff;
  double2* Q = smd;                                             // [nitems]
  float* m = reinterpret_cast<float*>(Q + nitems);              // [nrows] row norms
  float2* X = reinterpret_cast<float2*>(m + ((nrows + 3) & ~3));  // [nrows][ld]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const bool pow2B = (B & (B - 1)) == 0;
  const float invBf = 1.0f / (float)B;
  // the B cells in chunks of CB: each chunk is summed error-free on its own
  // grid and added to Q in FP64
  for (int c0 = 0; c0 < B; c0 += CB) {
    const int cc = min(CB, B - c0);
    const int ce = (cc + 1) & ~1;                  // cells come in pairs: a zero follows an odd last one
    __syncthreads();
    for (int row = warp; row < nrows; row += nwarps) {   // rows (bin j, channel c)
      const int j = row / C, c = row - j * C;
      const int kk = wrap_bin(k0 - h + j, K);
      const float2* src = dop + ((size_t)c * K + kk) * ldr + (size_t)b * B + c0;
      float2* dst = X + row * ld;
      float ss = 0.f;
      for (int cell = lane; cell < ce; cell += 32) {
        const bool ok = cell < cc && in_bounds(((long long)c * K + kk) * ldr + (long long)b * B + c0 + cell,
                                               ((long long)C * K - 1) * ldr + (long long)NB * B, kSiteCovIn);
        const float2 x = ok ? __ldg(src + cell) : make_float2(0.f, 0.f);
        dst[cell] = x;
        ss = fmaf(x.x, x.x, ss);
        ss = fmaf(x.y, x.y, ss);
      }
      for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
      float n = sqrtf(ss);
      if (!(ss > 1e-24f && ss < 1e36f)) {          // warp-uniform: squares may have over- or underflowed
        // again from values scaled by the power of two next to the largest; a
        // row with an infinity or NaN keeps its largest value, its entries are
        // not finite either.  A row whose norm is beyond 2^62 is kept divided by
        // kFar, with the sign of its norm as the mark, so that the grid and
        // the sums of any two rows whose own sums FP32 holds stay inside it
        float mx = 0.f;
        for (int cell = lane; cell < cc; cell += 32) mx = fmaxf(mx, fmaxf(fabsf(dst[cell].x), fabsf(dst[cell].y)));
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        n = mx;
        if (mx > 0.f && mx < __int_as_float(0x7f800000)) {
          const float up = pow2_ceil(mx), dn = 1.0f / up;
          ss = 0.f;
          for (int cell = lane; cell < cc; cell += 32) {
            const float2 x = dst[cell];
            ss = fmaf(x.x * dn, x.x * dn, ss);
            ss = fmaf(x.y * dn, x.y * dn, ss);
          }
          for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
          n = up * sqrtf(ss);
          if (n > 0x1p62f) {
            __syncwarp();
            for (int cell = lane; cell < cc; cell += 32) {
              dst[cell].x *= 1.0f / kFar;
              dst[cell].y *= 1.0f / kFar;
            }
            n = -(up * (1.0f / kFar)) * sqrtf(ss);
          }
        }
      }
      if (lane == 0) m[row] = n;
    }
    __syncthreads();

    for (int it = threadIdx.x; it < nitems; it += blockDim.x) {
      int d = 0, rem = it;
      if (rem >= NBIN * Ediag) {
        rem -= NBIN * Ediag;
        d = 1;
        while (rem >= (NBIN - d) * Eoff) {
          rem -= (NBIN - d) * Eoff;
          ++d;
        }
      }
      int j1, c1, c2;
      if (d == 0) {
        j1 = rem / Ediag;
        unpack_lower(rem - j1 * Ediag, c1, c2);
      } else {
        j1 = rem / Eoff;
        const int e = rem - j1 * Eoff;
        c1 = e / C;
        c2 = e - c1 * C;
      }
      const int ra = j1 * C + c1, rb = (j1 + d) * C + c2;
      const float4* xa = reinterpret_cast<const float4*>(X + ra * ld);   // two cells each
      const float4* xb = reinterpret_cast<const float4*>(X + rb * ld);
      const float na = m[ra], nb = m[rb];
      const float s0 = 1.5f * pow2_ceil(fabsf(2.01f * na * nb));
      float sr = s0, si = s0, lr = 0.f, li = 0.f;
#pragma unroll (SHORT ? 1 : 4)
      for (int p = 0; p < ce / 2; ++p) {
        const float4 a = xa[p], bb = xb[p];
        grid_add(sr, lr, a.x, bb.x);
        grid_add(si, li, a.y, bb.x);
        grid_add(sr, lr, a.y, bb.y);
        grid_add(si, li, -a.x, bb.y);
        grid_add(sr, lr, a.z, bb.z);
        grid_add(si, li, a.w, bb.z);
        grid_add(sr, lr, a.w, bb.w);
        grid_add(si, li, -a.z, bb.w);
      }
      const float hr = __fsub_rn(sr, s0), hi = __fsub_rn(si, s0);   // exact
      double2 v;
      if (pow2B) {  // 1/B is a power of two: scaling the pair in FP32 is exact
        v = make_double2(ff::f2d_exact(hr * invBf) + ff::f2d_exact(lr * invBf),
                         ff::f2d_exact(hi * invBf) + ff::f2d_exact(li * invBf));
      } else {
        v = make_double2((ff::f2d_exact(hr) + ff::f2d_exact(lr)) * invB, (ff::f2d_exact(hi) + ff::f2d_exact(li)) * invB);
      }
      if (na < 0.f || nb < 0.f) {                  // rows kept divided by kFar
        const double f = (na < 0.f ? (double)kFar : 1.0) * (nb < 0.f ? (double)kFar : 1.0);
        v.x *= f;
        v.y *= f;
      }
      if (c0 > 0) {
        const double2 p = Q[it];
        v.x += p.x;
        v.y += p.y;
      }
      Q[it] = v;
    }
  }
  __syncthreads();

  // assemble R_k for the KT bins of this tile
  const int D = C * T;
  auto qat = [&](int j1, int d, int c1, int c2) -> double2 {  // Q(bin j1, bin j1+d)[c1][c2]
    if (d == 0) {
      if (c1 >= c2) return Q[j1 * Ediag + c1 * (c1 + 1) / 2 + c2];
      const double2 v = Q[j1 * Ediag + c2 * (c2 + 1) / 2 + c1];
      return make_double2(v.x, ff::dneg(v.y));
    }
    // blocks d' < d come first: NBIN Ediag + sum_{e=1}^{d-1} (NBIN - e) Eoff
    const int off = NBIN * Ediag + Eoff * ((d - 1) * NBIN - d * (d - 1) / 2);
    return Q[off + j1 * Eoff + c1 * C + c2];
  };
  for (int idx = threadIdx.x; idx < KT * D * D; idx += blockDim.x) {
    const int kl = idx / (D * D);
    const int e = idx - kl * D * D;
    const int i = e / D, l = e - i * D;
    if (prm.lower && l > i) continue;
    const int t1 = i / C, c1 = i - t1 * C, t2 = l / C, c2 = l - t2 * C;
    double2 v;
    if (t1 <= t2) {
      v = qat(kl + t1, t2 - t1, c1, c2);
    } else {
      const double2 w = qat(kl + t2, t1 - t2, c2, c1);
      v = make_double2(w.x, ff::dneg(w.y));
    }
    if (i == l) v.y = 0.0;
    const long long o = (((long long)(k0 + kl) * NB + b) * D + i) * D + l;
    if (in_bounds(o, (long long)K * NB * D * D, kSiteCovOut)) cov[o] = v;
  }
}

template <bool SHORT>
__global__ void __launch_bounds__(kPairMaxThreads, SHORT ? 2 : 0)   // (0: no say)
covariance_pairs_kernel(CovPairsParams p) {
  covariance_pairs_body<SHORT>(p, blockIdx.x, blockIdx.y);
}

// the same covariances as a persistent launch over the CPIs of a batch
template <bool SHORT>
__global__ void __launch_bounds__(kPairMaxThreads, SHORT ? 2 : 0)
covariance_pairs_batched(BatchCtl ctl) {
  batched_loop<CovPairsParams>(ctl, [&](const CovPairsParams& p, int bx, int by, int) {
    covariance_pairs_body<SHORT>(p, bx, by);
  });
}

template <bool SHORT>
cudaError_t launch_pairs(const CovPairsParams& p, dim3 grid, int threads, size_t smem, cudaStream_t s) {
  static int set_bytes[64] = {0}, set_bytes_b[64] = {0};
  cudaError_t e = ensure_smem(covariance_pairs_kernel<SHORT>, smem, set_bytes);
  if (e == cudaSuccess) e = ensure_smem(covariance_pairs_batched<SHORT>, smem, set_bytes_b);
  if (e != cudaSuccess) return e;
  return launch_params(reinterpret_cast<const void*>(covariance_pairs_kernel<SHORT>),
                       reinterpret_cast<const void*>(covariance_pairs_batched<SHORT>), grid, threads, smem, s, p);
}

// Entries of KT bins, and the threads that take them: whole warps, at most
// kPairMaxThreads with the rounds balanced above that.
int pair_items(int C, int T, int KT) {
  const int nbin = KT + T - 1;
  return nbin * (C * (C + 1) / 2) + (T - 1) * (2 * nbin - T) / 2 * C * C;
}
int pair_threads(int items) {
  const int rounds = (items + kPairMaxThreads - 1) / kPairMaxThreads;
  const int threads = ((items + rounds - 1) / rounds + 31) / 32 * 32;
  return threads < 64 ? 64 : threads;
}

}  // namespace

cudaError_t launch_covariance_fp32(const float2* dop, double2* cov, int C, int K, int R, int ldr,
                                   int T, int B, cudaStream_t s, const Tune& tn, bool lower_only) {
  const int D = C * T;
  const int E = D * (D + 1) / 2;
  const int NB = R / B;
  if (NB == 0) return cudaSuccess;
  // bin-pair kernel: the B cells of KT + T - 1 bins in shared memory, in
  // chunks of CB cells when the whole block does not fit
  {
    constexpr size_t kPairBudget = 200 * 1024;
    auto pair_smem = [&](int kt, int cb) {
      const size_t nrows = (size_t)(kt + T - 1) * C;
      return (size_t)pair_items(C, T, kt) * sizeof(double2) + ((nrows + 3) & ~(size_t)3) * sizeof(float) +
             nrows * pair_ld(cb) * sizeof(float2);
    };
    // Bins per CTA, the least time by a model of the rounds of CTAs over the
    // SMs: more bins share more products, but fewer CTAs fit an SM beside one
    // another, and w resident warps reach about w / (w + 12) of the issue rate
    // (fitted to the measured times of KT = 1 .. 16 at ten shapes of D = 4 to
    // 80; within 9% of the fastest KT on each).
    int KT = 1;
    double best = 1e300;
    for (int kt = 1; kt <= 16 && kt <= K; kt *= 2) {   // K is a power of two, so kt divides it
      const size_t sm = pair_smem(kt, B);
      if (sm > kPairBudget) break;
      const int items = pair_items(C, T, kt), threads = pair_threads(items);
      const int slots = (items + threads - 1) / threads * threads;   // whole rounds of the CTA
      const double ctas = (double)NB * (K / kt), warps = threads / 32;
      double per = (double)((228 * 1024) / (sm + 1024));             // CTAs per SM: shared memory,
      per = std::min({per, std::floor((B <= kShort ? 64.0 : 51.0) / warps), std::ceil(ctas / 152.0)});   // registers, the grid
      if (per < 1.0) per = 1.0;
      const double w = per * warps;
      const double t = std::max(ctas / (152.0 * per), 1.0) * per * slots * (w + 12.0) / w;
      if (t < best) {
        best = t;
        KT = kt;
      }
    }
    if (tn.cov_kt > 0 && tn.cov_kt <= K && K % tn.cov_kt == 0 && pair_smem(tn.cov_kt, B) <= kPairBudget)
      KT = tn.cov_kt;
    int CB = B;
    while (CB > 32 && pair_smem(KT, CB) > kPairBudget) CB = (CB + 1) / 2;
    if (pair_smem(KT, CB) <= kPairBudget) {
      const size_t smem = pair_smem(KT, CB);
      dim3 grid(NB, K / KT);
      const CovPairsParams p{dop, cov, C, K, ldr, T, B, NB, KT, CB, lower_only ? 1 : 0, 1.0 / (double)B, (int)grid.x};
      const int threads = pair_threads(pair_items(C, T, KT));
      return B <= kShort ? launch_pairs<true>(p, grid, threads, smem, s) : launch_pairs<false>(p, grid, threads, smem, s);
    }
  }
  // general form: one tile per system, cells in chunks
  constexpr size_t kSmemBudget = 96 * 1024;
  int BC = B;
  if ((size_t)D * (BC + 1) * sizeof(float2) > kSmemBudget)
    BC = (int)(kSmemBudget / ((size_t)D * sizeof(float2))) - 1;
  if (BC < 1) return cudaErrorInvalidValue;
  int NS = E >= 256 ? 1 : 256 / E;
  NS = min(NS, NB);
  while (NS > 1 && (size_t)NS * D * (BC + 1) * sizeof(float2) > kSmemBudget) --NS;
  const size_t smem = (size_t)NS * D * (BC + 1) * sizeof(float2);
  static int set_bytes[64] = {0};
  cudaError_t e = ensure_smem(covariance_ff_kernel, smem, set_bytes);
  if (e != cudaSuccess) return e;
  dim3 grid((NB + NS - 1) / NS, K);
  return launch_or_defer(s, [=](cudaStream_t st) {
    covariance_ff_kernel<<<grid, 256, smem, st>>>(dop, cov, C, K, ldr, T, B, NB, NS, BC, 1.0 / (double)B);
    return cudaGetLastError();
  });
}

}  // namespace stap

namespace stap {
cudaError_t check_record_covariance(CheckRecord* out) { return read_check_record(out); }
}  // namespace stap
