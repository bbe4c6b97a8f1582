// Weight application: output power of every range-Doppler cell,
//   out[s][k][r] = | w_{k, r/B, s}^H x_{k,r} |^2,
// the last step of the STAP kernel of arXiv 2203.06233 Sec. 4.2 (the adaptive
// filter output |w^H x|^2).
//
// Two kernels: a tiled one for any shape, and a register-resident one for
// small even D.  Both sum over the snapshot entries in increasing order with
// the same FMAs, so their results are the same bit for bit.
#include "batch.cuh"
#include "checked.cuh"
#include "snapshots.cuh"

namespace stap {
namespace {

// Parameters of one apply launch (one CPI); gx = the launch's grid.x.
struct ApplyParams {
  const float2* dop;
  const float2* wts;
  float* out;
  int C, K, R, ldr, T, B, S;
  int nct, nst;   // tiled kernel: cell tiles per training block, steering tiles
  int gx;
};

// Tiled form: a CTA owns one training block's tile of up to 32 CELLS range
// cells of one Doppler bin and up to 64 steering vectors, a GEMM of [S][D]
// weights by [D][cells] snapshots.  Warp w owns 8 steering vectors, a lane
// CELLS cells: 8 CELLS complex accumulators in registers, fed per snapshot
// entry by CELLS / 2 16-byte reads of its cells and four broadcast 16-byte
// reads of the warp's weights for 32 CELLS FMAs, so that the FP32 pipe and not
// shared memory bounds it.  Both operands come in chunks of DC snapshot
// entries, two buffers filled by cp.async (8 bytes each: any alignment of the
// range axis, and the weights land transposed), the next chunk in flight
// under this chunk's FMAs.  CELLS = 4, 2 or 1 by the block size, so that a
// tile is not mostly empty lanes.
//
// Before: one cell and 8 steering vectors per thread, the whole [D][256]
// tile staged, then computed, by the one CTA that fits an SM.  C16 K256 R4096
// T4 B128 S32 (D = 64): 1326 -> 417 us (41 TFLOP/s); C32 K512 R2048 T4 B256 S64
// (D = 128): 4201 -> 1492 us (46 TFLOP/s).
constexpr int DC = 16;         // snapshot entries per chunk
constexpr int kTileS = 64;     // steering vectors per CTA at most

__device__ __forceinline__ void cp_async8(void* dst, const void* src, bool valid) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  const int n = valid ? 8 : 0;   // 0: the eight bytes are zeroed, nothing is read
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}

template <int CELLS>
__device__ __forceinline__ void apply_tile_body(const ApplyParams& prm, int bx, int by) {
  const float2* __restrict__ dop = prm.dop;
  const float2* __restrict__ wts = prm.wts;
  float* __restrict__ out = prm.out;
  const int C = prm.C, K = prm.K, R = prm.R, ldr = prm.ldr, T = prm.T, B = prm.B, S = prm.S;
  constexpr int RT = 32 * CELLS;
  extern __shared__ float4 sm4[];
  __shared__ long long rowbase[128];               // dop offset of snapshot row d
  const int nw = blockDim.x >> 5, SP = 8 * nw + 2;
  float2* xs = reinterpret_cast<float2*>(sm4);     // [2][DC][RT]
  float2* ws = xs + 2 * DC * RT;                   // [2][DC][SP]
  const int D = C * T, NB = R / B;
  const int k = by;
  const int st = bx % prm.nst, bt = bx / prm.nst;
  const int b = bt / prm.nct, ct = bt - b * prm.nct;
  const int tc = (B + prm.nct - 1) / prm.nct;      // cells of a tile
  const int c0 = ct * tc, nc = min(tc, B - c0);    // the tile's first cell in the block, its cells
  const int r0 = b * B + c0;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int d = tid; d < D; d += blockDim.x) {
    const int t = d / C, c = d - t * C;
    rowbase[d] = ((long long)c * K + wrap_bin(k + t - T / 2, K)) * ldr + r0;
  }
  __syncthreads();
  const long long w0 = (((long long)k * NB + b) * S + st * kTileS) * D;
  const int ns = min(kTileS, S - st * kTileS);     // this CTA's steering vectors
  auto fill = [&](int d0, int buf) {
    const int dn = min(DC, D - d0);
    for (int e = tid; e < dn * RT; e += blockDim.x) {
      const int d = e / RT, c = e % RT;
      const long long o = rowbase[d0 + d] + c;
      const bool ok = c < nc && in_bounds(o, ((long long)C * K - 1) * ldr + R, kSiteApplyIn);
      cp_async8(xs + (buf * DC + d) * RT + c, dop + (ok ? o : 0), ok);
    }
    for (int e = tid; e < 8 * nw * DC; e += blockDim.x) {
      const int s = e / DC, d = e % DC;
      const long long o = w0 + (long long)s * D + d0 + d;
      const bool ok = s < ns && d < dn && in_bounds(o, (long long)K * NB * S * D, kSiteApplyIn);
      cp_async8(ws + (buf * DC + d) * SP + s, wts + (ok ? o : 0), ok);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float2 acc[8][CELLS];
#pragma unroll
  for (int s = 0; s < 8; ++s)
#pragma unroll
    for (int c = 0; c < CELLS; ++c) acc[s][c] = make_float2(0.f, 0.f);
  fill(0, 0);
  const int nch = (D + DC - 1) / DC;
  for (int ch = 0; ch < nch; ++ch) {
    const int buf = ch & 1;
    if (ch + 1 < nch) {
      fill((ch + 1) * DC, buf ^ 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const int dn = min(DC, D - ch * DC);
    const float2* xb = xs + buf * DC * RT;
    const float2* wb = ws + buf * DC * SP + 8 * warp;
#pragma unroll 2
    for (int d = 0; d < dn; ++d) {
      float2 x[CELLS];
      if constexpr (CELLS == 1) {
        x[0] = xb[d * RT + lane];
      } else {
#pragma unroll
        for (int c = 0; c < CELLS; c += 2) {       // cells 32 c + 2 lane and the next
          const float4 v = *reinterpret_cast<const float4*>(xb + d * RT + 32 * c + 2 * lane);
          x[c] = make_float2(v.x, v.y);
          x[c + 1] = make_float2(v.z, v.w);
        }
      }
#pragma unroll
      for (int s = 0; s < 8; s += 2) {
        const float4 w = *reinterpret_cast<const float4*>(wb + d * SP + s);
#pragma unroll
        for (int c = 0; c < CELLS; ++c) {          // acc += conj(w) x
          acc[s][c].x = fmaf(w.x, x[c].x, acc[s][c].x);
          acc[s][c].x = fmaf(w.y, x[c].y, acc[s][c].x);
          acc[s][c].y = fmaf(w.x, x[c].y, acc[s][c].y);
          acc[s][c].y = fmaf(-w.y, x[c].x, acc[s][c].y);
          acc[s + 1][c].x = fmaf(w.z, x[c].x, acc[s + 1][c].x);
          acc[s + 1][c].x = fmaf(w.w, x[c].y, acc[s + 1][c].x);
          acc[s + 1][c].y = fmaf(w.z, x[c].y, acc[s + 1][c].y);
          acc[s + 1][c].y = fmaf(-w.w, x[c].x, acc[s + 1][c].y);
        }
      }
    }
    __syncthreads();                               // the buffer is refilled next
  }
  const long long ext = ((long long)S * K - 1) * ldr + R;
  const bool even = ((r0 | ldr) & 1) == 0 && (reinterpret_cast<uintptr_t>(out) & 7) == 0;
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    if (8 * warp + s >= ns) break;
    const long long o = ((long long)(st * kTileS + 8 * warp + s) * K + k) * ldr + r0;
    float p[CELLS];
#pragma unroll
    for (int c = 0; c < CELLS; ++c) p[c] = fmaf(acc[s][c].x, acc[s][c].x, acc[s][c].y * acc[s][c].y);
    if constexpr (CELLS == 1) {
      if (lane < nc && in_bounds(o + lane, ext, kSiteApplyOut)) out[o + lane] = p[0];
    } else {
#pragma unroll
      for (int c = 0; c < CELLS; c += 2) {
        const int cell = 32 * c + 2 * lane;
        if (even && cell + 1 < nc) {
          if (in_bounds(o + cell + 1, ext, kSiteApplyOut))
            *reinterpret_cast<float2*>(out + o + cell) = make_float2(p[c], p[c + 1]);
        } else {
          if (cell < nc && in_bounds(o + cell, ext, kSiteApplyOut)) out[o + cell] = p[c];
          if (cell + 1 < nc && in_bounds(o + cell + 1, ext, kSiteApplyOut)) out[o + cell + 1] = p[c + 1];
        }
      }
    }
  }
}

template <int CELLS>
__global__ void __launch_bounds__(256, CELLS == 4 ? 2 : (CELLS == 2 ? 3 : 4))
apply_tile_kernel(ApplyParams p) {
  apply_tile_body<CELLS>(p, blockIdx.x, blockIdx.y);
}

// the same apply as a persistent launch over the CPIs of a batch
template <int CELLS>
__global__ void __launch_bounds__(256, CELLS == 4 ? 2 : (CELLS == 2 ? 3 : 4))
apply_tile_batched(BatchCtl ctl) {
  batched_loop<ApplyParams>(ctl, [&](const ApplyParams& p, int bx, int by, int) {
    apply_tile_body<CELLS>(p, bx, by);
  });
}

template <int CELLS>
cudaError_t launch_apply_tile(const float2* dop, const float2* wts, float* out, int C, int K, int R, int ldr,
                              int T, int B, int S, cudaStream_t s) {
  constexpr int RT = 32 * CELLS;
  const int nct = (B + RT - 1) / RT, nst = (S + kTileS - 1) / kTileS;
  const int nw = (min(S, kTileS) + 7) / 8;
  const size_t smem = 2 * (size_t)DC * (RT + 8 * nw + 2) * sizeof(float2);
  static int set_bytes[64] = {0}, set_bytes_b[64] = {0};
  cudaError_t e = ensure_smem(apply_tile_kernel<CELLS>, smem, set_bytes);
  if (e == cudaSuccess) e = ensure_smem(apply_tile_batched<CELLS>, smem, set_bytes_b);
  if (e != cudaSuccess) return e;
  dim3 grid((unsigned)(R / B) * nct * nst, K);
  const ApplyParams p{dop, wts, out, C, K, R, ldr, T, B, S, nct, nst, (int)grid.x};
  return launch_params(reinterpret_cast<const void*>(apply_tile_kernel<CELLS>),
                       reinterpret_cast<const void*>(apply_tile_batched<CELLS>), grid, 32 * nw, smem, s, p);
}

// Register-resident form for small even D (the common shapes).  A thread owns
// two adjacent range cells: their 2 x D snapshot entries are loaded straight
// from the Doppler cube with one 16-byte load per entry (coalesced along
// range; T neighbouring bins are re-read through L2 by neighbouring CTAs) and
// stay in registers, while the weights of the CTA's blocks sit in shared
// memory as [block][s][d].  For each steering vector the thread reads its
// weights as D/2 broadcast 16-byte loads and does 8 D FMAs: FMA-bound.
// 128-thread CTAs: in a one-CPI run the apply of one range slab shares the
// SMs with the solves of others, and a smaller CTA takes fewer of a
// solve's warp slots (registers, shared memory) wherever it lands.
constexpr int kRegThreads = 128;
constexpr int kRegCells = 2 * kRegThreads;  // range cells per CTA

// registers: 64 while the snapshots fit, more for larger D
template <int D>
__device__ __forceinline__ void apply_reg_body(const ApplyParams& prm, int bx, int by) {
  const float2* __restrict__ dop = prm.dop;
  const float2* __restrict__ wts = prm.wts;
  float* __restrict__ out = prm.out;
  const int C = prm.C, K = prm.K, R = prm.R, ldr = prm.ldr, T = prm.T, B = prm.B, S = prm.S;
  extern __shared__ float4 sm4[];
  float2* ws = reinterpret_cast<float2*>(sm4);    // [nblk][S][D]
  const int NB = R / B;
  const int k = by;
  const int cta_r0 = bx * kRegCells;
  const int jb0 = cta_r0 / B;
  const int jb1 = min(NB - 1, (min(cta_r0 + kRegCells, R) - 1) / B);
  const int nblk = jb1 - jb0 + 1;
  {
    const float2* src = wts + ((size_t)k * NB + jb0) * S * D;
    const int n = nblk * S * D;
    for (int i = threadIdx.x; i < n; i += blockDim.x)
      ws[i] = in_bounds(((long long)k * NB + jb0) * S * D + i, (long long)K * NB * S * D, kSiteApplyIn)
                  ? __ldg(src + i) : make_float2(0.f, 0.f);
  }
  const int r0 = cta_r0 + 2 * threadIdx.x;
  float4 x[D];                                    // (cell r0, cell r0 + 1) per entry
  if (r0 < R) {
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const int t = d / C, c = d - t * C;
      const int kk = wrap_bin(k + t - T / 2, K);
      const long long o = ((long long)c * K + kk) * ldr + r0;
      x[d] = in_bounds(o + 1, ((long long)C * K - 1) * ldr + R, kSiteApplyIn)
                 ? __ldg(reinterpret_cast<const float4*>(dop + o)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  __syncthreads();
  if (r0 >= R) return;
  const int j = r0 / B - jb0;                      // B even: both cells in one block
  const float4* wj = reinterpret_cast<const float4*>(ws + (size_t)j * S * D);
  for (int s = 0; s < S; ++s) {
    float a0r = 0.f, a0i = 0.f, a1r = 0.f, a1i = 0.f;
#pragma unroll
    for (int d2 = 0; d2 < D / 2; ++d2) {
      const float4 w = wj[s * (D / 2) + d2];        // w_d = (w.x, w.y), w_{d+1} = (w.z, w.w)
      const float4 xa = x[2 * d2], xb = x[2 * d2 + 1];
      // acc += conj(w) * x for both cells
      a0r = fmaf(w.x, xa.x, a0r); a0r = fmaf(w.y, xa.y, a0r);
      a0i = fmaf(w.x, xa.y, a0i); a0i = fmaf(-w.y, xa.x, a0i);
      a1r = fmaf(w.x, xa.z, a1r); a1r = fmaf(w.y, xa.w, a1r);
      a1i = fmaf(w.x, xa.w, a1i); a1i = fmaf(-w.y, xa.z, a1i);
      a0r = fmaf(w.z, xb.x, a0r); a0r = fmaf(w.w, xb.y, a0r);
      a0i = fmaf(w.z, xb.y, a0i); a0i = fmaf(-w.w, xb.x, a0i);
      a1r = fmaf(w.z, xb.z, a1r); a1r = fmaf(w.w, xb.w, a1r);
      a1i = fmaf(w.z, xb.w, a1i); a1i = fmaf(-w.w, xb.z, a1i);
    }
    if (in_bounds(((long long)s * K + k) * ldr + r0 + 1, ((long long)S * K - 1) * ldr + R, kSiteApplyOut))
      *reinterpret_cast<float2*>(out + ((size_t)s * K + k) * ldr + r0) =
          make_float2(fmaf(a0r, a0r, a0i * a0i), fmaf(a1r, a1r, a1i * a1i));
  }
}

template <int D>
__global__ void __launch_bounds__(kRegThreads, D <= 12 ? 8 : (D <= 18 ? 6 : 4))
apply_reg_kernel(ApplyParams p) {
  apply_reg_body<D>(p, blockIdx.x, blockIdx.y);
}

template <int D>
__global__ void __launch_bounds__(kRegThreads, D <= 12 ? 8 : (D <= 18 ? 6 : 4))
apply_reg_batched(BatchCtl ctl) {
  batched_loop<ApplyParams>(ctl, [&](const ApplyParams& p, int bx, int by, int) {
    apply_reg_body<D>(p, bx, by);
  });
}

template <int D>
cudaError_t launch_apply_reg(const float2* dop, const float2* wts, float* out, int C, int K, int R,
                             int ldr, int T, int B, int S, cudaStream_t s) {
  const int NB = R / B;
  const int max_blk = kRegCells / B + 2;
  const size_t smem = (size_t)(max_blk < NB ? max_blk : NB) * S * D * sizeof(float2);
  static int set_bytes[64] = {0}, set_bytes_b[64] = {0};
  cudaError_t e = ensure_smem(apply_reg_kernel<D>, smem, set_bytes);
  if (e == cudaSuccess) e = ensure_smem(apply_reg_batched<D>, smem, set_bytes_b);
  if (e != cudaSuccess) return e;
  dim3 grid((R + kRegCells - 1) / kRegCells, K);
  const ApplyParams p{dop, wts, out, C, K, R, ldr, T, B, S, 1, 1, (int)grid.x};
  return launch_params(reinterpret_cast<const void*>(apply_reg_kernel<D>),
                       reinterpret_cast<const void*>(apply_reg_batched<D>), grid, kRegThreads, smem, s, p);
}

}  // namespace

cudaError_t launch_apply(const float2* dop, const float2* wts, float* out, int C, int K, int R,
                         int ldr, int T, int B, int S, cudaStream_t s, const Tune& tn) {
  const int D = C * T;
  const int NB = R / B;
  if (NB == 0) return cudaSuccess;
  // register-resident form: even D <= 24, even B and row stride (cell pairs
  // never straddle a block and 16-byte loads stay aligned), weights of a CTA
  // within 160 KB
  const bool aligned = (reinterpret_cast<uintptr_t>(dop) & 15) == 0 &&
                       (reinterpret_cast<uintptr_t>(out) & 7) == 0 && ldr % 2 == 0;
  if (tn.apply_kind != 2 && aligned && D % 2 == 0 && D <= 24 && B % 2 == 0 &&
      (size_t)(kRegCells / B + 2) * S * D * sizeof(float2) <= 160 * 1024) {
    switch (D) {
      case 2: return launch_apply_reg<2>(dop, wts, out, C, K, R, ldr, T, B, S, s);
      case 4: return launch_apply_reg<4>(dop, wts, out, C, K, R, ldr, T, B, S, s);
      case 6: return launch_apply_reg<6>(dop, wts, out, C, K, R, ldr, T, B, S, s);
      case 8: return launch_apply_reg<8>(dop, wts, out, C, K, R, ldr, T, B, S, s);
      case 10: return launch_apply_reg<10>(dop, wts, out, C, K, R, ldr, T, B, S, s);
      case 12: return launch_apply_reg<12>(dop, wts, out, C, K, R, ldr, T, B, S, s);
      case 14: return launch_apply_reg<14>(dop, wts, out, C, K, R, ldr, T, B, S, s);
      case 16: return launch_apply_reg<16>(dop, wts, out, C, K, R, ldr, T, B, S, s);
      case 18: return launch_apply_reg<18>(dop, wts, out, C, K, R, ldr, T, B, S, s);
      case 20: return launch_apply_reg<20>(dop, wts, out, C, K, R, ldr, T, B, S, s);
      case 22: return launch_apply_reg<22>(dop, wts, out, C, K, R, ldr, T, B, S, s);
      case 24: return launch_apply_reg<24>(dop, wts, out, C, K, R, ldr, T, B, S, s);
      default: break;
    }
  }
  // cells per lane: the tile size (128, 64 or 32 cells) that pads the block
  // least, and where a tile is one or two chunks deep, i.e. nothing hides its
  // loads but other CTAs, the smaller tiles of which more fit an SM
  // (D = 15, K128 R3000 B100 S11: 38.7 us with 64-cell tiles, 41.9 with 128)
  // Up to 8 steering vectors are one warp per CTA: 32-cell tiles, whose 11 KB let 21
  // of them share an SM (D = 36, K64 R8192 B256 S4: 57 us, with 128-cell tiles
  // 74; D = 128 B256 S8: 0.7 of the time)
  if (S <= 8) return launch_apply_tile<1>(dop, wts, out, C, K, R, ldr, T, B, S, s);
  auto padded = [&](int cells) { return (B + 32 * cells - 1) / (32 * cells) * cells; };
  if (D > 2 * DC && padded(4) <= padded(2) && padded(4) <= padded(1))
    return launch_apply_tile<4>(dop, wts, out, C, K, R, ldr, T, B, S, s);
  if (padded(2) <= padded(1)) return launch_apply_tile<2>(dop, wts, out, C, K, R, ldr, T, B, S, s);
  return launch_apply_tile<1>(dop, wts, out, C, K, R, ldr, T, B, S, s);
}

}  // namespace stap

namespace stap {
cudaError_t check_record_apply(CheckRecord* out) { return read_check_record(out); }
}  // namespace stap
