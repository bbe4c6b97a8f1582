// Reduced-DOF front end (beyond the paper, whose cubes have 1000 channels):
// the N element channels of an element cube x[N][P][R] are combined into the
// C channels of the STAP cube by a matrix W[C][N],
//   y[c][p][r] = sum_{n<N} conj(W[c][n]) x[n][p][r],
// one chunk of Nc elements at a time (the first chunk writes y, later chunks
// add to it).
//
// HBM-bound: every element sample is read once per pass of CB = 4 output
// channels (one pass for C <= 4), y is read and written once per chunk.  A
// thread owns VEC adjacent (pulse, range) positions, two where the rows stay
// 16-byte aligned, so a warp reads 64 consecutive complex samples of one
// element row.  W's four channels lie side by side in shared memory, kW
// elements at a time: two broadcast 16-byte reads serve 2 VEC x 16 FMAs.  (With
// one position per thread and W through L1, five load instructions per sample
// held the load/store unit: N 1000 P 100 R 3000 to C 4, 2.4 GB, 633 us, 3.8
// TB/s; now 380 us, 6.3 TB/s.)  64 registers, four CTAs per SM.  Rounding: the
// elements of a chunk are summed in blocks of kBlk into a partial sum that is
// then added to the thread's total, which bounds the FP32 error growth by about
// (kBlk + Nc / kBlk) u instead of Nc u.
#include "stap_internal.cuh"

namespace stap {
namespace {

constexpr int kBlk = 32;
constexpr int kCB = 4;
constexpr int kThreads = 256;
constexpr int kW = 512;        // elements of W in shared memory at a time, a multiple of kBlk

template <int VEC>
__global__ void __launch_bounds__(kThreads, 4)
reduce_channels_kernel(const float2* __restrict__ x, const float2* __restrict__ W,
                       float2* __restrict__ y, int N, int n0, int Nc, int C, long long PR,
                       int accumulate) {
  __shared__ float4 sw[kW][kCB / 2];   // channels c0 .. c0 + 3 of an element (zero past C)
  const long long q = VEC * ((long long)blockIdx.x * kThreads + threadIdx.x);   // (p, r)
  const int c0 = blockIdx.y * kCB;
  const bool mine = q < PR;            // every thread keeps the barriers
  const float2* xq = x + (mine ? q : 0);
  float2 tot[kCB][VEC];
#pragma unroll
  for (int j = 0; j < kCB; ++j)
#pragma unroll
    for (int v = 0; v < VEC; ++v) tot[j][v] = make_float2(0.f, 0.f);
  for (int w0 = 0; w0 < Nc; w0 += kW) {
    const int wn = min(kW, Nc - w0);
    __syncthreads();
    for (int e = threadIdx.x; e < wn * kCB; e += kThreads) {
      const int j = e / wn, n = e - j * wn;
      reinterpret_cast<float2*>(sw[n])[j] =
          c0 + j < C ? __ldg(W + (size_t)(c0 + j) * N + n0 + w0 + n) : make_float2(0.f, 0.f);
    }
    __syncthreads();
    for (int b0 = 0; b0 < wn; b0 += kBlk) {
      const int b1 = min(wn, b0 + kBlk);
      float2 part[kCB][VEC];
#pragma unroll
      for (int j = 0; j < kCB; ++j)
#pragma unroll
        for (int v = 0; v < VEC; ++v) part[j][v] = make_float2(0.f, 0.f);
#pragma unroll (8 / VEC)
      for (int n = b0; n < b1; ++n) {
        float2 s[VEC];
        const float2* src = xq + (size_t)(w0 + n) * PR;
        if constexpr (VEC == 2) {
          const float4 v = __ldg(reinterpret_cast<const float4*>(src));
          s[0] = make_float2(v.x, v.y);
          s[VEC - 1] = make_float2(v.z, v.w);
        } else {
          s[0] = __ldg(src);
        }
#pragma unroll
        for (int h = 0; h < kCB / 2; ++h) {
          const float4 w = sw[n][h];
#pragma unroll
          for (int v = 0; v < VEC; ++v) {
            // conj(w) s = (wr sr + wi si) + i (wr si - wi sr)
            float2 &p = part[2 * h][v], &r = part[2 * h + 1][v];
            p.x = fmaf(w.x, s[v].x, p.x);
            p.x = fmaf(w.y, s[v].y, p.x);
            p.y = fmaf(w.x, s[v].y, p.y);
            p.y = fmaf(-w.y, s[v].x, p.y);
            r.x = fmaf(w.z, s[v].x, r.x);
            r.x = fmaf(w.w, s[v].y, r.x);
            r.y = fmaf(w.z, s[v].y, r.y);
            r.y = fmaf(-w.w, s[v].x, r.y);
          }
        }
      }
#pragma unroll
      for (int j = 0; j < kCB; ++j)
#pragma unroll
        for (int v = 0; v < VEC; ++v) {
          tot[j][v].x += part[j][v].x;
          tot[j][v].y += part[j][v].y;
        }
    }
  }
  if (!mine) return;
#pragma unroll
  for (int j = 0; j < kCB; ++j) {
    if (c0 + j >= C) break;
    float2* dst = y + (size_t)(c0 + j) * PR + q;
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
      float2 o = tot[j][v];
      if (accumulate) {
        const float2 a = dst[v];
        o.x = a.x + o.x;
        o.y = a.y + o.y;
      }
      dst[v] = o;
    }
  }
}

// The same sums for cubes of few positions: a CTA takes 32 of them and its
// eight warps eight blocks of kBlk elements at once; the block sums are then
// added to the total in the blocks' order, so the bits are the same.
__global__ void __launch_bounds__(kThreads)
reduce_channels_split_kernel(const float2* __restrict__ x, const float2* __restrict__ W,
                             float2* __restrict__ y, int N, int n0, int Nc, int C, long long PR,
                             int accumulate) {
  constexpr int NW = kThreads / 32;
  __shared__ float2 sp[NW][kCB][32];   // block sums of a round
  __shared__ float4 sw[NW * kBlk][kCB / 2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long q = 32LL * blockIdx.x + lane;
  const int c0 = blockIdx.y * kCB;
  const bool mine = q < PR;            // every thread keeps the barriers
  const float2* xq = x + (mine ? q : 0);
  float2 tot = make_float2(0.f, 0.f);  // channel c0 + warp, warps 0 .. 3
  for (int w0 = 0; w0 < Nc; w0 += NW * kBlk) {
    const int wn = min(NW * kBlk, Nc - w0);
    for (int e = threadIdx.x; e < wn * kCB; e += kThreads) {
      const int j = e / wn, n = e - j * wn;
      reinterpret_cast<float2*>(sw[n])[j] =
          c0 + j < C ? __ldg(W + (size_t)(c0 + j) * N + n0 + w0 + n) : make_float2(0.f, 0.f);
    }
    __syncthreads();
    const int b0 = warp * kBlk, b1 = min(wn, b0 + kBlk);
    float2 part[kCB];
#pragma unroll
    for (int j = 0; j < kCB; ++j) part[j] = make_float2(0.f, 0.f);
#pragma unroll 8
    for (int n = b0; n < b1; ++n) {
      const float2 v = __ldg(xq + (size_t)(w0 + n) * PR);
#pragma unroll
      for (int h = 0; h < kCB / 2; ++h) {
        const float4 w = sw[n][h];
        float2 &p = part[2 * h], &r = part[2 * h + 1];
        p.x = fmaf(w.x, v.x, p.x);
        p.x = fmaf(w.y, v.y, p.x);
        p.y = fmaf(w.x, v.y, p.y);
        p.y = fmaf(-w.y, v.x, p.y);
        r.x = fmaf(w.z, v.x, r.x);
        r.x = fmaf(w.w, v.y, r.x);
        r.y = fmaf(w.z, v.y, r.y);
        r.y = fmaf(-w.w, v.x, r.y);
      }
    }
#pragma unroll
    for (int j = 0; j < kCB; ++j) sp[warp][j][lane] = part[j];
    __syncthreads();
    if (warp < kCB)
      for (int b = 0; b < NW && w0 + b * kBlk < Nc; ++b) {
        tot.x += sp[b][warp][lane].x;
        tot.y += sp[b][warp][lane].y;
      }
    __syncthreads();
  }
  if (warp < kCB && c0 + warp < C && mine) {
    float2* dst = y + (size_t)(c0 + warp) * PR + q;
    if (accumulate) {
      const float2 a = *dst;
      tot.x = a.x + tot.x;
      tot.y = a.y + tot.y;
    }
    *dst = tot;
  }
}

}  // namespace

cudaError_t launch_reduce_channels(const float2* x_chunk, const float2* W, float2* y, int N, int n0,
                                   int Nc, int C, int P, int R, bool accumulate, cudaStream_t s) {
  if (N < 1 || C < 1 || Nc < 1 || n0 < 0 || n0 + Nc > N) return cudaErrorInvalidValue;
  const long long PR = (long long)P * R;
  const int cblocks = (C + kCB - 1) / kCB;
  // positions per thread by the CTAs that makes: two where three CTAs per SM
  // come of it, one, or (few positions: nothing else would hide the loads) the
  // split form.  N 1000, C 4, before and now: 300000 positions 638 -> 380 us (two),
  // 150000 334 -> 189 (one; the split form as long as 240 at half of that),
  // 77000 314 -> 127 (one), 32768 312 -> 87 and 8192 116 -> 24 (split).
  auto ctas = [&](int per) { return (PR + per - 1) / per * cblocks; };
  const bool two = PR % 2 == 0 && (reinterpret_cast<uintptr_t>(x_chunk) & 15) == 0 &&
                   ctas(2 * kThreads) >= 3 * 152;
  const bool one = two || ctas(kThreads) >= 3 * 152 / 2;
  const long long per = two ? 2 * kThreads : (one ? kThreads : 32);
  const long long blocks = (PR + per - 1) / per;
  if (blocks > 0x7fffffffLL || cblocks > 65535) return cudaErrorInvalidValue;
  dim3 grid((unsigned)blocks, (unsigned)cblocks);
  if (two)
    reduce_channels_kernel<2><<<grid, kThreads, 0, s>>>(x_chunk, W, y, N, n0, Nc, C, PR, accumulate ? 1 : 0);
  else if (one)
    reduce_channels_kernel<1><<<grid, kThreads, 0, s>>>(x_chunk, W, y, N, n0, Nc, C, PR, accumulate ? 1 : 0);
  else
    reduce_channels_split_kernel<<<grid, kThreads, 0, s>>>(x_chunk, W, y, N, n0, Nc, C, PR, accumulate ? 1 : 0);
  return cudaGetLastError();
}

}  // namespace stap
