// Training with guard cells (an option beyond the paper's own-block training,
// which leaves the cell under test in its training data): the covariance that
// block b's weights use is the mean of the covariances of the adjacent blocks
// b-1 and b+1, or the one of them that exists at either end of the range, so
// that the cell under test and the other cells of its own block act as guard
// cells.  With equal block sizes the mean of two sample covariances is the
// sample covariance of their 2B cells.
//
// Reads two c128 matrices and writes one per system (in 16-byte elements,
// coalesced along a matrix row); the halving is exact.  The FP64 pipe (a warp
// instruction holds it 16 cycles) and not memory bounds both kernels, so inside
// a run, whose solve reads nothing else, they take the lower triangles only,
// and the window's mean divides by a power of two -- most groups' count for
// half = 1, 2, 4 -- as an exact product.
//
// The sliding window below generalises it: a guard band of `guard` groups on
// each side of the group under test and `half` training groups beyond it on
// each side (guard 0, half 1 is the neighbour-block form).
#include "batch.cuh"
#include "checked.cuh"
#include "stap_internal.cuh"

namespace stap {
namespace {

// Entry n of the launch: the system and the entry's place in its matrix, over
// all D^2 entries or (lower) those of the lower triangle, row by row.
__device__ __forceinline__ void entry_of(long long n, int D, int lower, long long& sys, long long& e) {
  const long long per = lower ? (long long)D * (D + 1) / 2 : (long long)D * D;
  sys = n / per;
  e = n - sys * per;
  if (lower) {
    const int q = (int)e;
    int i = (int)((sqrtf(8.0f * (float)q + 1.0f) - 1.0f) * 0.5f);
    while (i * (i + 1) / 2 > q) --i;
    while ((i + 1) * (i + 2) / 2 <= q) ++i;
    e = (long long)i * D + (q - i * (i + 1) / 2);
  }
}

__global__ void __launch_bounds__(256)
train_neighbours_kernel(const double2* __restrict__ in, double2* __restrict__ out, int NB, int D,
                        int lower, long long count, long long total) {
  const long long DD = (long long)D * D;
  for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < count;
       n += (long long)gridDim.x * blockDim.x) {
    long long sys, e;
    entry_of(n, D, lower, sys, e);
    const long long idx = sys * DD + e;
    const int b = (int)(sys % NB);
    const bool lo = b > 0, hi = b + 1 < NB;
    double2 v;
    if (lo && hi && in_bounds(idx - DD, total, kSiteTrain) && in_bounds(idx + DD, total, kSiteTrain)) {
      const double2 p = __ldg(in + idx - DD), q = __ldg(in + idx + DD);
      v = make_double2((p.x + q.x) * 0.5, (p.y + q.y) * 0.5);
    } else {
      const long long src = idx + (lo ? -DD : DD);
      v = in_bounds(src, total, kSiteTrain) ? __ldg(in + src) : make_double2(0.0, 0.0);
    }
    out[idx] = v;
  }
}

// Sliding training window: group j (B cells) takes the mean of the
// covariances of the groups j-guard-half .. j-guard-1 and j+guard+1 ..
// j+guard+half that exist, summed left side first in increasing group order
// and then divided component by component by their count -- the same
// operations in the same order as the definition, so the result is exact to
// the last bit.  One thread per (k, j, entry), entries fastest (coalesced);
// neighbouring groups read overlapping windows, which the L2 serves.
// Measured: D 15, K 128, 30 groups, guard 1, half 2: 62.3 -> 26.6 us inside a run.
__global__ void __launch_bounds__(256)
train_window_kernel(const double2* __restrict__ in, double2* __restrict__ out, int NB, int D, int lower,
                    long long n_entries, long long total, int guard, int half) {
  const long long DD = (long long)D * D;
  for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < n_entries;
       n += (long long)gridDim.x * blockDim.x) {
    long long sys, e;
    entry_of(n, D, lower, sys, e);
    const int j = (int)(sys % NB);
    const long long idx = sys * DD + e;
    const double2* base = in + (sys - j) * DD + e;   // group 0 of this bin, entry e
    double re = 0.0, im = 0.0;
    int count = 0;
    for (int side = 0; side < 2; ++side) {
      const int i0 = side == 0 ? j - guard - half : j + guard + 1;
      for (int m = 0; m < half; ++m) {
        const int i = i0 + m;
        if (i < 0 || i >= NB) continue;
        const double2 v = in_bounds((sys - j + i) * DD + e, total, kSiteTrain) ? __ldg(base + (long long)i * DD)
                                                                               : make_double2(0.0, 0.0);
        re += v.x;
        im += v.y;
        ++count;
      }
    }
    if ((count & (count - 1)) == 0) {              // 1 / count is exact
      const double r = __hiloint2double((1023 - (31 - __clz(count))) << 20, 0);
      out[idx] = make_double2(re * r, im * r);
    } else {
      out[idx] = make_double2(re / (double)count, im / (double)count);
    }
  }
}

}  // namespace

namespace {
long long train_entries(int K, int NB, int D, bool lower) {
  return (long long)K * NB * (lower ? (long long)D * (D + 1) / 2 : (long long)D * D);
}
unsigned train_blocks(long long entries) {
  const long long blocks = (entries + 255) / 256;
  return (unsigned)(blocks > 152LL * 16 ? 152LL * 16 : blocks);
}
}  // namespace

cudaError_t launch_train_window(const double2* in, double2* out, int K, int NB, int D, int guard,
                                int half, cudaStream_t s, bool lower_only) {
  if (guard < 0 || half < 1 || NB < 2 * guard + 2) return cudaErrorInvalidValue;
  const long long total = (long long)K * NB * D * D, n = train_entries(K, NB, D, lower_only);
  return launch_or_defer(s, [=](cudaStream_t st) {
    train_window_kernel<<<train_blocks(n), 256, 0, st>>>(in, out, NB, D, lower_only ? 1 : 0, n, total, guard, half);
    return cudaGetLastError();
  });
}

cudaError_t launch_train_neighbours(const double2* in, double2* out, int K, int NB, int D,
                                    cudaStream_t s, bool lower_only) {
  if (NB < 2) return cudaErrorInvalidValue;
  const long long total = (long long)K * NB * D * D, n = train_entries(K, NB, D, lower_only);
  return launch_or_defer(s, [=](cudaStream_t st) {
    train_neighbours_kernel<<<train_blocks(n), 256, 0, st>>>(in, out, NB, D, lower_only ? 1 : 0, n, total);
    return cudaGetLastError();
  });
}

}  // namespace stap

namespace stap {
cudaError_t check_record_train(CheckRecord* out) { return read_check_record(out); }
}  // namespace stap
