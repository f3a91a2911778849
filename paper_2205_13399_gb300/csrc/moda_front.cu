// Reading an archive's front (Sec. 3.3 "return all non-dominated solutions
// from archive A"): each replica's own non-dominated members, found and
// packed on the device, so that the host merges a few thousand points instead
// of copying and sorting every archive; and the states of chosen members,
// gathered into one buffer.
//
// The filter compares every pair of a replica's members (400 of them on the
// n = 75 workload: 160,000 comparisons a block, a few microseconds); a member
// goes if another dominates it, or equals it in a lower slot, neither of
// which can keep it in the union's front.
#include <cstdint>

#include "moda_internal.h"

namespace moda {
namespace {

// Threads of a block: few enough to fit beside the annealing blocks (n = 75, one
// an SM: a read beside such a run took 89 ms with 256, 0.5 with 128; alone 0.47
// and 0.56).
constexpr int kFrontTile = 128;

__global__ void __launch_bounds__(kFrontTile) front_kernel(const int32_t *counts, const int64_t *E,
                                                           int s, int ns, int j, int first,
                                                           FrontPoint *out, uint32_t *total) {
  __shared__ longlong2 tile[kFrontTile];
  const int q = first + blockIdx.x;
  const size_t row = (size_t)q * ns + j;
  const int cnt = counts[row] < s ? counts[row] : s;
  const longlong2 *e = reinterpret_cast<const longlong2 *>(E) + row * s;
  for (int base = 0; base < cnt; base += kFrontTile) {
    const int y = base + threadIdx.x;
    const longlong2 me = e[y < cnt ? y : 0];
    bool keep = y < cnt;
    for (int t0 = 0; t0 < cnt; t0 += kFrontTile) {
      __syncthreads();
      if (t0 + (int)threadIdx.x < cnt) tile[threadIdx.x] = e[t0 + threadIdx.x];
      __syncthreads();
      const int tn = cnt - t0 < kFrontTile ? cnt - t0 : kFrontTile;
      for (int k = 0; k < tn; ++k) {
        const longlong2 o = tile[k];
        if (o.x <= me.x && o.y <= me.y && (o.x != me.x || o.y != me.y || t0 + k < y)) keep = false;
      }
    }
    if (keep) {
      FrontPoint p;
      p.e1 = me.x;
      p.e2 = me.y;
      p.rep = q;
      p.slot = y;
      out[atomicAdd(total, 1u)] = p;  // the host sorts them
    }
  }
}

__global__ void gather_kernel(const uint32_t *bits, const FrontPoint *pts, int n, int s, int ns,
                              int j, int W, uint32_t *out) {
  const int k = blockIdx.x;
  if (k >= n) return;
  const uint32_t *src = bits + (((size_t)pts[k].rep * ns + j) * s + pts[k].slot) * W;
  for (int w = threadIdx.x; w < W; w += blockDim.x) out[(size_t)k * W + w] = src[w];
}

}  // namespace

cudaError_t launch_front(const int32_t *counts, const int64_t *E, int s, int ns, int j, int first,
                         int rows, FrontPoint *out, uint32_t *total, cudaStream_t stream) {
  front_kernel<<<rows, kFrontTile, 0, stream>>>(counts, E, s, ns, j, first, out, total);
  return cudaGetLastError();
}

cudaError_t launch_gather(const uint32_t *bits, const FrontPoint *pts, int n, int s, int ns, int j,
                          int W, uint32_t *out, cudaStream_t stream) {
  gather_kernel<<<n, 128, 0, stream>>>(bits, pts, n, s, ns, j, W, out);
  return cudaGetLastError();
}

}  // namespace moda
