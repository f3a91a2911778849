// Register annealer, strict acceptance, Delta E within int32 (see
// moda_reg_body.cuh), and the choice and launch of every variant.
#include <algorithm>

#include "moda_reg_body.cuh"

namespace moda {

const void *reg_kernel_strict(int K, bool narrow) {
  if (!narrow) return reg_kernel_strict_wide(K);
  return K == 1    ? reinterpret_cast<const void *>(reg_anneal_kernel<1, false, false, false, false>)
         : K == 2  ? reinterpret_cast<const void *>(reg_anneal_kernel<2, false, false, false, false>)
         : K == 4  ? reinterpret_cast<const void *>(reg_anneal_kernel<4, false, false, true, false>)
         : K == 8  ? reinterpret_cast<const void *>(reg_anneal_kernel<8, false, false, true, false>)
         : K == 16 ? reinterpret_cast<const void *>(reg_anneal_kernel<16, false, false, true, false>)
         : K == 24 ? reinterpret_cast<const void *>(reg_anneal_kernel<24, false, false, true, false>)
                   : nullptr;
}

cudaError_t reg_function(int K, bool narrow, bool lenient, bool ext, int optin,
                         const void **func) {
  const void *f = ext       ? reg_kernel_ext(K)
                  : lenient ? reg_kernel_lenient(K, narrow)
                            : reg_kernel_strict(K, narrow);
  if (f == nullptr) return cudaErrorInvalidValue;
  // the device's limit, always: launches of one kernel with other sizes may
  // be under way in a graph or on another thread
  cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  if (e == cudaSuccess) *func = f;
  return e;
}

// Uncrowded, measured on n = 8: 4.2 ms with one word, 4.8 with two; n = 25
// (128 replicas): 14.4, 13.7 and 14.6 ms with one, two and four; n = 33: four
// and two alike, eight a fifth slower; n = 75: 67 ms with eight, 113 with 16.
// Crowded: n = 20 97 ms with four, 138 with eight; n = 40 131 and 165; n = 60
// 235 with eight, 293 with 16 (72 registers spill there).
int reg_words(int W, bool draws, bool crowded) {
  if (!crowded) {
    if (draws && W <= 8) return 1;
    if (draws && W <= 40) return 2;
    if (W <= 88) return 4;
    if (W <= 176) return 8;
  }
  return W <= 56 ? 4 : W <= 176 ? 8 : W <= 16 * kRegMaxWorkers ? 16 : 24;
}

// Rebuilds: planes of Fs where no slot has to go for them, then matrix
// products from the rows, then neither.  Products from n = 29 up: n = 20 (3,000
// replicas) 81 ms without and 104 with them, n = 25 13.6 and 13.8, n = 33 28.7
// and 27.8, n = 50 59.1 and 48.6, n = 75 88.1 and 60.2.
constexpr int kRegMma = 29;

// Warps that the registers of a kernel of K words allow in one block: each
// quarter of an SM holds whole warps only (K = 24: 5 of 96 registers).
static int reg_most_warps(int K) { return 4 * (16384 / (32 * reg_regs(K))); }

RegFit reg_fit(int n, int64_t fmax, int64_t dmax, int s, bool narrow, bool ext, int optin) {
  const int m = n * n, W = (m + 31) / 32;
  const bool wide = !narrow || ext, draws = narrow || ext;
  RegFit f{kRegSlots, 2};
  if (fmax > 65535 || dmax > 65535) return RegFit{};
  for (const bool crowded : {false, true}) {
    const int K = reg_words(W, draws, crowded), workers = (W + K - 1) / K;
    if (workers > kRegMaxWorkers || workers + 2 > reg_most_warps(K)) return RegFit{};
    RegFit g;
    for (int mma = 2 * dmax <= 65535 && n >= kRegMma ? 2 : 0; mma >= 0 && g.se == 0; --mma)
      for (int se = std::min(s, kRegSlots); se >= 1 && g.se == 0; se = se > 64 ? se / 2 : se / 8) {
        if (mma == 2 && se < std::min(s, kRegSlots)) break;
        if ((int64_t)reg_smem(n, m, se, workers, K, wide, K >= 4, mma,
                              reg_split_flows(fmax, dmax, n))
                         .total <= optin)
          g = RegFit{se, mma};
      }
    f.se = std::min(f.se, g.se);
    f.mma = std::min(f.mma, g.mma);
  }
  return f;
}

int32_t reg_hm_limit(int64_t b1, int64_t b2, int64_t w1, int64_t w2) {
  int64_t lim = 1 << 20;
  const int64_t b[2] = {b1, b2}, w[2] = {w1, w2};
  for (int k = 0; k < 2; ++k)
    if (w[k] > 0) lim = std::min<int64_t>(lim, (INT64_C(2147483646) - b[k]) / w[k] - 8);
  return (int32_t)std::max<int64_t>(lim, -1);
}

cudaError_t reg_choose(WarpRun *runs, int count, int64_t items, bool ext, int sms, int optin,
                       RegChoice *out) {
  *out = RegChoice{};
  int W = 1;
  for (int k = 0; k < count; ++k) W = std::max(W, runs[k].W);
  const bool narrow = runs[0].narrow != 0, wide = !narrow || ext, draws = narrow || ext;
  const int crowded = reg_words(W, draws, true);
  for (int K = reg_words(W, draws, false); K <= 24; K = K < 8 ? 2 * K : K + 8) {
    const int g = (W + K - 1) / K, d = K < 4 ? std::min((W + 3) / 4, 6) : 0;
    const bool inl = K >= 4;
    auto need_of = [&](int most) {
      size_t need = 0;
      for (int k = 0; k < count; ++k)
        need = std::max<size_t>(need, reg_smem(runs[k].n, runs[k].m, runs[k].se, g, K, wide, inl,
                                               std::min(runs[k].mma, most), runs[k].fbig != 0)
                                          .total);
      return need;
    };
    size_t need = need_of(2);
    if (g > kRegMaxWorkers || need_of(1) > (size_t)optin) continue;
    const void *func = nullptr;
    cudaError_t e = reg_function(K, narrow, runs[0].accept != 0, ext, optin, &func);
    if (e != cudaSuccess) return e;
    int blocks = 0, lean = 0;
    if (need <= (size_t)optin) e = reg_occupancy(func, g + d + 2, need, &blocks);
    if (e == cudaSuccess) e = reg_occupancy(func, g + d + 2, need_of(1), &lean);
    if (e != cudaSuccess) return e;
    if (lean > blocks && (int64_t)blocks * sms < items) {
      for (int k = 0; k < count; ++k) runs[k].mma = std::min(runs[k].mma, 1);
      need = need_of(1);
      blocks = lean;
    }
    if (blocks >= 1 && ((int64_t)blocks * sms >= items || K >= crowded)) {
      *out = RegChoice{K, g, d, need, func};
      return cudaSuccess;
    }
  }
  return cudaSuccess;
}

cudaError_t reg_occupancy(const void *func, int warps, size_t smem, int *blocks) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, func, 32 * warps, smem);
}

cudaError_t launch_reg(const RegLaunch &L, const void *func, int grid, size_t smem,
                       cudaStream_t stream) {
  void *args[1] = {const_cast<RegLaunch *>(&L)};
  cudaError_t e =
      cudaLaunchKernel(func, dim3((unsigned)grid),
                       dim3((unsigned)(32 * (L.workers + L.draws + 2))), args, smem, stream);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace moda
