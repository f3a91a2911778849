// Multi-objective Digital Annealer (Alg. 3 of arXiv 2205.13399) on K
// objectives given as explicit QUBO matrices: the generalisation of the
// bi-objective QAP path from outer-product fields to a stored P (Eq. cale),
// for QUBOs without QAP structure and for more than two objectives.
//
// One thread block per replica, laid out as the register annealer
// (moda_reg_body.cuh) is: G worker warps own N state words each (lane l has
// bit 32 w + l of word w) and keep Delta E of every objective in registers, a
// scan warp keeps the archive (all of its energies, record numbers and least
// penalties in shared memory) and runs the jumps, up to three helpers share
// its search for the first dominated member (with three objectives few
// members are dominated and archives fill: one warp took 2,400 cycles for
// 1,024 members, the workers' round 1,500), a store warp keeps the state
// words, writes members' states and fills the ring of schedule entries
// and draws.  A flip of bit p changes every other Delta E_j(q) by
// (1 - 2 x_q) s P_j[p][q] (s = +1 when p turns on): one coalesced read of row
// p of each P_j, from L2, which is what bounds a flip (m = 1,024, K = 3: 12 KB
// a flip and its latency).  Barriers of iteration t: A(t), the whole block,
// after the trial's counts; B(t), the workers, after the flipped bit was
// published.
//
// A jump to a member whose least penalty is above hi_t accepts nothing in
// the next iteration, so the scan warp settles it by one compare, 32
// iterations at a time.  For the members that may accept, Delta E comes back
// from a record in global memory: the workers write the state's record after
// every flip, into a buffer whose number the scan warp assigned ahead (the
// slot is known only an iteration later), and slots carry record numbers;
// without records Delta E is rebuilt from the state words.
#include <algorithm>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "moda_device.cuh"
#include "moda_host.h"
#include "moda_internal.h"

namespace moda {
namespace {

constexpr int kMaxK = 3;
constexpr int kMaxQBits = 4096;
constexpr int kQRing = 128;
constexpr int kQPad = 256;  // entries after the matrices: workers read whole words past the last row
constexpr int kQSpare = 4;  // records beyond one per slot: flips in flight

enum : uint32_t { kQEnd = 0, kQLoad = 1, kQStay = 2, kQStayEnd = 3 };

// Ring entry of one iteration (as the register annealer's).
struct QRing {
  double delta;
  float cln, margin;
  uint32_t sel, hi;
  uint32_t pad[2];
};
static_assert(sizeof(QRing) == 32, "ring entry layout");

struct QFlip {
  int32_t ps, x;
  int64_t d[kMaxK];
};
static_assert(sizeof(QFlip) == 32, "flip record layout");

// Shared-memory carve-up (byte offsets, 16-byte aligned regions).
struct QLayout {
  size_t ring, cnt, min, flip, tgt, rec, jump, scan, x, sum, draw, aE, aM, aR, total;
};
__host__ __device__ inline QLayout qubo_layout(int K, int G, int W, int s, bool narrow) {
  QLayout L;
  size_t o = 0;
  L.ring = o; o = align_up(o + sizeof(QRing) * kQRing, 16);
  L.cnt = o;  o = align_up(o + 4 * 2 * 32, 16);
  L.min = o;  o = align_up(o + 4 * 2 * 32, 16);
  L.flip = o; o = align_up(o + sizeof(QFlip) * 4, 16);
  L.tgt = o;  o = align_up(o + 4 * 4, 16);
  L.rec = o;  o = align_up(o + 4 * 4, 16);
  L.jump = o; o = align_up(o + 4 * 4, 16);
  L.scan = o; o = align_up(o + 4 * 4, 16);
  L.x = o;    o = align_up(o + 4 * (size_t)((W + 3) / 4 * 4), 16);
  L.sum = o;  o = align_up(o + 8 * 32 * kMaxK, 16);
  L.draw = o; o = align_up(o + 512 * (size_t)G, 16);
  // slot s only takes stores
  L.aE = o;   o = align_up(o + (narrow ? 4 : 8) * (size_t)K * ((size_t)s + 1), 16);
  L.aM = o;   o = align_up(o + 4 * ((size_t)s + 1), 16);
  L.aR = o;   o = align_up(o + 2 * ((size_t)s + 1), 16);
  L.total = o;
  return L;
}

struct QArgs {
  int32_t m, W, s, nsched, workers, helpers;
  int64_t I_max, beta;
  uint32_t replica_base, seed_lo, seed_hi;
  int32_t accept, archive, escape;
  const int32_t *P;          // [K][m][m]: P_j = Q_j + Q_j^T, diagonal Q_pp; kQPad more
  const double *sch_delta;
  const int64_t *sch_lo, *sch_hi;
  const double *table;
  void *records;             // [R][s + kQSpare][K][m] Delta E, or nullptr
  int64_t *arch_E;           // [R][s][K]
  uint32_t *arch_bits;       // [R][s][W]
  int32_t *arch_count;       // [R]
  uint32_t *x_final;         // [R][W]
  int64_t *E_final;          // [R][K]
  int64_t *stats;            // [R][4]
  int64_t *trace;            // [R][I_max][K + 1] or nullptr
};

__device__ __forceinline__ int uni(int v) { return __shfl_sync(kFull, v, 0); }
__device__ __forceinline__ uint32_t uni(uint32_t v) { return __shfl_sync(kFull, v, 0); }

// NARROW: every |Delta E_j| and |E_j| < 2^30 (int32, penalties in uint32), else
// int64.
template <int K, int N, bool NARROW>
__global__ void __maxnreg__(N == 4 ? 80 : 96) qubo_kernel(const QArgs A) {
  using dE_t = typename std::conditional<NARROW, int32_t, int64_t>::type;
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, wid = uni((int)(threadIdx.x >> 5));
  const int G = A.workers, H = A.helpers, warps = G + H + 2, threads = 32 * warps;
  const int m = A.m, W = A.W, s = A.s;
  const size_t mm = (size_t)m * m;
  const int rb = blockIdx.x;
  const uint32_t rep = A.replica_base + (uint32_t)rb;
  const uint32_t k0 = A.seed_lo, k1 = A.seed_hi;
  const uint32_t I_max = (uint32_t)A.I_max, nsched = (uint32_t)A.nsched;
  const bool lenient = A.accept != 0, by_offset = A.escape != 0;
  const QLayout L = qubo_layout(K, G, W, s, NARROW);
  QRing *const ring = reinterpret_cast<QRing *>(smem + L.ring);
  int32_t *const sCnt = reinterpret_cast<int32_t *>(smem + L.cnt);    // [2][32]
  uint32_t *const sMin = reinterpret_cast<uint32_t *>(smem + L.min);  // [2][32]
  QFlip *const sFlip = reinterpret_cast<QFlip *>(smem + L.flip);      // [4]
  int32_t *const sTgt = reinterpret_cast<int32_t *>(smem + L.tgt);    // [4]
  int32_t *const sRec = reinterpret_cast<int32_t *>(smem + L.rec);    // [4] by flip number
  uint32_t *const sJ = reinterpret_cast<uint32_t *>(smem + L.jump);   // mode, t, slot, record
  uint32_t *const sX = reinterpret_cast<uint32_t *>(smem + L.x);
  int64_t *const sSum = reinterpret_cast<int64_t *>(smem + L.sum);    // [32][kMaxK]
  float *const sDraw = reinterpret_cast<float *>(smem + L.draw);      // [G][128]
  int32_t *const sScan = reinterpret_cast<int32_t *>(smem + L.scan);  // [1 + H] first dominated
  dE_t *const sAE = reinterpret_cast<dE_t *>(smem + L.aE);            // [K][s + 1]
  uint32_t *const sAM = reinterpret_cast<uint32_t *>(smem + L.aM);
  uint16_t *const sAR = reinterpret_cast<uint16_t *>(smem + L.aR);
  int64_t *const gE = A.arch_E + (size_t)rb * s * K;
  uint32_t *const gB = A.arch_bits + (size_t)rb * s * W;
  dE_t *const gR = A.records ? static_cast<dE_t *>(A.records) +
                                   (size_t)rb * (size_t)(s + kQSpare) * K * m
                             : nullptr;

  // initial state: bit p is bit p % 32 of word (p / 32) % 4 of the draw
  // (p / 128, 0, replica, init) -- Alg. 3 "a random binary solution"
  for (int w = threadIdx.x; w < W; w += threads) {
    uint32_t c[4] = {(uint32_t)w >> 2, 0u, rep, kTagInit};
    philox10(c, k0, k1);
    const uint32_t v = word_of(c, w & 3);
    sX[w] = w * 32 + 32 <= m ? v : (v & ((1u << (m - w * 32)) - 1u));
  }
  auto fill = [&](uint32_t first) {  // iterations first .. first + 31 (one warp)
    const uint32_t q = first + (uint32_t)lane;
    const uint32_t sn = sched_entry(q, nsched);
    QRing e;
    e.delta = A.sch_delta[sn];
    e.cln = accept_scale(e.delta);
    e.margin = accept_margin(e.delta);
    const int64_t hi = A.sch_hi[sn];
    e.hi = hi < 0xFFFFFFFFll ? (uint32_t)hi : 0xFFFFFFFFu;
    uint32_t c[4] = {0u, q, rep, kTagSelect};
    philox10(c, k0, k1);
    e.sel = c[0];
    e.pad[0] = e.pad[1] = 0u;
    ring[q % kQRing] = e;
  };
  uint32_t filled = 64;
  if (wid == warps - 1) {
    fill(1);
    fill(33);
  }

  // ---- the workers' bits
  dE_t dE[K][N];
  uint32_t xn = 0u;  // bit k: the lane's bit of word k
  const int w0 = wid < G ? wid * N : W;
  auto bit_of = [&](int k) { return 32 * (w0 + k) + lane; };
  // Delta E of the state in sX from scratch: with phi_j(q) = sum_{r in x}
  // P_j[r][q], Delta E_j(q) = P_j[q][q] + phi_j(q), or -phi_j(q) where x_q = 1;
  // energies: also E_j = sum_{q in x} (P_j[q][q] + phi_j(q)) / 2 per warp into
  // sSum, doubled.  Rows of P come from L2, one for each set bit, so a worker
  // reads those of kRows bits for all of its words at once.  (Word after word,
  // one row at a time: 361 ms for 16 replicas of m = 200 with two objectives
  // whose 6,000 iterations mostly rebuild, 45 like this; 600 of m = 700 with
  // three 3,023 and 550; 64 of m = 300 with three in 64 bits 677 and 136.)
  constexpr int kRows = K * N <= 8 ? 4 : K * N <= 16 ? 2 : 1;
  auto rebuild = [&](bool energies) {
    __syncthreads();  // sX is complete
    xn = 0u;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      if (w0 + k < W) xn |= ((sX[w0 + k] >> lane) & 1u) << k;
#pragma unroll
      for (int j = 0; j < K; ++j) dE[j][k] = 0;
    }
    const int32_t *own[K];  // the lane's first entry of row 0 (entries past m count for nobody)
#pragma unroll
    for (int j = 0; j < K; ++j) own[j] = A.P + j * mm + 32 * w0 + lane;
    for (int w = 0; wid < G && w < W; ++w) {
      uint32_t word = uni(sX[w]);
      while (word) {
        int32_t pv[kRows][K][N];
#pragma unroll
        for (int u = 0; u < kRows; ++u) {
          // (row 0 for nobody past the word's last bit: a mask and not a test,
          // which would keep the rows' loads apart)
          const int32_t some = word != 0u ? -1 : 0;
          const int at = (some ? 32 * w + __ffs(word) - 1 : 0) * m;
          word &= word - 1u;
#pragma unroll
          for (int j = 0; j < K; ++j)
#pragma unroll
            for (int k = 0; k < N; ++k) pv[u][j][k] = __ldg(own[j] + at + 32 * k) & some;
        }
#pragma unroll
        for (int u = 0; u < kRows; ++u)
#pragma unroll
          for (int k = 0; k < N; ++k)
#pragma unroll
            for (int j = 0; j < K; ++j) dE[j][k] += pv[u][j][k];
      }
    }
    int64_t part[K];
#pragma unroll
    for (int j = 0; j < K; ++j) part[j] = 0;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const int q = bit_of(k);
      const bool in = q < m, xq = (xn >> k) & 1u;
#pragma unroll
      for (int j = 0; j < K; ++j) {
        const int32_t d = in ? A.P[j * mm + (size_t)q * m + q] : 0;
        if (xq) part[j] += (int64_t)d + dE[j][k];
        // (past m: a value no trial accepts)
        dE[j][k] = !in ? (dE_t)0x3FFFFFFF : xq ? -dE[j][k] : d + dE[j][k];
      }
    }
    if (energies) {
#pragma unroll
      for (int j = 0; j < K; ++j) {
        int64_t v = part[j];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
        if (lane == 0) sSum[wid * kMaxK + j] = v;
      }
    }
    __syncthreads();
  };
  auto count_of = [&](uint32_t t) { return lane < G ? sCnt[32 * (int)(t & 1u) + lane] : 0; };

  __syncthreads();
  rebuild(true);

  if (wid < G) {
    // ================= workers =================
    uint32_t accb = 0u, amin = 0u;  // accepted bits: word k at bit N - 1 - k
    int cnt = 0;
    int64_t Eoff = 0;
    uint32_t nflip = 0;
    bool fresh = false;  // a flip's state whose record is not written yet
    auto penalty = [&](int k) -> int64_t {  // exact
      int64_t a = 0;
#pragma unroll
      for (int j = 0; j < K; ++j) {
        const int64_t e = (int64_t)dE[j][k] - Eoff;
        const int64_t v = e > 0 ? e : 0;
        if (j == 0) a = v;
        else a = lenient ? (v < a ? v : a) : a + v;
      }
      return a;
    };
    auto trial = [&](uint32_t t) {
      const QRing &r = ring[t % kQRing];
      const float margin = r.margin, cln = r.cln;
      const uint32_t hi = r.hi;
      const int32_t off = (int32_t)(Eoff < 0x3FFFFFFF ? Eoff : 0x3FFFFFFF);
      uint32_t a[N];
      float near = 3.0e38f;
      amin = 0xFFFFFFFFu;
      accb = 0u;
#pragma unroll
      for (int k = 0; k < N; ++k) {
        if (NARROW) {
          uint32_t v = 0u;
#pragma unroll
          for (int j = 0; j < K; ++j) {
            const uint32_t aj = (uint32_t)max((int32_t)dE[j][k] - off, 0);
            if (j == 0) v = aj;
            else v = lenient ? min(v, aj) : v + aj;
          }
          a[k] = v;
        } else {
          const int64_t v = penalty(k);
          a[k] = v >= 0xFFFFFFFFll ? 0xFFFFFFFFu : (uint32_t)v;
        }
        amin = min(amin, a[k]);
      }
      float *const mine = sDraw + 128 * wid;  // the chunk's levels by bit
#pragma unroll
      for (int kc = 0; kc < N; kc += 4) {
        const uint32_t mn = min(min(a[kc], a[kc + 1]), min(a[kc + 2], a[kc + 3]));
        if (w0 + kc < W && __any_sync(kFull, mn <= hi)) {
          const int g = 8 * (w0 + kc) + lane;
          uint32_t d[4] = {(uint32_t)g, t, rep, kTagAccept};
          philox10(d, k0, k1);
          float4 v;
          v.x = 4 * g < m ? accept_level(d[0], cln) : -3.0e38f;
          v.y = 4 * g + 1 < m ? accept_level(d[1], cln) : -3.0e38f;
          v.z = 4 * g + 2 < m ? accept_level(d[2], cln) : -3.0e38f;
          v.w = 4 * g + 3 < m ? accept_level(d[3], cln) : -3.0e38f;
          __syncwarp();  // the last chunk's levels have been read
          reinterpret_cast<float4 *>(mine)[lane] = v;
          __syncwarp();
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float af = NARROW ? __uint2float_rn(a[kc + q]) : penalty_f32(penalty(kc + q));
            const float diff = af - mine[32 * q + lane];
            near = fminf(near, fabsf(diff));
            accb = __funnelshift_l(__float_as_uint(diff), accb, 1);
          }
        } else {
          accb <<= 4;
        }
      }
      if (__any_sync(kFull, near <= margin)) {
        // within the error of the FP32 test: the IEEE double test of R7
        const double delta = r.delta;
        accb = 0u;
#pragma unroll 1
        for (int kk = 0; kk < N; ++kk) {
          int64_t av = 0;
#pragma unroll
          for (int k = 0; k < N; ++k)
            if (k == kk) av = penalty(k);
          const int p = bit_of(kk);
          uint32_t d[4] = {(uint32_t)(p >> 2), t, rep, kTagAccept};
          philox10(d, k0, k1);
          const bool ok =
              p < m && (double)av <= __dmul_rn(delta, __ldg(&A.table[word_of(d, p & 3) >> 16]));
          accb = accb << 1 | (ok ? 1u : 0u);
        }
      }
      cnt = __reduce_add_sync(kFull, __popc(accb));
      if (lane == 0) sCnt[32 * (int)(t & 1u) + wid] = cnt;
    };
    auto write_record = [&]() {  // the state after flip nflip
      dE_t *const to = gR + (size_t)uni(sRec[nflip & 3u]) * K * m;
#pragma unroll
      for (int k = 0; k < N; ++k) {
        const int q = bit_of(k);
        if (q < m) {
#pragma unroll
          for (int j = 0; j < K; ++j) to[(size_t)j * m + q] = dE[j][k];
        }
      }
    };
    uint32_t t = 1;
    while (t <= I_max) {
      trial(t);  // (its only place: the kernel's three roles share the instruction cache)
      const uint32_t sel = ring[t % kQRing].sel;
      __syncthreads();  // A(t)
      const uint32_t c = (uint32_t)count_of(t);
      const uint32_t mnw = __reduce_min_sync(kFull, amin);
      const uint32_t sums = __reduce_add_sync(kFull, lane < wid ? c | c << 16 : c);
      const int total = (int)(sums & 0xFFFFu), before = (int)(sums >> 16);
      if (lane == 0) sMin[32 * (int)(t & 1u) + wid] = mnw;
      if (total == 0 && by_offset) {  // Alg. 1: raise the offset
        Eoff += A.beta;
        if (t == I_max) {
          __syncthreads();
          __syncthreads();
          break;
        }
        ++t;
        continue;
      }
      if (total == 0) {
        if (fresh && gR != nullptr) write_record();
        fresh = false;
        __syncthreads();  // least penalties and the record are complete
        __syncthreads();  // the scan warp has settled the jumps
        const uint32_t mode = uni(sJ[0]);
        t = uni(sJ[1]);
        if (mode == kQEnd || mode == kQStayEnd) break;
        if (mode == kQLoad) {
          if (gR != nullptr) {
            // (the record, while the store warp fetches the member's state)
            const dE_t *from = gR + (size_t)uni((int)sJ[3]) * K * m;
#pragma unroll
            for (int k = 0; k < N; ++k) {
              const int q = bit_of(k);
#pragma unroll
              for (int j = 0; j < K; ++j)
                dE[j][k] = q < m ? from[(size_t)j * m + q] : (dE_t)0x3FFFFFFF;
            }
            __syncthreads();  // sX is complete
            xn = 0u;
#pragma unroll
            for (int k = 0; k < N; ++k)
              if (w0 + k < W) xn |= ((sX[w0 + k] >> lane) & 1u) << k;
          } else {
            rebuild(false);
          }
        }
        continue;
      }
      // ---- one accepted bit at random (R11): rank r in ascending bit
      // order; the lane that holds it publishes it
      const int r = uni(pick(sel, total)) - before;
      if (r >= 0 && r < cnt) {
        int kw = 0, rw = r;
        uint32_t bw = __ballot_sync(kFull, (accb >> (N - 1)) & 1u);
        int upto = __popc(bw);
#pragma unroll
        for (int k = 1; k < N; ++k) {
          const uint32_t b = __ballot_sync(kFull, (accb >> (N - 1 - k)) & 1u);
          if (r >= upto) {
            kw = k;
            bw = b;
            rw = r - upto;
          }
          upto += __popc(b);
        }
        const bool mine = ((bw >> lane) & 1u) && __popc(bw & ((1u << lane) - 1u)) == rw;
#pragma unroll
        for (int k = 0; k < N; ++k)
          if (kw == k && mine) {
            QFlip f;
            f.ps = bit_of(k);
            f.x = (int)((xn >> k) & 1u);
#pragma unroll
            for (int j = 0; j < kMaxK; ++j) f.d[j] = j < K ? (int64_t)dE[j < K ? j : 0][k] : 0;
            sFlip[t & 3u] = f;
          }
      }
      if (t == I_max) {
        __syncthreads();  // the scan and the store warp settle the last flip
        __syncthreads();
        break;
      }
      // the state's record, while the flip is being published
      if (fresh && gR != nullptr) write_record();
      if (G > 1) asm volatile("bar.sync 1, %0;" ::"r"(32 * G) : "memory");  // B(t)
      else __syncwarp();
      Eoff = 0;
      const int ps = uni(sFlip[t & 3u].ps), x = uni(sFlip[t & 3u].x);
      const int32_t *const prow = A.P + (size_t)ps * m;
      int32_t pv[K][N];
#pragma unroll
      for (int k = 0; k < N; ++k) {
        const int q = bit_of(k);
#pragma unroll
        for (int j = 0; j < K; ++j) pv[j][k] = q < m ? __ldg(&prow[j * mm + q]) : 0;
      }
      const uint32_t mw = (uint32_t)((ps >> 5) - w0);
      const uint32_t xs = x ? ~xn : xn;  // bit k set: this bit's change is negative
#pragma unroll
      for (int k = 0; k < N; ++k) {
        const dE_t g = (dE_t)1 - (dE_t)(2u * ((xs >> k) & 1u));
        if (mw == (uint32_t)k && lane == (ps & 31)) {  // the flipped bit: only its sign changes
#pragma unroll
          for (int j = 0; j < K; ++j) {
            pv[j][k] = 0;
            dE[j][k] = -dE[j][k];
          }
          xn ^= 1u << k;
        }
#pragma unroll
        for (int j = 0; j < K; ++j) dE[j][k] += g * (dE_t)pv[j][k];
      }
      ++nflip;
      fresh = true;
      ++t;
    }
    return;
  }

  if (wid == warps - 1) {
    // ================= store warp =================
    auto store = [&](uint32_t tp) {
      const int ps = uni(sFlip[tp & 3u].ps), target = uni(sTgt[tp & 3u]);
      if (lane == 0) sX[ps >> 5] ^= 1u << (ps & 31);
      __syncwarp();
      if (target >= 0)
        for (int q = lane; q < W; q += 32) gB[(size_t)target * W + q] = sX[q];
      __syncwarp();
    };
    auto refill = [&](uint32_t t) {  // the ring holds t .. t + 47 at least
      while (ring_short(filled, t)) {
        fill(filled + 1u);
        filled += 32u;
      }
    };
    uint32_t t = 1;
    bool p1 = false, p2 = false;  // flips of iterations t - 1, t - 2 not stored yet
    while (t <= I_max) {
      __syncthreads();  // A(t)
      const bool flip = __any_sync(kFull, count_of(t) > 0);
      if (p2) store(t - 2u);
      if (flip || by_offset) {
        p2 = p1;
        p1 = flip;
        if (t == I_max) {
          __syncthreads();
          if (p2) store(t - 1u);
          __syncthreads();
          if (p1) store(t);
          break;
        }
        refill(t + 2u);
        ++t;
        continue;
      }
      __syncthreads();
      if (p1) store(t - 1u);
      p1 = p2 = false;
      __syncthreads();
      const uint32_t mode = uni(sJ[0]);
      const int slot = uni((int)sJ[2]);
      filled = ring_skip(filled, t, uni(sJ[1]));
      t = uni(sJ[1]);
      if (mode == kQEnd || mode == kQLoad)  // the member the jumps ended on (written here)
        for (int q = lane; q < W; q += 32) sX[q] = gB[(size_t)slot * W + q];
      if (mode == kQEnd || mode == kQStayEnd) break;
      refill(t);
      if (mode == kQLoad) {
        if (gR != nullptr) __syncthreads();
        else rebuild(false);
      }
    }
    __syncwarp();
    for (int q = lane; q < W; q += 32) A.x_final[(size_t)rb * W + q] = sX[q];
    return;
  }

  // ================= scan warp (wid == G) and helpers =================
  const int part = wid - G;
  const bool lead = part == 0;
  int64_t E[K];
#pragma unroll
  for (int j = 0; j < K; ++j) {
    int64_t t2 = 0;
    for (int w = 0; w < G; ++w) t2 += sSum[w * kMaxK + j];
    E[j] = t2 / 2;
  }
  const bool exploit = A.archive != 0;
  int64_t *const trace = A.trace ? A.trace + (size_t)rb * (size_t)I_max * (K + 1) : nullptr;
  const int64_t hiF = A.sch_hi[nsched - 1];
  const uint32_t hiF32 = hiF < 0xFFFFFFFFll ? (uint32_t)hiF : 0xFFFFFFFFu;
  int acount = 0;
  uint32_t nflip = 0, njump = 0, nempty = 0, nraise = 0;
  // Records: numbers handed out in order, then those that were freed (at most
  // one a flip, and every flip takes one); flips nflip + 1 and nflip + 2 have
  // theirs.
  int rec_new = 0;
  uint32_t q_put = 0, q_get = 0;  // freed numbers, a queue of 8
  uint32_t q_lo = 0u, q_hi = 0u, q_lo2 = 0u, q_hi2 = 0u;
  auto q_push = [&](uint32_t v) {
    const uint32_t at = (q_put++ & 7u) * 16u, mask = 0xFFFFu << (at & 31u), x = v << (at & 31u);
    uint32_t &w = at < 32u ? q_lo : at < 64u ? q_hi : at < 96u ? q_lo2 : q_hi2;
    w = (w & ~mask) | x;
  };
  auto assign = [&](uint32_t f) {  // flip f's record
    uint32_t v;
    if (q_get != q_put) {
      const uint32_t at = (q_get++ & 7u) * 16u;
      const uint32_t w = at < 32u ? q_lo : at < 64u ? q_hi : at < 96u ? q_lo2 : q_hi2;
      v = (w >> (at & 31u)) & 0xFFFFu;
    } else {
      v = (uint32_t)rec_new++;
    }
    sRec[f & 3u] = (int)v;
  };
  assign(1u);
  assign(2u);
  auto state_min = [&](int par) {
    return __reduce_min_sync(kFull, lane < G ? sMin[32 * par + lane] : 0xFFFFFFFFu);
  };
  // x dominates slot y (all differences >= 0, some > 0); y >= s: the spare
  auto dom = [&](int y) {
    dE_t any = 0;
#pragma unroll
    for (int j = 0; j < K; ++j) any |= sAE[(size_t)j * (s + 1) + y] - (dE_t)E[j];
    return any > 0;
  };
  auto dominated = [&](int y) {
    dE_t any = 0;
#pragma unroll
    for (int j = 0; j < K; ++j) any |= (dE_t)E[j] - sAE[(size_t)j * (s + 1) + y];
    return any > 0;
  };
  // the first member x dominates among this warp's stretches of 128, or -1
  auto search = [&]() -> int {
    for (int base = 128 * part; base < acount; base += 128 * (H + 1)) {
      unsigned bal[4];
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        const int y = base + 32 * g + lane;
        bal[g] = __ballot_sync(kFull, y < acount && dom(y < s ? y : s));
      }
      if (bal[0] | bal[1] | bal[2] | bal[3]) {
        const unsigned b = bal[0] ? bal[0] : bal[1] ? bal[1] : bal[2] ? bal[2] : bal[3];
        return base + (bal[0] ? 0 : bal[1] ? 32 : bal[2] ? 64 : 96) + __ffs(b) - 1;
      }
    }
    return -1;
  };
  // Alg. 4's target for the energies E: the team's first dominated member,
  // else the next slot, else none (-1)
  auto explore_target = [&](bool &appended) -> int {
    int target = search();
    if (H > 0) {
      sScan[part] = target;
      asm volatile("bar.sync 2, %0;" ::"r"(32 * (H + 1)) : "memory");
      for (int h = 0; h <= H; ++h) {
        const int f = uni(sScan[h]);
        if (f >= 0 && (target < 0 || f < target)) target = f;
      }
      // (written again only after the next barrier A)
    }
    if (target < 0 && acount < s) {
      target = acount++;
      appended = true;
    }
    return target;
  };
  auto settle = [&](uint32_t tp) -> int {
    const QFlip &f = sFlip[tp & 3u];
#pragma unroll
    for (int j = 0; j < K; ++j) E[j] += f.d[j];
    ++nflip;
    int target = -1;
    bool appended = false;
    if (!exploit) {
      target = explore_target(appended);
    } else {  // Alg. 5
      int nb = 0;
      bool anyd = false;
      for (int base = 0; base < acount; base += 32) {
        const int y = base + lane;
        nb += __popc(__ballot_sync(kFull, y < acount && dom(y < s ? y : s)));
        anyd |= __any_sync(kFull, y < acount && dominated(y < s ? y : s)) != 0;
      }
      if (!anyd) {
        if (nb > 0) {
          uint32_t x[4] = {0u, tp, rep, kTagExploit};
          philox10(x, k0, k1);
          int want = uni(pick(x[0], nb));
          for (int base = 0; base < acount; base += 32) {
            const int y = base + lane;
            const unsigned bal = __ballot_sync(kFull, y < acount && dom(y < s ? y : s));
            const int cb = __popc(bal);
            if (want < cb) {
              target = base + nth_set_bit(bal, want);
              break;
            }
            want -= cb;
          }
        } else if (acount < s) {
          target = acount++;
          appended = true;
        }
      }
    }
    // the flip's record goes to its slot; the one it had, or the flip's if no
    // slot took it, is free again
    const uint32_t mine = (uint32_t)sRec[nflip & 3u];
    if (!appended) q_push(target >= 0 ? (uint32_t)sAR[target] : mine);
    __syncwarp();
    sAR[target >= 0 ? target : s] = (uint16_t)mine;
    assign(nflip + 2u);
    sTgt[tp & 3u] = target;
#pragma unroll
    for (int j = 0; j < K; ++j) sAE[(size_t)j * (s + 1) + (target >= 0 ? target : s)] = (dE_t)E[j];
    if (trace != nullptr && lane == 0) {
      int64_t *tr = trace + (size_t)(tp - 1) * (K + 1);
#pragma unroll
      for (int j = 0; j < K; ++j) tr[j] = E[j];
      tr[K] = (int64_t)f.ps;
    }
    __syncwarp();
    return target;
  };
  auto idle_row = [&](uint32_t t) {  // trace row of an iteration without flip or jump
    if (trace != nullptr && lane == 0) {
      int64_t *tr = trace + (size_t)(t - 1) * (K + 1);
#pragma unroll
      for (int j = 0; j < K; ++j) tr[j] = E[j];
      tr[K] = INT64_MIN;
    }
  };

  uint32_t t = 1;
  bool pend = false;  // the previous iteration flipped a bit, not settled yet
  if (!lead) {  // a helper follows the energies and the archive's size
    while (t <= I_max) {
      __syncthreads();  // A(t)
      const bool flip = __any_sync(kFull, count_of(t) > 0);
      bool appended = false;
      if (pend && !exploit) {
#pragma unroll
        for (int j = 0; j < K; ++j) E[j] += sFlip[(t - 1u) & 3u].d[j];
        explore_target(appended);
      }
      pend = flip;
      if (flip || by_offset) {
        if (t == I_max) {
          __syncthreads();
          if (flip && !exploit) {
#pragma unroll
            for (int j = 0; j < K; ++j) E[j] += sFlip[t & 3u].d[j];
            explore_target(appended);
          }
          __syncthreads();
          break;
        }
        ++t;
        continue;
      }
      __syncthreads();
      __syncthreads();
      const uint32_t mode = uni(sJ[0]);
      t = uni(sJ[1]);
      if (mode == kQEnd || mode == kQStayEnd) break;
      if (mode == kQLoad) {
        const int slot = uni((int)sJ[2]);
#pragma unroll
        for (int j = 0; j < K; ++j) E[j] = sAE[(size_t)j * (s + 1) + slot];
        if (gR != nullptr) __syncthreads();
        else rebuild(false);
      }
    }
    return;
  }
  int slot_new = -1;  // the slot whose least penalty the last trial gives
  while (t <= I_max) {
    __syncthreads();  // A(t)
    const int par = (int)(t & 1u);
    const bool flip = __any_sync(kFull, count_of(t) > 0);
    const uint32_t mn = state_min(par ^ 1);  // trial t - 1's
    const int slot_old = slot_new;
    slot_new = pend ? settle(t - 1u) : -1;
    sAM[slot_old >= 0 ? slot_old : s] = mn;
    if (flip || by_offset) {
      if (!flip) {
        ++nraise;
        idle_row(t);
      }
      pend = flip;
      if (t == I_max) {
        __syncthreads();
        if (flip) settle(t);
        __syncthreads();
        break;
      }
      ++t;
      continue;
    }
    pend = false;
    __syncthreads();  // trial t's least penalties
    sAM[slot_new >= 0 ? slot_new : s] = state_min(par);
    slot_new = -1;
    __syncwarp();
    if (acount == 0) {  // empty archive: nothing happens (R12)
      idle_row(t);
      ++nempty;
      const bool end = t == I_max;
      if (!end) ++t;
      if (lane == 0) {
        sJ[0] = end ? kQStayEnd : kQStay;
        sJ[1] = t;
        sJ[2] = 0u;
      }
      __syncthreads();
      if (end) break;
      continue;
    }
    // ---- jumps from iteration t on, one iteration per lane
    int slot = 0;
    bool end = false;
    const uint32_t ring_to = t + 46u;  // the ring holds the iterations up to here
    for (;;) {
      const uint32_t it = t + (uint32_t)lane;  // may pass I_max: such lanes stop
      uint32_t d[4] = {0u, it, rep, kTagRestart};
      philox10(d, k0, k1);
      const int y = pick(d[0], acount);
      const uint32_t least = sAM[y];
      const bool last = it >= I_max || it < t;  // (it < t: past 2^32)
      uint32_t hi = hiF32;                      // iteration it + 1's threshold
      if (t < nsched && !last) {
        if (it + 1u <= ring_to) {
          hi = ring[(it + 1u) % kQRing].hi;
        } else if (it + 1u < nsched) {
          const int64_t h = A.sch_hi[it];
          hi = h < 0xFFFFFFFFll ? (uint32_t)h : 0xFFFFFFFFu;
        }
      }
      const unsigned stop = __ballot_sync(kFull, last || least <= hi);
      const int k = stop ? __ffs(stop) - 1 : 31;
      if (trace != nullptr && lane <= k) {
        int64_t *tr = trace + (size_t)(it - 1) * (K + 1);
#pragma unroll
        for (int j = 0; j < K; ++j) tr[j] = sAE[(size_t)j * (s + 1) + y];
        tr[K] = -1 - (int64_t)y;
      }
      njump += (uint32_t)(k + 1);
      slot = __shfl_sync(kFull, y, k);
      if (stop) {
        end = I_max - t <= (uint32_t)k;
        t = end ? I_max : t + (uint32_t)k + 1u;
        break;
      }
      t += 32u;
    }
    if (lane == 0) {
      sJ[0] = end ? kQEnd : kQLoad;
      sJ[1] = t;
      sJ[2] = (uint32_t)slot;
      sJ[3] = sAR[slot];
    }
#pragma unroll
    for (int j = 0; j < K; ++j) E[j] = sAE[(size_t)j * (s + 1) + slot];
    __syncthreads();
    if (end) break;
    if (gR != nullptr) __syncthreads();
    else rebuild(false);
  }

  // ---- results
  __syncwarp();
  for (int y = lane; y < acount; y += 32)
#pragma unroll
    for (int j = 0; j < K; ++j) gE[(size_t)y * K + j] = sAE[(size_t)j * (s + 1) + y];
  if (lane == 0) {
    A.arch_count[rb] = acount;
#pragma unroll
    for (int j = 0; j < K; ++j) A.E_final[(size_t)rb * K + j] = E[j];
    A.stats[(size_t)rb * 4 + 0] = nflip;
    A.stats[(size_t)rb * 4 + 1] = njump;
    A.stats[(size_t)rb * 4 + 2] = nempty;
    A.stats[(size_t)rb * 4 + 3] = nraise;
  }
}

// Words per worker: four while the workers' warps fit a block beside the two
// others at 80 registers (24 warps), else eight.
inline int qubo_words(int W) { return W <= 88 ? 4 : 8; }

template <int K, int N>
const void *qubo_variant(bool narrow) {
  return narrow ? reinterpret_cast<const void *>(qubo_kernel<K, N, true>)
                : reinterpret_cast<const void *>(qubo_kernel<K, N, false>);
}

cudaError_t launch_qubo(const QArgs &a, int K, int R, int N, bool narrow, size_t smem,
                        cudaStream_t st) {
  const void *f = K == 1   ? (N == 4 ? qubo_variant<1, 4>(narrow) : qubo_variant<1, 8>(narrow))
                  : K == 2 ? (N == 4 ? qubo_variant<2, 4>(narrow) : qubo_variant<2, 8>(narrow))
                           : (N == 4 ? qubo_variant<3, 4>(narrow) : qubo_variant<3, 8>(narrow));
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  if (e != cudaSuccess) return e;
  void *args[1] = {const_cast<QArgs *>(&a)};
  e = cudaLaunchKernel(f, dim3((unsigned)R), dim3((unsigned)(32 * (a.workers + a.helpers + 2))), args, smem, st);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace
}  // namespace moda

namespace {

using moda::kMaxK;
using moda::kMaxQBits;
using moda::QArgs;

moda_status qfail(moda_status st, const std::string &msg) {
  moda::set_last_error(msg);
  return st;
}

}  // namespace

struct moda_qubo_s {
  int32_t K = 0, m = 0, W = 0;
  int device = 0;
  bool narrow = false;  // every |Delta E_j| and |E_j| < 2^30
  int32_t *dP = nullptr;
};

struct moda_qrun_s {
  moda_qubo q = nullptr;
  int32_t R = 0, s = 0;
  int64_t I_max = 0;
  bool traced = false;
  cudaStream_t stream = nullptr;
  cudaEvent_t start = nullptr, stop = nullptr;
  void *records = nullptr;
  int64_t *arch_E = nullptr, *E_final = nullptr, *stats = nullptr, *trace = nullptr;
  uint32_t *arch_bits = nullptr, *x_final = nullptr;
  int32_t *arch_count = nullptr;
};

namespace {
void free_qrun(moda_qrun r) {
  void *ptrs[] = {r->records, r->arch_E, r->E_final, r->stats, r->trace, r->arch_bits,
                  r->x_final, r->arch_count};
  for (void *p : ptrs)
    if (p) cudaFree(p);
  if (r->start) cudaEventDestroy(r->start);
  if (r->stop) cudaEventDestroy(r->stop);
}
}  // namespace

extern "C" {

moda_status moda_qubo_create(int32_t K, int32_t m, const int32_t *Q, moda_qubo *out) {
  if (!out) return qfail(MODA_EINVAL, "out is NULL");
  *out = nullptr;
  if (!Q) return qfail(MODA_EINVAL, "NULL matrix");
  if (K < 1 || K > kMaxK) return qfail(MODA_EINVAL, "K must be in [1, 3]");
  if (m < 1 || m > kMaxQBits) return qfail(MODA_EINVAL, "m must be in [1, 4096]");
  const size_t mm = (size_t)m * m;
  std::vector<int32_t> P((size_t)K * mm + moda::kQPad, 0);
  for (int j = 0; j < K; ++j) {
    const int32_t *Qj = Q + (size_t)j * mm;
    for (int p = 0; p < m; ++p)
      for (int r = 0; r < m; ++r) {
        const int lo = p < r ? p : r, hi = p < r ? r : p;
        const int64_t v = p == r ? (int64_t)Qj[(size_t)p * m + p]
                                 : (int64_t)Qj[(size_t)lo * m + hi];  // upper triangle
        if (v > 2147483647ll || v < -2147483647ll)
          return qfail(MODA_EOVERFLOW, "an entry of Q + Q^T exceeds int32");
        P[(size_t)j * mm + (size_t)p * m + r] = (int32_t)v;
      }
  }
  // the largest sum of |P_j| over a row bounds every |Delta E_j|, half of it
  // over the matrix (with the whole diagonal) every |E_j|
  int64_t most = 0;
  for (int j = 0; j < K; ++j) {
    int64_t all = 0;
    for (int p = 0; p < m; ++p) {
      int64_t sum = 0;
      for (int r = 0; r < m; ++r) sum += std::abs((int64_t)P[((size_t)j * m + p) * m + r]);
      most = std::max(most, sum);
      all += sum;
    }
    most = std::max(most, all);  // (twice the bound of |E_j|: simple and rarely binding)
  }
  moda_qubo q = new (std::nothrow) moda_qubo_s;
  if (!q) return qfail(MODA_ENOMEM, "host allocation");
  q->narrow = most < (INT64_C(1) << 30);
  q->K = K;
  q->m = m;
  q->W = (m + 31) / 32;
  cudaGetDevice(&q->device);
  cudaError_t e = cudaMalloc(&q->dP, sizeof(int32_t) * P.size());
  if (e == cudaSuccess)
    e = cudaMemcpy(q->dP, P.data(), sizeof(int32_t) * P.size(), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    if (q->dP) cudaFree(q->dP);
    delete q;
    return qfail(MODA_ECUDA, std::string("upload: ") + cudaGetErrorString(e));
  }
  *out = q;
  return MODA_OK;
}

void moda_qubo_destroy(moda_qubo q) {
  if (!q) return;
  cudaFree(q->dP);
  delete q;
}

moda_status moda_qubo_anneal(moda_qubo q, const moda_params *p, void *cuda_stream,
                             moda_qrun *out) {
  if (!out) return qfail(MODA_EINVAL, "out is NULL");
  *out = nullptr;
  if (!q || !p) return qfail(MODA_EINVAL, "NULL argument");
  const int m = q->m, K = q->K;
  if (p->replicas < 1) return qfail(MODA_EINVAL, "replicas must be >= 1");
  if (p->I_max < 0 || p->I_max > 0xFFFFFFFFll)
    return qfail(MODA_EINVAL, "I_max must be in [0, 2^32)");
  if (!(p->delta0 > 0) || !(p->deltaf > 0) || !(p->xi > 0) || !(p->xi < 1))
    return qfail(MODA_EINVAL, "need delta0 > 0, deltaf > 0, 0 < xi < 1");
  if (p->beta < 0) return qfail(MODA_EINVAL, "beta must be >= 0");
  if (p->archive_size < 0 || p->archive_size > m)
    return qfail(MODA_EINVAL, "archive_size must be in [0, m]");
  if ((p->accept != MODA_STRICT && p->accept != MODA_LENIENT) ||
      (p->archive != MODA_EXPLORE && p->archive != MODA_EXPLOIT) ||
      (p->escape != MODA_ESC_ARCHIVE && p->escape != MODA_ESC_OFFSET))
    return qfail(MODA_EINVAL, "bad accept, archive or escape mode");
  if (p->normalize || p->snapshot_every || p->fast_forward)
    return qfail(MODA_EUNSUPPORTED,
                 "normalisation, snapshots and fast-forward are bQAP-path options");
  const int s = p->archive_size > 0 ? p->archive_size : m;
  moda::ScheduleView sv{};
  cudaSetDevice(q->device);
  moda_status st = moda::schedule_view(q->device, p->delta0, p->deltaf, p->xi, p->I_max, &sv);
  if (st != MODA_OK) return st;
  moda_qrun r = new (std::nothrow) moda_qrun_s;
  if (!r) return qfail(MODA_ENOMEM, "host allocation");
  r->q = q;
  r->R = p->replicas;
  r->s = s;
  r->I_max = p->I_max;
  r->traced = p->trace != 0 && p->I_max > 0;
  r->stream = static_cast<cudaStream_t>(cuda_stream);
  const size_t R = (size_t)r->R, W = (size_t)q->W;
  cudaError_t e = cudaSuccess;
  auto alloc = [&](void **ptr, size_t nb) {
    if (e == cudaSuccess) e = cudaMalloc(ptr, nb);
  };
  alloc((void **)&r->arch_E, R * s * K * sizeof(int64_t));
  alloc((void **)&r->arch_bits, R * s * W * sizeof(uint32_t));
  alloc((void **)&r->arch_count, R * sizeof(int32_t));
  alloc((void **)&r->x_final, R * W * sizeof(uint32_t));
  alloc((void **)&r->E_final, R * K * sizeof(int64_t));
  alloc((void **)&r->stats, R * 4 * sizeof(int64_t));
  if (r->traced) alloc((void **)&r->trace, R * (size_t)p->I_max * (K + 1) * sizeof(int64_t));
  // Delta E records of the archive members, when the escape jumps and they
  // fit in 60 % of the free memory (else jumps rebuild Delta E)
  const size_t cache_bytes = R * (size_t)(s + moda::kQSpare) * (size_t)K * m *
                             (q->narrow ? sizeof(int32_t) : sizeof(int64_t));
  if (e == cudaSuccess && p->escape == MODA_ESC_ARCHIVE && p->field_cache != 2) {
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) == cudaSuccess && cache_bytes <= free_b / 10 * 6)
      alloc(&r->records, cache_bytes);
  }
  if (e == cudaSuccess) e = cudaEventCreate(&r->start);
  if (e == cudaSuccess) e = cudaEventCreate(&r->stop);
  if (e != cudaSuccess) {
    free_qrun(r);
    delete r;
    return qfail(MODA_ENOMEM, std::string("device allocation: ") + cudaGetErrorString(e));
  }
  QArgs a{};
  a.m = m;
  a.W = q->W;
  a.s = s;
  a.nsched = sv.count;
  a.I_max = p->I_max;
  a.beta = p->beta;
  a.replica_base = (uint32_t)p->replica_base;
  a.seed_lo = (uint32_t)(p->seed & 0xFFFFFFFFull);
  a.seed_hi = (uint32_t)(p->seed >> 32);
  a.accept = p->accept;
  a.archive = p->archive;
  a.escape = p->escape;
  a.P = q->dP;
  a.sch_delta = sv.delta;
  a.sch_lo = sv.lo;
  a.sch_hi = sv.hi;
  a.table = sv.table;
  a.records = r->records;
  a.arch_E = r->arch_E;
  a.arch_bits = r->arch_bits;
  a.arch_count = r->arch_count;
  a.x_final = r->x_final;
  a.E_final = r->E_final;
  a.stats = r->stats;
  a.trace = r->trace;
  const int N = moda::qubo_words(q->W);
  a.workers = (q->W + N - 1) / N;
  // helpers of the archive scan: with more than 128 slots, as the registers
  // allow beside the workers (24 warps of 80, 20 of 96)
  a.helpers = std::min({3, (s - 1) / 128, (N == 4 ? 24 : 20) - 2 - a.workers});
  const size_t smem = moda::qubo_layout(K, a.workers, q->W, s, q->narrow).total;
  e = cudaEventRecord(r->start, r->stream);
  if (e == cudaSuccess) e = moda::launch_qubo(a, K, r->R, N, q->narrow, smem, r->stream);
  if (e == cudaSuccess) e = cudaEventRecord(r->stop, r->stream);
  if (e != cudaSuccess) {
    cudaStreamSynchronize(r->stream);
    free_qrun(r);
    delete r;
    return qfail(MODA_ECUDA, std::string("launch: ") + cudaGetErrorString(e));
  }
  *out = r;
  return MODA_OK;
}

moda_status moda_qrun_wait(moda_qrun r) {
  if (!r) return qfail(MODA_EINVAL, "NULL run");
  cudaSetDevice(r->q->device);
  const cudaError_t e = cudaEventSynchronize(r->stop);
  if (e != cudaSuccess) return qfail(MODA_ECUDA, std::string("run: ") + cudaGetErrorString(e));
  return MODA_OK;
}

moda_status moda_qrun_read(moda_qrun r, int32_t *count, int64_t *E, uint32_t *bits,
                           uint32_t *x, int64_t *E_final, int64_t *stats, int64_t *trace) {
  if (!r) return qfail(MODA_EINVAL, "NULL run");
  cudaSetDevice(r->q->device);
  if (cudaEventQuery(r->stop) != cudaSuccess) return qfail(MODA_EBUSY, "run still executing");
  const size_t R = (size_t)r->R, s = (size_t)r->s, K = (size_t)r->q->K, W = (size_t)r->q->W;
  struct Item {
    void *dst;
    const void *src;
    size_t bytes;
  } items[] = {
      {count, r->arch_count, R * sizeof(int32_t)},
      {E, r->arch_E, R * s * K * sizeof(int64_t)},
      {bits, r->arch_bits, R * s * W * sizeof(uint32_t)},
      {x, r->x_final, R * W * sizeof(uint32_t)},
      {E_final, r->E_final, R * K * sizeof(int64_t)},
      {stats, r->stats, R * 4 * sizeof(int64_t)},
      {trace, r->trace, r->traced ? R * (size_t)r->I_max * (K + 1) * sizeof(int64_t) : 0},
  };
  for (const Item &it : items) {
    if (!it.dst || !it.bytes) continue;
    const cudaError_t e = cudaMemcpy(it.dst, it.src, it.bytes, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return qfail(MODA_ECUDA, std::string("read: ") + cudaGetErrorString(e));
  }
  if (trace && !r->traced) return qfail(MODA_EINVAL, "the run kept no trace");
  return MODA_OK;
}

moda_status moda_qrun_elapsed_ms(moda_qrun r, float *ms) {
  if (!r || !ms) return qfail(MODA_EINVAL, "NULL argument");
  const cudaError_t e = cudaEventElapsedTime(ms, r->start, r->stop);
  if (e != cudaSuccess) return qfail(MODA_ECUDA, cudaGetErrorString(e));
  return MODA_OK;
}

void moda_qrun_destroy(moda_qrun r) {
  if (!r) return;
  cudaSetDevice(r->q->device);
  if (r->stop) cudaEventSynchronize(r->stop);
  free_qrun(r);
  delete r;
}

}  // extern "C"
