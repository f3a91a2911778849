// The register annealer: Alg. 3 of arXiv 2205.13399 (the multi-objective
// Digital Annealer, Sec. 3.3) for the bi-objective QAP with one thread block
// per replica whose Delta E of both objectives stays in registers.  The
// kernel's instantiations are in moda_reg_*.cu.
//
// What bounds it.  A replica is a serial chain of iterations.  While the
// schedule cools (about 11,500 iterations on Table 1's) nearly every one
// flips a bit, and a flip changes Delta E of every bit.  A warp issues a
// dependent instruction about every four cycles, so an iteration takes as
// long as the instructions of the longest warp between its barriers; with
// more replicas than SMs integer issue bounds it.  Once the schedule has
// cooled nearly every iteration jumps to an archive member that cannot
// accept anything.
//
// Roles of the block's warps.
//   G workers own the bits: lane l of the worker that owns state word w has
//   bit 32 w + l, K words (bits per lane) to a worker.  Per bit they keep
//   Delta E_1 and Delta E_2 (modulo 2^32) and its sign 1 - 2 x.  A flip of
//   bit (j, v), s = +1 when it turns on, adds
//     (1 - 2 x_p) s (Fs^k_ij d_uv + w_k [i = j] + w_k [u = v])
//   to Delta E_k of every other bit (i, u) (Eq. cale): the flow row j and the
//   distance row v come from shared memory, Q is never stored, and since
//   both matrices have a zero diagonal the product vanishes where a penalty
//   term applies.  No field, penalty or record goes to global memory.
//   D draw warps compute delta_t T of every bit two iterations ahead, where
//   latency counts: the draws do not depend on the state, and Philox's ten
//   dependent rounds leave the workers' chain.  Where issue counts (INL) the
//   workers draw for themselves, and only for chunks of 128 bits with a bit
//   that can be accepted.
//   The scan warp keeps the archive's energies and, per slot, the least
//   acceptance penalty of the member's bits (shared memory), and runs the
//   jumps; the store warp keeps the state words, writes members' states to
//   global memory and fills the ring of schedule entries and draws.  They
//   settle the archive update of flip t - 1 while the workers are at
//   iteration t, so neither is on their chain.
// Barriers of iteration t: A(t), the whole block, after the trial's counts;
// B(t), the workers, after the warp that holds the selected bit published it.
//
// Jumps.  A bit can be accepted at iteration t only if its penalty a <= hi_t
// = floor(delta_t T_max) (every draw rejects above it, R21), so a member
// whose least penalty is above hi_t accepts nothing in that iteration,
// whatever its draws are: all of its bits are decided by one compare.  The
// scan warp takes 32 iterations at a time, one per lane (the restart draws
// and |A| are known), and stops at the first whose member may accept.  Only
// that member's Delta E are rebuilt (from its state words).  Traces of the
// n = 25 .. 75 workloads show that practically every such trial does accept
// (of 1,072 on n = 75, all), and that a run has about 1,000 of them.
//
// Rebuilds.  L_k = Fs_k M with M = X D is a contraction of three n x n
// matrices, and with at most two bits a row it runs on the tensor cores
// exactly: fp16 holds integers up to 2,048, so entries of Fs_k and M (or
// their bytes, where a sum could pass 2^24) are multiplied and summed in
// float without rounding.  (The 8-bit integer form of the same instruction
// is slow on this part: a strip of 16 rows took 3,700 cycles on n = 75.)
#pragma once

#include <cstdint>
#include <type_traits>

#include "moda_device.cuh"
#include "moda_internal.h"

namespace moda {
namespace {

// Ring entry of one iteration.
struct RRing {
  double delta;
  float cln;        // fl32(delta ln 2)
  float margin;     // half width of the band the FP32 test leaves undecided
  uint32_t sel;     // select draw
  uint32_t hi;      // floor(delta T_max), at most 2^32 - 1
  int32_t hm;       // WIDE: largest R_i + C_u of the state tried, lagging
  uint32_t pad;
};
static_assert(sizeof(RRing) == 32, "ring entry layout");

// The flipped bit of an iteration: row | column << 8 | old state << 16, and
// its Delta E.
struct RFlip {
  uint32_t code, pad;
  int64_t d1, d2;
};
static_assert(sizeof(RFlip) == 24, "flip record layout");

// A value the whole warp shares, told to the compiler as such: it then
// neither guards the votes and reductions below against divergence nor
// keeps it in a register per lane.
__device__ __forceinline__ int uni(int v) { return __shfl_sync(kFull, v, 0); }
__device__ __forceinline__ uint32_t uni(uint32_t v) { return __shfl_sync(kFull, v, 0); }

// D (16 x 8, float) += A (16 x 16 fp16, rows) B (16 x 8 fp16, columns).
__device__ __forceinline__ void mma_f16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                        uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// fp16 of an integer up to 2,048 (exact), in the low half
__device__ __forceinline__ uint32_t half_of(uint32_t v) {
  uint16_t h;
  asm("cvt.rn.f16.u16 %0, %1;" : "=h"(h) : "h"((uint16_t)v));
  return h;
}
// fp16 pair of two integers below 1,024 in the halves of x: 1,024 + v has v in
// its mantissa, less 1,024
__device__ __forceinline__ uint32_t halves_of(uint32_t x) {
  uint32_t r;
  asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(x | 0x64006400u), "r"(0xE400E400u));
  return r;
}

// EXT carries the options beyond the default algorithm, chosen at run time:
// normalisation (Sec. 4.2), the offset escape (Alg. 1) and archive snapshots;
// it takes either acceptance rule and either Delta E range.  Its penalties are
// floats s_k Delta E_k - E_off, decided by the FP32 test with a margin for
// their rounding and near it by the double operations as written.
template <int K, bool WIDE, bool LEN, bool INL, bool EXT>
__global__ void __maxnreg__(reg_regs(K)) reg_anneal_kernel(const RegLaunch L) {
  static_assert(!INL || K % 4 == 0, "inline draws come four words at a time");
  static_assert(!EXT || WIDE, "the extensions take either range");
  constexpr bool F64 = reg_f64(K);  // flows as (f1, f2) int32 pairs, else f1 | f2 << 16
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, wid = uni((int)(threadIdx.x >> 5));
  const int G = L.workers, D = INL ? 0 : L.draws;
  const int warps = G + D + 2, threads = 32 * warps;
  const bool worker = wid < G;
  const int2 item = L.items != nullptr ? L.items[blockIdx.x] : make_int2(0, (int)blockIdx.x);
  const WarpRun &R = L.runs[item.x];
  const int row = uni(item.y);
  const int n = uni(R.n), m = uni(R.m), W = uni(R.W), s = uni(R.s), se = uni(R.se);
  const int nc = (m + 127) / 128;
  if ((!EXT && (((uni(R.narrow) != 0) == WIDE) || ((uni(R.accept) != 0) != LEN))) || W > G * K) {
    // the host launches matching variants only
    if (threadIdx.x == 0) atomicExch(R.error, kErrVariant);
    return;
  }
  const uint32_t rep = uni(R.replica_base) + (uint32_t)row;
  const uint32_t k0 = uni(R.seed_lo), k1 = uni(R.seed_hi);
  const uint32_t I_max = uni((uint32_t)R.I_max);
  const uint32_t nsched = uni((uint32_t)R.nsched);
  const int64_t w1l = R.w1, w2l = R.w2;
  const uint32_t w1 = uni((uint32_t)(uint64_t)w1l), w2 = uni((uint32_t)(uint64_t)w2l);  // mod 2^32
  const uint32_t magic = uni(R.magic);
  const double *const table = R.table;
  const int hm_limit = uni(R.hm_limit);
  const int use_mma = uni(R.mma);  // 1: fragments from the flow rows, 2: from fp16 planes of Fs
  const bool fbig = uni(R.fbig) != 0;
  const int dmax = uni(R.dmax);
  auto divn = [&](int p) { return (int)__umulhi((uint32_t)p, magic); };
  const bool lenient = EXT ? uni(R.accept) != 0 : LEN;
  const bool norm = EXT && uni(R.normalize) != 0;
  const bool by_offset = EXT && uni(R.escape) != 0;
  const double s1 = EXT ? R.s1 : 1.0, s2 = EXT ? R.s2 : 1.0;
  const float s1f = (float)s1, s2f = (float)s2;
  const int64_t beta = EXT ? R.beta : 0;
  const uint32_t snap_every = EXT ? uni((uint32_t)R.snap_every) : 0u;
  const size_t nsnap = EXT ? (size_t)R.nsnap : 0;
  // a value no penalty that any draw accepts passes: floor(delta T_max), at
  // most 2^32 - 1; EXT: the bits of a float that the float form of such a
  // penalty does not pass while E_off = 0 (a trial adds 1e-6 E_off)
  auto top = [&](double delta, int64_t hi) -> uint32_t {
    if (EXT) return __float_as_uint((float)__dmul_rn(delta, __ldg(&table[0])) * (1.f + 2e-6f));
    return hi < 0xFFFFFFFFll ? (uint32_t)hi : 0xFFFFFFFFu;
  };

  const RegSmem SL = reg_smem(n, m, se, G, K, WIDE, INL, use_mma, fbig);
  constexpr int kFb = F64 ? 8 : 4;       // bytes of a flow pair
  const int fcols = reg_fcols(n, F64);
  const int frow = fcols * kFb;          // bytes of a flow row: n pairs and zeros
  unsigned char *const sFs = smem + SL.fs;
  unsigned char *const sD = smem + SL.d;
  RRing *const ring = reinterpret_cast<RRing *>(smem + SL.ring);
  int32_t *const sCnt = reinterpret_cast<int32_t *>(smem + SL.cnt);    // [2][32] accepted
  uint32_t *const sMin = reinterpret_cast<uint32_t *>(smem + SL.min);  // [2][32] least penalty
  RFlip *const sFlip = reinterpret_cast<RFlip *>(smem + SL.flip);      // [4]
  int32_t *const sTgt = reinterpret_cast<int32_t *>(smem + SL.tgt);    // [4] slot of the flip
  uint32_t *const sJ = reinterpret_cast<uint32_t *>(smem + SL.jump);   // jump: mode, t, slot
  uint32_t *const sFlags = sJ + 4;  // rebuild: 1 a row with two bits, 2 one with more
  int32_t *const sR = reinterpret_cast<int32_t *>(smem + SL.rc);       // row counts
  int32_t *const sC = sR + kMaxN;                                      // column counts
  unsigned char *const sV = smem + SL.v2;                              // [n][2] bits of a row
  uint32_t *const sX = reinterpret_cast<uint32_t *>(smem + SL.x);      // state words
  int64_t *const sSum = reinterpret_cast<int64_t *>(smem + SL.sum);    // [32][2]
  float *const sDraw = reinterpret_cast<float *>(smem + SL.draw);  // [2][128 nc] or [G][128]
  longlong2 *const sAE = reinterpret_cast<longlong2 *>(smem + SL.aE);  // archive energies
  uint32_t *const sAM = reinterpret_cast<uint32_t *>(smem + SL.aM);    // least penalties

  // ---- matrices, ring, initial state (R10) into shared memory
  for (int e = threadIdx.x; e < n * fcols; e += threads) {
    const int j = e / fcols, i = e - j * fcols;
    const int32_t f1 = i < n ? R.Fs1[j * n + i] : 0, f2 = i < n ? R.Fs2[j * n + i] : 0;
    if (F64) reinterpret_cast<int2 *>(sFs)[e] = make_int2(f1, f2);
    else reinterpret_cast<uint32_t *>(sFs)[e] = (uint32_t)f1 | ((uint32_t)f2 << 16);
  }
  for (int e = threadIdx.x; e < m; e += threads) reinterpret_cast<int32_t *>(sD)[e] = R.D[e];
  for (int c = threadIdx.x; c < nc; c += threads) {
    // chunk c's 128 bits are the four words of Philox block (c, 0, replica,
    // init): state word 4c + w is word w
    uint32_t b[4] = {(uint32_t)c, 0u, rep, kTagInit};
    philox10(b, k0, k1);
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const int lo = 32 * (4 * c + w);
      uint32_t v = b[w];
      if (lo >= m) v = 0u;
      else if (lo + 32 > m) v &= (1u << (m - lo)) - 1u;
      sX[4 * c + w] = v;
    }
  }
  // Iterations first .. first + 31 into the ring (one warp): the schedule
  // entry (Alg. 3's cooling, the last entry held once delta reaches delta_f)
  // and the select draw (0, q, replica, select).
  auto fill = [&](uint32_t first) {
    const uint32_t q = first + (uint32_t)lane;
    const uint32_t sn = sched_entry(q, nsched);
    RRing e;
    e.delta = R.sch_delta[sn];
    e.cln = accept_scale(e.delta);
    // (EXT: and 1e-6 of the penalty, see ext_penalty)
    e.margin = accept_margin(e.delta) * (EXT ? 1.6f : 1.f);
    e.hi = top(e.delta, R.sch_hi[sn]);
    uint32_t c[4] = {0u, q, rep, kTagSelect};
    philox10(c, k0, k1);
    e.sel = c[0];
    e.hm = 0;
    e.pad = 0u;
    ring[q % kRegRing] = e;
  };
  uint32_t filled = 64;
  if (wid == warps - 1) {
    fill(1);
    fill(33);
  }

  // ---- the workers' bits
  constexpr bool SMALL = K <= 8;  // registers to spare: offsets and signs unpacked
  uint32_t e1[K], e2[K];   // Delta E modulo 2^32
  uint32_t xn = 0u;        // state bits, bit k: the lane's bit of word k
  uint32_t sg[SMALL ? K : 1];  // 1 - 2 x
  // byte offsets of the bit's flow pair in a flow row and its distance in a
  // distance row (packed: fa << 16 | da); a bit past m has the zero pair
  // (and a Delta E that never changes)
  uint32_t fo[K], dof[SMALL ? K : 1];
  const int w0 = worker ? wid * K : W;  // first word (others: none)
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int p = 32 * (w0 + k) + lane;
    const int i = divn(p), u = p - i * n;
    // (a distance past the row, which no column matches)
    const uint32_t fa = (uint32_t)((p < m ? i : n) * kFb), da = (uint32_t)((p < m ? u : n) * 4);
    if (SMALL) {
      fo[k] = fa;
      dof[SMALL ? k : 0] = da;
      sg[SMALL ? k : 0] = 1u;
    } else {
      fo[k] = fa << 16 | da;
    }
    e1[k] = e2[k] = 0u;
  }
  auto fa_of = [&](int k) { return SMALL ? fo[k] : fo[k] >> 16; };
  auto da_of = [&](int k) { return SMALL ? dof[SMALL ? k : 0] : fo[k] & 0xFFFFu; };
  auto flow = [&](uint32_t at, uint32_t &f1, uint32_t &f2) {
    if (F64) {
      const uint2 f = *reinterpret_cast<const uint2 *>(sFs + at);
      f1 = f.x;
      f2 = f.y;
    } else {
      const uint32_t f = *reinterpret_cast<const uint32_t *>(sFs + at);
      f1 = f & 0xFFFFu;
      f2 = f >> 16;
    }
  };
  // row and column of the lane's bit of word k (i = n past m)
  auto i_of = [&](int k) { return (int)(fa_of(k) / kFb); };
  auto u_of = [&](int k) { return (int)(da_of(k) / 4u); };
  unsigned char *const rcp = smem + SL.rcp + 2 * kMaxN * (size_t)wid;  // WIDE: this warp's counts
  // WIDE: Delta E_1 and Delta E_2 of a bit in 64 bits, from its value modulo
  // 2^32 and the counts: L_k = +-dE_k - w_k h lies in [0, 2^31) (R20).
  auto exact64 = [&](int k, int64_t &o1, int64_t &o2) {
    const int i = i_of(k), u = u_of(k);
    if (i >= n) {
      o1 = o2 = 0x3FFFFFFF;
      return;
    }
    const int x = (int)((xn >> k) & 1u);
    const int64_t h = (int64_t)rcp[i] + rcp[kMaxN + u] - 1 - 2 * x;
    const uint32_t t1 = x ? 0u - e1[k] : e1[k];
    const uint32_t t2 = x ? 0u - e2[k] : e2[k];
    const int64_t l1 = (int64_t)(t1 - (uint32_t)((uint64_t)w1l * (uint64_t)h));
    const int64_t l2 = (int64_t)(t2 - (uint32_t)((uint64_t)w2l * (uint64_t)h));
    const int64_t f1 = l1 + w1l * h, f2 = l2 + w2l * h;
    o1 = x ? -f1 : f1;
    o2 = x ? -f2 : f2;
  };
  auto penalty64 = [&](int k) -> int64_t {
    int64_t a1, a2;
    exact64(k, a1, a2);
    a1 = a1 > 0 ? a1 : 0;
    a2 = a2 > 0 ? a2 : 0;
    return lenient ? (a1 < a2 ? a1 : a2) : a1 + a2;
  };
  // WIDE: Delta E of word k's bit in float, for states whose Delta E pass
  // int32: with h > 0 both terms of L + w h are positive, so the sum is within
  // 3 2^-24 of it, else it fits int32 exactly (w < 2^31); the sum of two
  // penalties is within 4 2^-24 (2.8e-6 delta where it is near 11.8 delta,
  // inside the margin of the FP32 test).
  auto wide_floats = [&](int k, float &f1, float &f2) {
    const int i = i_of(k), u = u_of(k);
    f1 = f2 = 1.0e38f;
    if (i >= n) return;
    const int x = (int)((xn >> k) & 1u);
    const int h = (int)rcp[i] + (int)rcp[kMaxN + u] - 1 - 2 * x;
    const uint32_t l1 = (x ? 0u - e1[k] : e1[k]) - w1 * (uint32_t)h;
    const uint32_t l2 = (x ? 0u - e2[k] : e2[k]) - w2 * (uint32_t)h;
    const float hf = (float)h;
    f1 = h > 0 ? __fmaf_rn(hf, (float)w1, __uint2float_rn(l1))
               : __int2float_rn((int32_t)(l1 + w1 * (uint32_t)h));
    f2 = h > 0 ? __fmaf_rn(hf, (float)w2, __uint2float_rn(l2))
               : __int2float_rn((int32_t)(l2 + w2 * (uint32_t)h));
    f1 = x ? -f1 : f1;
    f2 = x ? -f2 : f2;
  };
  auto penalty_wide = [&](int k) -> float {
    float f1, f2;
    wide_floats(k, f1, f2);
    f1 = fmaxf(f1, 0.f);
    f2 = fmaxf(f2, 0.f);
    return lenient ? fminf(f1, f2) : f1 + f2;
  };
  // EXT: the penalty sum_k (min_k) max(0, s_k Delta E_k - E_off) in float.
  // Near a draw's level each term is at most E_off + 11.8 delta, and its
  // error at most 6 2^-24 of that (Delta E 3, s_k and the product 2, E_off
  // 1), so two terms are within 7.2e-7 (E_off + 11.8 delta) = 7.2e-7 E_off +
  // 8.5e-6 delta.  The margin of the test adds 1e-6 (E_off + 12 delta).  The
  // bound above which a chunk is left out without its draws is (1 + 2e-6)
  // delta T_max (2.3e-5 delta) and 1e-6 E_off above delta T_max: E_off has no
  // bound in terms of delta, and its rounding alone can exceed delta T_max.
  auto ext_penalty = [&](int k, bool nar, float off) -> float {
    float f1, f2;
    if (nar) {
      f1 = __int2float_rn((int32_t)e1[k]);
      f2 = __int2float_rn((int32_t)e2[k]);
    } else if (w1l < (INT64_C(1) << 31) && w2l < (INT64_C(1) << 31)) {
      wide_floats(k, f1, f2);
    } else {
      int64_t x1, x2;
      exact64(k, x1, x2);
      f1 = __ll2float_rn(x1);
      f2 = __ll2float_rn(x2);
    }
    f1 = fmaxf(__fmaf_rn(s1f, f1, -off), 0.f);
    f2 = fmaxf(__fmaf_rn(s2f, f2, -off), 0.f);
    // (+ 0: never -0, its bits are compared as an integer)
    return (lenient ? fminf(f1, f2) : f1 + f2) + 0.f;
  };
  const bool wfloat = w1l < (INT64_C(1) << 31) && w2l < (INT64_C(1) << 31);
  // WIDE: largest R_i + C_u (the store warp).  It goes into the ring entry of
  // the trial it is for, before the barrier that trial follows: the entry of t +
  // 2 between A(t) and A(t + 1), three flips behind that trial's state.  Which
  // warp is faster then decides neither the form of a trial nor the least
  // penalty it reports, nor the counters that hang on it.
  auto bits_hm = [&]() -> int {
    int a = 0, b = 0;
    for (int i = lane; i < n; i += 32) {
      a = max(a, sR[i]);
      b = max(b, sC[i]);
    }
    a = __reduce_max_sync(kFull, a);
    b = __reduce_max_sync(kFull, b);
    return a + b;
  };

  if (use_mma == 2) {
    // Fs as fp16 for the rebuilds, zero past n: one plane an objective, or
    // (fbig) its low and its high bytes
    const int ms = reg_mstride(n), rows = (n + 15) / 16 * 16;
    for (int e = threadIdx.x; e < rows * (ms / 4); e += threads) {
      const int i = e / (ms / 4), j = 2 * (e - i * (ms / 4));
      uint32_t b[4] = {0u, 0u, 0u, 0u};
#pragma unroll
      for (int q = 0; q < 2; ++q)
        if (i < n && j + q < n) {
          const uint32_t f1 = (uint32_t)R.Fs1[i * n + j + q], f2 = (uint32_t)R.Fs2[i * n + j + q];
          b[0] |= half_of(fbig ? f1 & 255u : f1) << (16 * q);
          b[1] |= half_of(f1 >> 8) << (16 * q);
          b[2] |= half_of(fbig ? f2 & 255u : f2) << (16 * q);
          b[3] |= half_of(f2 >> 8) << (16 * q);
        }
#pragma unroll
      for (int f = 0; f < 4; ++f)
        if (fbig || f % 2 == 0)
          *reinterpret_cast<uint32_t *>(smem + SL.pl +
                                        (size_t)(fbig ? f : f / 2) * rows * ms + 4 * e) = b[f];
    }
  }

  // Delta E of the state in sX from scratch (Alg. 3's initial state, or the
  // member a jump landed on), by the whole block: the counts, then
  // L_k(i,u) = sum_j Fs^k_ij M_ju with M = X D, by matrix products where the
  // rows have at most two bits, else from blocks of rows of M in shared
  // memory.  Starts with a block barrier after which sX must be complete and
  // ends on one.  energies: also sums over the set bits of L_1 and L_2
  // (2 c_k) per warp into sSum.  at: the iteration to be tried next.  aside(): what the last (store) warp does while
  // the others scatter the set bits and form M.
  auto rebuild = [&](bool energies, uint32_t at, auto &&aside) {
    const bool helps = wid != warps - 1;
    for (int i = threadIdx.x; i < 2 * kMaxN; i += threads) sR[i] = 0;
    for (int i = threadIdx.x; i < kMaxN / 2; i += threads)
      reinterpret_cast<uint32_t *>(sV)[i] = 0xFFFFFFFFu;
    if (threadIdx.x == 0) *sFlags = 0u;
    __syncthreads();
    for (int w = threadIdx.x; helps && w < W; w += threads - 32) {
      uint32_t v = sX[w];
      while (v) {
        const int p = 32 * w + __ffs(v) - 1;
        v &= v - 1u;
        const int i = divn(p), u = p - i * n;
        const int had = atomicAdd(&sR[i], 1);
        atomicAdd(&sC[u], 1);
        if (had < 2) sV[2 * i + had] = (unsigned char)u;
        if (had >= 1) atomicOr(sFlags, had == 1 ? 1u : 2u);
      }
    }
    if (!helps) aside();
    xn = 0u;
#pragma unroll
    for (int k = 0; k < K; ++k)
      if (w0 + k < W) xn |= ((sX[w0 + k] >> lane) & 1u) << k;
    __syncthreads();
    const uint32_t flags = uni(*reinterpret_cast<volatile uint32_t *>(sFlags));
    if (use_mma != 0 && (flags & 2u) == 0u) {
      const int ms = reg_mstride(n), kq = (n + 15) / 16 * 4;
      unsigned char *const mt = smem + SL.mt;
      const int32_t *const dd = reinterpret_cast<const int32_t *>(sD);
      // one pass with whole entries of M where every sum of products stays
      // below 2^24 (the host chose fbig for the same), else one per byte
      const int mmax = (flags & 1u) ? 2 * dmax : dmax;
      const bool whole = reg_whole(mmax, n);
      int2 *const sL = reinterpret_cast<int2 *>(smem + SL.scr);
      const int gi = lane >> 2, ti = lane & 3, ut8 = (n + 7) / 8;
      const int prow = (n + 15) / 16 * 16;  // rows of a plane of Fs
      for (int mp = 0; mp < (whole ? 1 : 2); ++mp) {
        // ---- M^T as fp16: row u, column j holds sum_v x_jv d_uv (or its
        // byte mp)
        for (int jq = lane; helps && jq < kq; jq += 32) {
          uint32_t vv[4];  // two columns of each of the four rows 4 jq ..
#pragma unroll
          for (int q = 0; q < 4; ++q)
            vv[q] = 4 * jq + q < n ? reinterpret_cast<const uint16_t *>(sV)[4 * jq + q] : 0xFFFFu;
          for (int u = wid; u < n; u += warps - 1) {
            uint32_t h[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const uint32_t a = vv[q] & 255u, b = vv[q] >> 8;
              uint32_t mm = 0u;
              if (a != 255u) mm = (uint32_t)dd[a * n + u];
              if (b != 255u) mm += (uint32_t)dd[b * n + u];
              h[q] = half_of(whole ? mm : (mm >> (8 * mp)) & 255u);
            }
            *reinterpret_cast<uint2 *>(mt + u * ms + 8 * jq) =
                make_uint2(h[0] | h[1] << 16, h[2] | h[3] << 16);
          }
        }
        __syncthreads();
        // ---- strips of 32 rows, tiles of 16 rows by 8 columns shared out
        // over the warps.  A is Fs (symmetric: flow row j), from its planes
        // where they fit (a fragment register is one load), else formed from
        // the rows (whose stride keeps the loads free of bank conflicts).
        // Where there are more tiles than warps (n = 50) a warp takes both
        // halves of its columns at once, in the accumulators of the high
        // bytes: 51.4 -> 48.5 ms there, 8 words a worker.
        for (int is = 0; is < n; is += kRegStrip) {
          const int parts = is + 16 < n ? 2 : 1;  // halves of the strip with rows below n
          const bool both = K == 8 && use_mma == 2 && !fbig && parts == 2 && 2 * ut8 > warps;
          const int odd = both ? 16 * ms : prow * ms;
          for (int job = wid; job < (both ? 1 : parts) * ut8; job += warps) {
            const int half = job >= ut8 ? 1 : 0;
            const int ib = is + 16 * half, ut = 8 * (job - half * ut8);
            const unsigned char *const bm = mt + (ut + gi) * ms + 4 * ti;
            float c[4][4];  // [objective, low and high bytes of Fs or halves]
#pragma unroll
            for (int f = 0; f < 4; ++f) c[f][0] = c[f][1] = c[f][2] = c[f][3] = 0.f;
#pragma unroll 1
            for (int kb = 0; kb < n; kb += 16) {
              uint32_t a[4][4];  // [plane][fragment register]
              if (use_mma == 2) {
                const unsigned char *ap = smem + SL.pl + (ib + gi) * ms + 2 * kb + 4 * ti;
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                  const int o = 8 * (h & 1) * ms + 16 * (h >> 1);
                  a[0][h] = *reinterpret_cast<const uint32_t *>(ap + o);
                  a[2][h] = *reinterpret_cast<const uint32_t *>(ap + o + (fbig ? 2 : 1) * prow * ms);
                  if (fbig || both) {
                    a[1][h] = *reinterpret_cast<const uint32_t *>(ap + o + odd);
                    a[3][h] = *reinterpret_cast<const uint32_t *>(
                        ap + o + odd + (fbig ? 2 : 1) * prow * ms);
                  }
                }
              } else {
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                  const int i = min(ib + gi + 8 * (h & 1), n - 1);
                  const int j = kb + 2 * ti + 8 * (h >> 1);
                  uint32_t w[2];
#pragma unroll
                  for (int q = 0; q < 2; ++q) {
                    const unsigned char *fp = sFs + min(j + q, n - 1) * frow + i * kFb;
                    if (F64) {
                      const uint2 f = *reinterpret_cast<const uint2 *>(fp);
                      w[q] = __byte_perm(f.x, f.y, 0x5410);
                    } else {
                      w[q] = *reinterpret_cast<const uint32_t *>(fp);
                    }
                  }
                  const uint32_t x1 = __byte_perm(w[0], w[1], 0x5410),
                                 x2 = __byte_perm(w[0], w[1], 0x7632);
                  a[0][h] = halves_of(fbig ? x1 & 0x00FF00FFu : x1);
                  a[2][h] = halves_of(fbig ? x2 & 0x00FF00FFu : x2);
                  a[1][h] = fbig ? halves_of((x1 >> 8) & 0x00FF00FFu) : 0u;
                  a[3][h] = fbig ? halves_of((x2 >> 8) & 0x00FF00FFu) : 0u;
                }
              }
              const uint32_t b0 = *reinterpret_cast<const uint32_t *>(bm + 2 * kb);
              const uint32_t b1 = *reinterpret_cast<const uint32_t *>(bm + 2 * kb + 16);
              mma_f16(c[0], a[0], b0, b1);
              mma_f16(c[2], a[2], b0, b1);
              if (fbig || both) {
                mma_f16(c[1], a[1], b0, b1);
                mma_f16(c[3], a[3], b0, b1);
              }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              uint32_t v[4];
#pragma unroll
              for (int f = 0; f < 4; ++f) v[f] = __float2uint_rn(c[f][q]);
              const int r = 16 * half + gi + 8 * (q >> 1), u = ut + 2 * ti + (q & 1);
              if (u < n) {
                const uint32_t h1 = both ? 0u : v[1] << 8, h2 = both ? 0u : v[3] << 8;
                sL[r * n + u] =
                    make_int2((int)((v[0] + h1) << (8 * mp)), (int)((v[2] + h2) << (8 * mp)));
                if (both)
                  sL[(r + 16) * n + u] = make_int2((int)(v[1] << (8 * mp)), (int)(v[3] << (8 * mp)));
              }
            }
          }
          __syncthreads();
#pragma unroll
          for (int k = 0; k < K; ++k) {
            const int p = 32 * (w0 + k);
            if (p < (is + kRegStrip) * n && p + 32 > is * n) {
              const int i = i_of(k) - is;
              if (i >= 0 && i < kRegStrip && i + is < n) {
                const int2 v = sL[i * n + u_of(k)];
                e1[k] = (uint32_t)v.x + (mp ? e1[k] : 0u);
                e2[k] = (uint32_t)v.y + (mp ? e2[k] : 0u);
              }
            }
          }
          __syncthreads();
        }
      }
    } else {
      int32_t *const sM = reinterpret_cast<int32_t *>(smem + SL.scr);
#pragma unroll
      for (int k = 0; k < K; ++k) e1[k] = e2[k] = 0u;
      for (int jb = 0; jb < n; jb += 32) {
        const int jn = n - jb < 32 ? n - jb : 32;
        for (int e = threadIdx.x; e < jn * n; e += threads) {
          const int jj = divn(e), u = e - jj * n;
          const int b0 = (jb + jj) * n, b1 = b0 + n;  // the row's bits
          int32_t acc = 0;
          for (int w = b0 >> 5; w <= (b1 - 1) >> 5; ++w) {
            uint32_t v = sX[w];
            if (w == b0 >> 5) v &= 0xFFFFFFFFu << (b0 & 31);
            if (32 * w + 32 > b1) v &= (1u << (b1 & 31)) - 1u;
            while (v) {
              const int vv = 32 * w + __ffs(v) - 1 - b0;
              v &= v - 1u;
              acc += reinterpret_cast<const int32_t *>(sD)[vv * n + u];
            }
          }
          sM[e] = acc;
        }
        __syncthreads();
        for (int jj = 0; jj < jn; ++jj) {
#pragma unroll
          for (int k = 0; k < K; ++k) {
            uint32_t f1, f2;
            flow((uint32_t)((jb + jj) * frow) + fa_of(k), f1, f2);
            const uint32_t mm = (uint32_t)sM[jj * n + u_of(k)];
            e1[k] += f1 * mm;
            e2[k] += f2 * mm;
          }
        }
        __syncthreads();
      }
    }
    if (WIDE && worker) {
      for (int i = lane; i < kMaxN; i += 32) {
        rcp[i] = (unsigned char)sR[i];
        rcp[kMaxN + i] = (unsigned char)sC[i];
      }
      __syncwarp();
    }
    int64_t t1 = 0, t2 = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int i = i_of(k), u = u_of(k);
      const int x = (int)((xn >> k) & 1u);
      if (energies && x) {
        t1 += e1[k];
        t2 += e2[k];
      }
      if (i < n) {
        const int h = sR[i] + sC[u] - 1 - 2 * x;
        const uint32_t v1 = e1[k] + w1 * (uint32_t)h, v2 = e2[k] + w2 * (uint32_t)h;
        e1[k] = x ? 0u - v1 : v1;
        e2[k] = x ? 0u - v2 : v2;
      } else {
        e1[k] = e2[k] = 0x3FFFFFFFu;  // past m
      }
      if (SMALL) sg[SMALL ? k : 0] = 1u - 2u * (uint32_t)x;
    }
    if (energies) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        t1 += __shfl_xor_sync(kFull, t1, o);
        t2 += __shfl_xor_sync(kFull, t2, o);
      }
      if (lane == 0 && worker) {
        sSum[2 * wid] = t1;
        sSum[2 * wid + 1] = t2;
      }
    }
    if (WIDE && wid == warps - 1) {
      const int hm = bits_hm();
      if (lane < 2) ring[(at + (uint32_t)lane) % kRegRing].hm = hm;
    }
    __syncthreads();
  };

  // accepted bits of iteration t: lane w holds warp w's
  auto count_of = [&](uint32_t t) { return lane < G ? sCnt[32 * (int)(t & 1u) + lane] : 0; };

  // delta T of iteration t for the four bits 4 g .. 4 g + 3 of Philox group
  // g (see accept_level); a level below every penalty past m.
  auto levels = [&](uint32_t t, int g, float cln) -> float4 {
    uint32_t d[4] = {(uint32_t)g, t, rep, kTagAccept};
    philox10(d, k0, k1);
    float4 v;
    v.x = accept_level(d[0], cln);
    v.y = accept_level(d[1], cln);
    v.z = accept_level(d[2], cln);
    v.w = accept_level(d[3], cln);
    if (4 * g + 3 >= m) {
      if (4 * g >= m) v.x = -3.0e38f;
      if (4 * g + 1 >= m) v.y = -3.0e38f;
      if (4 * g + 2 >= m) v.z = -3.0e38f;
      v.w = -3.0e38f;
    }
    return v;
  };

  __syncthreads();
  rebuild(true, 1u, [] {});

  if (wid >= G && wid < G + D) {
    // ================= draw warps =================
    auto draw = [&](uint32_t t) {
      const float cln = ring[t % kRegRing].cln;
      float4 *to = reinterpret_cast<float4 *>(sDraw) + 32 * nc * (int)(t & 1u);
#pragma unroll 2
      for (int c = wid - G; c < nc; c += D) to[32 * c + lane] = levels(t, 32 * c + lane, cln);
    };
    uint32_t t = 1;
    if (I_max >= 1) {
      draw(1);
      draw(2);
      __syncthreads();
    }
    while (t <= I_max) {
      __syncthreads();  // A(t): trial t has read its draws
      const int total = __reduce_add_sync(kFull, count_of(t));
      if (total == 0 && !by_offset) {
        __syncthreads();
        __syncthreads();
        const uint32_t mode = uni(sJ[0]);
        t = uni(sJ[1]);
        if (mode == kRegEnd || mode == kRegStayEnd) break;
        if (mode == kRegRebuild) rebuild(false, t, [] {});
        draw(t);
        draw(t + 1u);
        __syncthreads();
        continue;
      }
      if (t == I_max) {
        __syncthreads();
        __syncthreads();
        break;
      }
      draw(t + 2u);
      ++t;
    }
    return;
  }

  if (worker) {
    // ================= workers =================
    // The parallel trial of iteration t (Eqs. pacceptms, pacceptml) on this
    // warp's words: accepted bits (ballots for a few words, else the lane's
    // own, word k at bit K - 1 - k), their count and the least penalty.
    constexpr bool BAL = K <= 4;
    // Whether the trial stands at one place, the head of the loop, or at the end
    // of each way through it.  Once is less code for the instruction cache that
    // the roles share and spills less with many words (n = 100, 32 replicas
    // 102.2 -> 95.2 ms, n = 76, 150 of them 84.7 -> 83.0, n = 50 48.6 -> 47.0, n = 60
    // with snapshots 46.4 -> 45.5); with few, or beyond int32 with eight, the ends
    // run on into the trial better (n = 41 beyond int32 61.5 against 65.7, n = 40
    // normalised 29.1 and 30.5, n = 75 110.6 and 111.6).
    constexpr bool ONCE = K >= 16 || (K == 8 && (!WIDE || EXT));
    uint32_t acc[BAL ? K : 1], accb = 0u, amin = 0u;
    int cnt = 0;
    int64_t Eoff = 0;  // the offset escape's E_off
    auto trial = [&](uint32_t t) {
      const RRing &r = ring[t % kRegRing];
      const float off = EXT ? __ll2float_rn(Eoff) : 0.f;
      const float margin = EXT ? r.margin + 1e-6f * off : r.margin;
      // every |Delta E_k| of the state fits int32 (a bound on the counts that
      // lags by at most three flips, which the limit allows for)
      const bool nar = !WIDE || uni(r.hm) <= hm_limit;
      uint32_t a[K];  // penalties; floats where not nar
      float near = 3.0e38f;
      accb = 0u;
      cnt = 0;
      if (EXT) {
        float least = 3.0e38f;
#pragma unroll
        for (int k = 0; k < K; ++k) {
          const float v = ext_penalty(k, nar, off);
          least = fminf(least, v);
          a[k] = __float_as_uint(v);
        }
        amin = nar ? __float_as_uint(least * (1.f - 2e-6f)) : 0u;
      } else if (!WIDE || nar) {
        amin = 0xFFFFFFFFu;
#pragma unroll
        for (int k = 0; k < K; ++k) {
          const uint32_t a1 = (uint32_t)max((int32_t)e1[k], 0),
                         a2 = (uint32_t)max((int32_t)e2[k], 0);
          a[k] = LEN ? min(a1, a2) : a1 + a2;
        }
        if (K == 1) {
          amin = a[0];
        } else {
#pragma unroll
          for (int k = 0; k < K; k += 2) amin = __vimin3_u32(amin, a[k], a[k + 1]);
        }
      } else {
        amin = 0u;  // not known exactly: the slot counts as able to accept
#pragma unroll
        for (int k = 0; k < K; ++k)
          a[k] = __float_as_uint(wfloat ? penalty_wide(k) : penalty_f32(penalty64(k)));
      }
      auto decide = [&](int k, float lv) {
        const float diff =
            (!EXT && (!WIDE || nar) ? __uint2float_rn(a[k]) : __uint_as_float(a[k])) - lv;
        near = fminf(near, fabsf(diff));
        if (BAL) {
          const uint32_t b = __ballot_sync(kFull, diff < 0.f);
          cnt += __popc(b);
          acc[BAL ? k : 0] = b;
        } else {
          accb = __funnelshift_l(__float_as_uint(diff), accb, 1);  // its sign
        }
      };
      if (INL) {
        const uint32_t hi =
            EXT ? __float_as_uint(__uint_as_float(r.hi) + 1e-6f * off) : r.hi;
        float *const mine = sDraw + 128 * wid;  // the chunk's levels by bit
#pragma unroll
        for (int kc = 0; kc < K; kc += 4) {
          bool any = w0 + kc < W;
          if (any && (EXT || !WIDE || nar))
            any = __any_sync(kFull, min(min(a[kc], a[kc + 1]), min(a[kc + 2], a[kc + 3])) <= hi);
          if (any) {
            __syncwarp();  // the last chunk's levels have been read
            reinterpret_cast<float4 *>(mine)[lane] = levels(t, 8 * (w0 + kc) + lane, r.cln);
            __syncwarp();
#pragma unroll
            for (int q = 0; q < 4; ++q) decide(kc + q, mine[32 * q + lane]);
          } else if (BAL) {
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[BAL ? kc + q : 0] = 0u;
          } else {
            accb <<= 4;
          }
        }
      } else {
        const float *from = sDraw + 128 * nc * (int)(t & 1u) + 32 * w0 + lane;
#pragma unroll
        for (int k = 0; k < K; ++k) {
          if (K == 1 || w0 + k < 4 * nc) decide(k, from[32 * k]);
          else if (BAL) acc[BAL ? k : 0] = 0u;
        }
      }
      if (__any_sync(kFull, near <= margin)) {
        // some bit lies within the error of the FP32 test: the IEEE double
        // test of R7 for this warp's words
        const double delta = r.delta;
        cnt = 0;
        accb = 0u;
#pragma unroll 1
        for (int kk = 0; kk < K; ++kk) {
          uint32_t ak = 0u;
          int64_t al = 0, x1 = 0, x2 = 0;
#pragma unroll
          for (int k = 0; k < K; ++k)
            if (k == kk) {
              ak = a[k];
              if (EXT) {
                if (nar) {
                  x1 = (int32_t)e1[k];
                  x2 = (int32_t)e2[k];
                } else {
                  exact64(k, x1, x2);
                }
              } else if (WIDE && !nar) {
                al = penalty64(k);
              }
            }
          const int p = 32 * (w0 + kk) + lane;
          uint32_t d[4] = {(uint32_t)(p >> 2), t, rep, kTagAccept};
          philox10(d, k0, k1);
          double ad = WIDE && !nar ? (double)al : (double)ak;
          if (EXT && norm) {  // s_1 Delta E_1 (- E_off), ... in IEEE double, as written
            double y1 = __dmul_rn(s1, (double)x1), y2 = __dmul_rn(s2, (double)x2);
            if (by_offset) {
              y1 = __dsub_rn(y1, (double)Eoff);
              y2 = __dsub_rn(y2, (double)Eoff);
            }
            y1 = y1 > 0.0 ? y1 : 0.0;
            y2 = y2 > 0.0 ? y2 : 0.0;
            ad = lenient ? (y1 < y2 ? y1 : y2) : __dadd_rn(y1, y2);
          } else if (EXT) {
            x1 = x1 > Eoff ? x1 - Eoff : 0;
            x2 = x2 > Eoff ? x2 - Eoff : 0;
            ad = (double)(lenient ? (x1 < x2 ? x1 : x2) : x1 + x2);
          }
          const bool ok = p < m && ad <= __dmul_rn(delta, __ldg(&table[word_of(d, p & 3) >> 16]));
          const uint32_t b = __ballot_sync(kFull, ok);
          cnt += __popc(b);
          accb = accb << 1 | (ok ? 1u : 0u);
          if (BAL) {
#pragma unroll
            for (int k = 0; k < K; ++k)
              if (k == kk) acc[BAL ? k : 0] = b;
          }
        }
      } else if (!BAL) {
        cnt = __reduce_add_sync(kFull, __popc(accb));
      }
      if (lane == 0) sCnt[32 * (int)(t & 1u) + wid] = cnt;
    };

    uint32_t t = 1;
    if (I_max >= 1 && D > 0) __syncthreads();
    if (!ONCE && I_max >= 1) trial(1);
    while (t <= I_max) {
      if (ONCE) trial(t);
      const uint32_t sel = ring[t % kRegRing].sel;
      __syncthreads();  // A(t): the trial's counts are complete
      const uint32_t c = (uint32_t)count_of(t);
      const uint32_t mnw = __reduce_min_sync(kFull, amin);
      // all accepted bits, and above bit 16 those of the warps before
      const uint32_t sums = __reduce_add_sync(kFull, lane < wid ? c | c << 16 : c);
      const int total = (int)(sums & 0xFFFFu), before = (int)(sums >> 16);
      if (lane == 0) sMin[32 * (int)(t & 1u) + wid] = mnw;
      if (EXT && total == 0 && by_offset) {  // Alg. 1: raise the offset
        Eoff += beta;
        if (t == I_max) {
          __syncthreads();
          __syncthreads();
          break;
        }
        ++t;
        if (!ONCE) trial(t);
        continue;
      }
      if (total == 0) {
        __syncthreads();  // the least penalties are complete
        __syncthreads();  // the scan warp has settled the jumps
        const uint32_t mode = uni(sJ[0]);
        t = uni(sJ[1]);
        if (mode == kRegEnd || mode == kRegStayEnd) break;
        if (mode == kRegRebuild) rebuild(false, t, [] {});
        if (D > 0) __syncthreads();  // draws
        if (!ONCE) trial(t);
        continue;
      }
      // ---- one accepted bit at random (R11): rank r in ascending bit
      // order; the lane that holds it publishes it
      const int r = uni(pick(sel, total)) - before;
      if (r >= 0 && r < cnt) {
        // its word (kw), that word's ballot and the rank within it
        int kw = 0, rw = r;
        uint32_t bw = BAL ? acc[0] : __ballot_sync(kFull, (accb >> (K - 1)) & 1u);
        if (K > 1) {
          int upto = __popc(bw);
#pragma unroll
          for (int k = 1; k < K; ++k) {
            const uint32_t b =
                BAL ? acc[BAL ? k : 0] : __ballot_sync(kFull, (accb >> (K - 1 - k)) & 1u);
            if (r >= upto) {
              kw = k;
              bw = b;
              rw = r - upto;
            }
            upto += __popc(b);
          }
        }
        const bool mine = ((bw >> lane) & 1u) && __popc(bw & ((1u << lane) - 1u)) == rw;
#pragma unroll
        for (int k = 0; k < K; ++k)
          if (kw == k && mine) {
            RFlip f;
            f.code = (uint32_t)i_of(k) | (uint32_t)u_of(k) << 8 | ((xn >> k) & 1u) << 16;
            f.pad = 0u;
            if (WIDE) {
              exact64(k, f.d1, f.d2);
            } else {
              f.d1 = (int32_t)e1[k];
              f.d2 = (int32_t)e2[k];
            }
            sFlip[t & 3u] = f;
          }
      }
      if (t == I_max) {
        __syncthreads();  // the scan and the store warp settle the last flip
        __syncthreads();
        break;
      }
      if (G > 1) asm volatile("bar.sync 1, %0;" ::"r"(32 * G) : "memory");  // B(t)
      else __syncwarp();
      if (EXT) Eoff = 0;
      const uint32_t fc = uni(sFlip[t & 3u].code);
      const uint32_t j = fc & 255u, v = (fc >> 8) & 255u;
      const uint32_t sgn = 1u - 2u * (fc >> 16);  // +1: the bit turns on
      if (WIDE) {
        if (lane == 0) {
          rcp[j] = (unsigned char)((uint32_t)rcp[j] + sgn);
          rcp[kMaxN + v] = (unsigned char)((uint32_t)rcp[kMaxN + v] + sgn);
        }
        __syncwarp();
      }
      // ---- the flip's outer product on this warp's bits
      const uint32_t fbase = j * (uint32_t)frow, dbase = v * 4u * (uint32_t)n;
      const uint32_t fj = j * kFb, dv = v * 4u;
      const int ps = (int)(j * (uint32_t)n + v);
      const uint32_t xs = fc >> 16 ? ~xn : xn;  // bit k set: this bit's change is negative
      const uint32_t mw = (uint32_t)((ps >> 5) - w0);  // its word among the warp's, if < K
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const uint32_t fa = fa_of(k), da = da_of(k);
        uint32_t f1, f2;
        flow(fbase + fa, f1, f2);
        const uint32_t d = *reinterpret_cast<const uint32_t *>(sD + dbase + da);
        const uint32_t sk = SMALL ? sg[SMALL ? k : 0] * sgn : 1u - 2u * ((xs >> k) & 1u);  // +-1
        const uint32_t dq = d * sk;
        e1[k] += f1 * dq;
        e2[k] += f2 * dq;
        if (fa == fj || da == dv) {
          e1[k] += sk * w1;
          e2[k] += sk * w2;
        }
      }
      // the flipped bit's Delta E only changes sign; above it got + w_k (its
      // products are 0)
      if (mw < (uint32_t)K) {
#pragma unroll
        for (int k = 0; k < K; ++k)
          if (mw == (uint32_t)k && lane == (ps & 31)) {
            e1[k] = w1 - e1[k];
            e2[k] = w2 - e2[k];
            xn ^= 1u << k;
            if (SMALL) sg[SMALL ? k : 0] = 0u - sg[SMALL ? k : 0];
          }
      }
      ++t;
      if (!ONCE) trial(t);
    }
    return;
  }

  int64_t *const gE = R.arch_E + (size_t)row * s * 2;
  uint32_t *const gB = R.arch_bits + (size_t)row * s * W;
  uint32_t *const gM = R.arch_min ? R.arch_min + (size_t)row * s : nullptr;

  if (wid == warps - 1) {
    // ================= store warp =================
    int members = 0;  // |A| as stored
    // EXT: the states of the snapshots up to iteration `upto`, whose flips are
    // stored (the scan warp copies the energies)
    uint32_t snap = snap_every;
    auto snapshots = [&](uint32_t upto) {
      if constexpr (EXT) {
        if (snap_every == 0u) return;
        for (; snap <= upto && snap != 0u; snap += snap_every) {
          const size_t j = snap / snap_every - 1u;
          if (j >= nsnap) break;
          uint32_t *to = R.snap_bits + ((size_t)row * nsnap + j) * (size_t)s * W;
          const int words = members * W;
#pragma unroll 8
          for (int q = lane; q < words; q += 32) to[q] = gB[q];
        }
      }
    };
    // The state words of the last stored flip in sX; flip tp's follow once
    // its slot is known, an iteration later than the scan warp settles it.
    auto store = [&](uint32_t tp) {
      const uint32_t fc = uni(sFlip[tp & 3u].code);
      const int target = uni(sTgt[tp & 3u]);
      const int fi = (int)(fc & 255u), fu = (int)((fc >> 8) & 255u), ps = fi * n + fu;
      if (lane == 0) sX[ps >> 5] ^= 1u << (ps & 31);
      __syncwarp();
      if (target >= 0) {
        for (int q = lane; q < W; q += 32) gB[(size_t)target * W + q] = sX[q];
        members = members > target ? members : target + 1;
      }
      if (WIDE) {
        if (lane == 0) {
          const int sgn = 1 - 2 * (int)(fc >> 16);
          sR[fi] += sgn;
          sC[fu] += sgn;
        }
        __syncwarp();
        const int hm = bits_hm();
        if (lane == 0) ring[(tp + 4u) % kRegRing].hm = hm;
      }
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
    if (I_max >= 1 && D > 0) __syncthreads();
    while (t <= I_max) {
      __syncthreads();  // A(t)
      const int total = __reduce_add_sync(kFull, count_of(t));
      if (p2) store(t - 2u);  // (with the bound of trial t + 2)
      else if (WIDE && lane == 0) ring[(t + 2u) % kRegRing].hm = ring[(t + 1u) % kRegRing].hm;
      if (EXT && t > 2u) snapshots(t - 2u);
      if (total > 0 || by_offset) {
        p2 = p1;
        p1 = total > 0;
        if (t == I_max) {
          __syncthreads();
          if (p2) store(t - 1u);
          if (EXT) snapshots(t - 1u);
          __syncthreads();
          if (p1) store(t);
          if (EXT) snapshots(t);
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
      if (EXT) snapshots(mode == kRegEnd || mode == kRegStayEnd ? I_max : t - 1u);
      if (mode == kRegEnd || mode == kRegRebuild)  // the member the jumps ended on
        for (int q = lane; q < W; q += 32) sX[q] = gB[(size_t)slot * W + q];  // (written here)
      if (mode == kRegEnd || mode == kRegStayEnd) break;
      if (mode == kRegRebuild) rebuild(false, t, [&] { refill(t); });
      else refill(t);
      if (D > 0) __syncthreads();  // draws
    }
    __syncwarp();
    for (int q = lane; q < W; q += 32) R.x_final[(size_t)row * W + q] = sX[q];
    return;
  }

  // ================= scan warp =================
  int64_t E1, E2;
  {
    int64_t t1 = 0, t2 = 0, gp = 0;
    for (int w = 0; w < G; ++w) {
      t1 += sSum[2 * w];
      t2 += sSum[2 * w + 1];
    }
    for (int i = 0; i < n; ++i) {
      const int64_t dr = 1 - (int64_t)sR[i], dc = 1 - (int64_t)sC[i];
      gp += dr * dr + dc * dc;
    }
    E1 = t1 / 2 + w1l * (gp / 2);
    E2 = t2 / 2 + w2l * (gp / 2);
  }
  const bool exploit = uni(R.archive) != 0;
  int64_t *const trace = R.trace ? R.trace + (size_t)row * (size_t)I_max * 3 : nullptr;
  const uint32_t hiF32 = top(R.sch_delta[nsched - 1], R.sch_hi[nsched - 1]);
  int acount = 0;
  uint32_t nflip = 0, njump = 0, nempty = 0, nrebuild = 0, nraise = 0;
  auto slotE = [&](int y) {
    return y < se ? sAE[y] : make_longlong2(gE[2 * y], gE[2 * y + 1]);
  };
  // the least penalty of the state of the trial of parity par
  auto state_min = [&](int par) {
    return __reduce_min_sync(kFull, lane < G ? sMin[32 * par + lane] : 0xFFFFFFFFu);
  };
  // (every lane stores the same value: no branch; slot se is never read)
  auto put_min = [&](int y, uint32_t mn) {
    sAM[y >= 0 && y < se ? y : se] = mn;
    if (y >= se) gM[y] = mn;
  };
  // x = (E1, E2) dominates (y1, y2): both differences y - x are >= 0 and not
  // both are 0
  auto dom = [&](const longlong2 &y) {
    const int64_t d1 = y.x - E1, d2 = y.y - E2;
    return (d1 | d2) > 0;  // (no sign bit set, some bit set)
  };
  // Settles the flip of iteration tp: energies and archive (Alg. 4 or 5).
  // Returns the slot that took the state, or -1; its least penalty follows
  // once the next trial's are in.
  auto settle = [&](uint32_t tp) -> int {
    const RFlip &f = sFlip[tp & 3u];
    E1 += f.d1;
    E2 += f.d2;
    int target = -1;
    if (!exploit) {
      // the first member x dominates is replaced; else x is appended
      const int on = acount < se ? acount : se;
      for (int base = 0; base < on; base += 128) {
        unsigned bal[4];
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          const int y = base + 32 * g + lane;
          bal[g] = __ballot_sync(kFull, y < on && dom(sAE[y <= se ? y : se]));
        }
        const unsigned any = bal[0] | bal[1] | bal[2] | bal[3];
        if (any) {
          const unsigned b = bal[0] ? bal[0] : bal[1] ? bal[1] : bal[2] ? bal[2] : bal[3];
          target = base + (bal[0] ? 0 : bal[1] ? 32 : bal[2] ? 64 : 96) + __ffs(b) - 1;
          break;
        }
      }
      if (acount > se)
        for (int base = se; base < acount && target < 0; base += 32) {
          const int y = base + lane;
          const unsigned bal = __ballot_sync(
              kFull, y < acount && dom(make_longlong2(gE[2 * y], gE[2 * y + 1])));
          if (bal) target = base + __ffs(bal) - 1;
        }
      if (target < 0 && acount < s) target = acount++;
    } else {
      // no member may dominate x; then a random dominated member is
      // replaced (exploit draw, slot order), else x is appended
      int nb = 0;
      bool anyd = false;
      for (int base = 0; base < acount; base += 32) {
        const int y = base + lane;
        bool dm = false, domd = false;
        if (y < acount) {
          const longlong2 ye = slotE(y);
          dm = dom(ye);
          domd = dominates(ye.x, ye.y, E1, E2);
        }
        nb += __popc(__ballot_sync(kFull, dm));
        anyd |= __any_sync(kFull, domd) != 0;
      }
      if (!anyd) {
        if (nb > 0) {
          uint32_t x[4] = {0u, tp, rep, kTagExploit};
          philox10(x, k0, k1);
          int want = uni(pick(x[0], nb));
          for (int base = 0; base < acount; base += 32) {
            const int y = base + lane;
            const unsigned bal = __ballot_sync(kFull, y < acount && dom(slotE(y)));
            const int cb = __popc(bal);
            if (want < cb) {
              target = base + nth_set_bit(bal, want);
              break;
            }
            want -= cb;
          }
        } else if (acount < s) {
          target = acount++;
        }
      }
    }
    sTgt[tp & 3u] = target;
    sAE[target >= 0 && target < se ? target : se] = make_longlong2(E1, E2);
    if (target >= se && lane == 0) {
      gE[2 * target] = E1;
      gE[2 * target + 1] = E2;
    }
    if (trace != nullptr && lane == 0) {
      int64_t *tr = trace + (size_t)(tp - 1) * 3;
      tr[0] = E1;
      tr[1] = E2;
      tr[2] = (int64_t)(f.code & 255u) * n + (int64_t)((f.code >> 8) & 255u);
    }
    ++nflip;
    __syncwarp();
    return target;
  };

  // EXT: the energies of the snapshots up to iteration `upto`, whose flips are
  // settled
  uint32_t snap = snap_every;
  auto snapshots = [&](uint32_t upto) {
    if constexpr (EXT) {
      if (snap_every == 0u) return;
      for (; snap <= upto && snap != 0u; snap += snap_every) {
        const size_t j = snap / snap_every - 1u;
        if (j >= nsnap) break;
        const size_t at = (size_t)row * nsnap + j;
        longlong2 *to = reinterpret_cast<longlong2 *>(R.snap_E) + at * (size_t)s;
        for (int y = lane; y < acount; y += 32) to[y] = slotE(y);
        if (lane == 0) R.snap_count[at] = acount;
      }
    }
  };

  uint32_t t = 1;
  bool pend = false;  // the previous iteration flipped a bit, not settled yet
  int slot_new = -1;  // the slot whose least penalty the last trial gives
  if (I_max >= 1 && D > 0) __syncthreads();
  while (t <= I_max) {
    __syncthreads();  // A(t)
    const int par = (int)(t & 1u);
    const bool flip = __any_sync(kFull, count_of(t) > 0);
    const uint32_t mn = state_min(par ^ 1);  // trial t - 1's
    const int slot_old = slot_new;
    slot_new = pend ? settle(t - 1u) : -1;
    put_min(slot_old, mn);
    if (EXT && t > 1u) snapshots(t - 1u);
    if (flip || by_offset) {
      if (EXT && !flip) {
        ++nraise;
        if (trace != nullptr && lane == 0) {
          int64_t *tr = trace + (size_t)(t - 1) * 3;
          tr[0] = E1;
          tr[1] = E2;
          tr[2] = INT64_MIN;
        }
      }
      pend = flip;
      if (t == I_max) {
        __syncthreads();
        if (flip) settle(t);
        if (EXT) snapshots(t);
        __syncthreads();
        break;
      }
      ++t;
      continue;
    }
    pend = false;
    __syncthreads();  // trial t's least penalties
    put_min(slot_new, state_min(par));
    slot_new = -1;
    __syncwarp();
    if (acount == 0) {  // empty archive: nothing happens (R12)
      if (trace != nullptr && lane == 0) {
        int64_t *tr = trace + (size_t)(t - 1) * 3;
        tr[0] = E1;
        tr[1] = E2;
        tr[2] = INT64_MIN;
      }
      ++nempty;
      const bool end = t == I_max;
      if (EXT) snapshots(t);
      if (!end) ++t;
      if (lane == 0) {
        sJ[0] = end ? kRegStayEnd : kRegStay;  // sX still holds the state
        sJ[1] = t;
        sJ[2] = 0u;
      }
      __syncthreads();
      if (end) break;
      if (D > 0) __syncthreads();
      continue;
    }
    // ---- jumps from iteration t on, one iteration per lane: lane k's
    // iteration t + k jumps to the member its restart draw picks, and
    // iteration t + k + 1 tries it
    int slot = 0;
    bool end = false;
    const uint32_t ring_to = t + 46u;  // the ring holds the iterations up to here
    for (;;) {
      if (trace == nullptr && t >= nsched) {
        // the schedule is frozen: four batches' draws at a time (they hide
        // one another's latency) while no member may accept
        while (I_max - t >= 128u) {
          bool live = false;
#pragma unroll
          for (uint32_t g = 0; g < 4u; ++g) {
            uint32_t d[4] = {0u, t + 32u * g + (uint32_t)lane, rep, kTagRestart};
            philox10(d, k0, k1);
            const int y = pick(d[0], acount);
            live |= (y < se ? sAM[y] : gM[y]) <= hiF32;
          }
          if (__any_sync(kFull, live)) break;
          njump += 128u;
          t += 128u;
        }
      }
      const uint32_t it = t + (uint32_t)lane;  // may pass I_max: such lanes stop
      uint32_t d[4] = {0u, it, rep, kTagRestart};
      philox10(d, k0, k1);
      const int y = pick(d[0], acount);
      const uint32_t mn = y < se ? sAM[y] : gM[y];
      const bool last = it >= I_max || it < t;  // (it < t: past 2^32)
      uint32_t hi = hiF32;                      // iteration it + 1's threshold
      if (t < nsched && !last) {
        if (it + 1u <= ring_to) {
          hi = ring[(it + 1u) % kRegRing].hi;
        } else if (it + 1u < nsched) {
          hi = top(R.sch_delta[it], R.sch_hi[it]);
        }
      }
      const unsigned stop = __ballot_sync(kFull, last || mn <= hi);
      const int k = stop ? __ffs(stop) - 1 : 31;
      if (trace != nullptr && lane <= k) {
        const longlong2 ye = slotE(y);
        int64_t *tr = trace + (size_t)(it - 1) * 3;
        tr[0] = ye.x;
        tr[1] = ye.y;
        tr[2] = -1 - (int64_t)y;
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
    if (EXT) snapshots(end ? I_max : t - 1u);
    if (lane == 0) {
      sJ[0] = end ? kRegEnd : kRegRebuild;
      sJ[1] = t;
      sJ[2] = (uint32_t)slot;
    }
    {
      const longlong2 ye = slotE(slot);
      E1 = ye.x;
      E2 = ye.y;
    }
    __syncthreads();
    if (end) break;
    ++nrebuild;
    rebuild(false, t, [] {});
    if (D > 0) __syncthreads();  // draws
  }

  // ---- results
  __syncwarp();
  for (int y = lane; y < acount && y < se; y += 32) {
    gE[2 * y] = sAE[y].x;
    gE[2 * y + 1] = sAE[y].y;
  }
  if (lane == 0) {
    R.E_final[2 * row] = E1;
    R.E_final[2 * row + 1] = E2;
    R.arch_count[row] = acount;
    int64_t *st = R.stats + (size_t)kStats * row;
    st[0] = nflip;
    st[1] = njump;
    st[2] = nempty;
    st[3] = nraise;
    st[4] = 0;
    st[5] = (int64_t)njump - (int64_t)nrebuild;
    st[6] = 0;
    st[7] = nrebuild;
  }
}

}  // namespace
}  // namespace moda
