// Host check of the iteration arithmetic the annealing kernels share
// (moda::in_run, in_run_ahead, sched_entry, ring_skip, ring_short) up to I_max =
// 2^32 - 1: loops end after the last iteration, targets past the end are not in
// the run, every schedule entry looked up exists, and the ring of 128 entries,
// filled 32 at a time, holds iterations t .. min(t + 47, I_max) however far t
// moves.
// Exits nonzero on the first violation.
#include <cstdio>
#include <random>

#include "moda_internal.h"

static int failures = 0;

static void check(bool ok, const char *what, uint64_t a, uint64_t b) {
  if (!ok && ++failures < 20)
    std::printf("%s: %llu %llu\n", what, (unsigned long long)a, (unsigned long long)b);
}

int main() {
  const uint32_t last = 0xFFFFFFFFu;
  for (uint32_t I_max : {0u, 1u, 2u, 47u, 1000u, last - 200u, last - 1u, last}) {
    check(moda::in_run(1u, I_max) == (I_max >= 1u), "first iteration", 1, I_max);
    check(!moda::in_run(I_max + 1u, I_max), "past the last iteration", I_max + 1ull, I_max);
    for (uint32_t back = 0; back < 64u && back < I_max; ++back) {
      const uint32_t t = I_max - back;
      check(moda::in_run(t, I_max), "in the run", t, I_max);
      for (uint32_t ahead = 0; ahead < 32u; ++ahead)
        check(moda::in_run_ahead(t, ahead, I_max) == ((uint64_t)t + ahead <= I_max), "ahead", t,
              ahead);
    }
  }
  for (uint32_t nsched : {1u, 2u, 11508u, 2147483647u})
    for (uint64_t q : {0ull, 1ull, 2ull, 11507ull, 11508ull, 11509ull, 4294967295ull}) {
      const uint32_t e = moda::sched_entry((uint32_t)q, nsched);
      check(e < nsched, "entry exists", q, nsched);
      if (q > 0) check(e == (q <= nsched ? q : nsched) - 1u, "entry of the iteration", q, nsched);
    }
  std::mt19937_64 rng(5);
  for (int run = 0; run < 3000; ++run) {
    // from the start, or from near the end, by steps of one and jumps of any
    // length; entry q % 128 of the ring holds iteration ring[q % 128]
    const uint32_t I_max = last - (uint32_t)(rng() % 100);
    uint32_t filled = 64;
    static uint32_t ring[128];
    for (uint32_t q = 1; q <= 64; ++q) ring[q % 128] = q;
    uint32_t t = 1;
    int fills = 0;
    for (int step = 0; step < 400 && moda::in_run(t, I_max); ++step) {
      for (uint32_t a = 0; a < 48u && moda::in_run_ahead(t, a, I_max); ++a)
        check(ring[(t + a) % 128] == t + a, "held", t + a, ring[(t + a) % 128]);
      if (t == I_max) break;
      const uint64_t left = I_max - t, kind = rng() % 8;
      const uint64_t by = kind < 5 || left < 2 ? 1
                          : kind == 5          ? 1 + rng() % (left < 128 ? left : 128)
                          : kind == 6          ? 1 + rng() % left
                          : left > 90          ? left - rng() % 90
                                               : 1;
      // a trial refills for the next iteration but one, a jump for where it lands
      const uint32_t from = t;
      t += (uint32_t)by;
      const uint32_t to = by > 1 ? t : from + 2u;
      filled = moda::ring_skip(filled, from, to);
      while (moda::ring_short(filled, to)) {
        const uint32_t first = filled + 1u;
        for (uint32_t l = 0; l < 32; ++l) {
          ring[(first + l) % 128] = first + l;
          check(moda::sched_entry(first + l, 11508u) < 11508u, "entry of a fill", first + l, 0);
        }
        filled += 32;
        if (++fills > 3 * 400) break;
      }
    }
    check(fills <= 3 * 400, "fills", (uint64_t)fills, 0);
    if (failures) return 1;
  }
  if (failures) return 1;
  std::printf("iterations ok\n");
  return 0;
}
