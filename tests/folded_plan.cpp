// Host checks of the folded skew-packed plan (k1t_plan), no GPU: the CTAs' row
// ranges cover every row of every group once and in order, every copy starts
// and ends on 16 bytes inside the tensor, a chunk fits a stage and its rows
// the consumer threads' registers, and the groups a CTA touches fit the
// scratch.  Built and run by tests/test_folded_layout.py.
#include <cstdio>

#include "grom_internal.h"

using namespace grom;

int main() {
  long bad = 0, checks = 0;
  auto check = [&](bool ok, const char* what, long n, int st) {
    ++checks;
    if (!ok && ++bad < 20) std::printf("FAIL %s n %ld storage %d\n", what, n, st);
  };
  for (int st : {GROM_F64, GROM_F32X2})
    for (int sm : {1, 132, 148, 152})
      for (long n : {1L, 2L, 3L, 4L, 5L, 17L, 63L, 64L, 65L, 96L, 129L, 200L, 511L, 513L, 769L, 1024L, 1025L, 2049L, 4096L}) {
        const K1TPlan p = k1t_plan(n, st, sm);
        check(p.grid >= 1 && p.grid <= sm && p.grid <= K1T_MAX_GRID && p.nb_max >= 1 && p.nb_max <= 4, "grid", n, st);
        check((int64_t)p.qm * K1T_CONSUMERS * p.epv >= n && p.qm >= 1, "positions", n, st);
        int m = 1, q = 0;
        for (int g = 0; g < p.grid; ++g) {
          const int4 r = p.ranges[g];
          check(r.x == m && r.y == q, "range starts where the last ended", n, st);
          const int last = k1t_last_group(r);
          check(last < n && (last < 0 || last - r.x + 1 <= p.maxseg), "groups of a CTA", n, st);
          const int ptop = last > 0 ? (last + p.epv - 1) / p.epv : 1;
          const int R = 4 * ptop <= K1T_CONSUMERS ? 4 : 2 * ptop <= K1T_CONSUMERS ? 2 : 1;
          check((int64_t)p.qm * (K1T_CONSUMERS / R) >= ptop, "positions of a CTA", n, st);
          for (; m <= last; ++m, q = 0) {
            const int rb = k1t_row_bytes(m);
            const int qe = m == r.z ? r.w : m + 1;
            check(rb % 128 == 0 && p.off[m] % 128 == 0, "alignment", n, st);
            for (int nb = 1; nb <= p.nb_max; ++nb) {
              const int rmax = k1t_rmax(st, p.qm, nb), rpc = k1t_rows_per_chunk(rb, rmax * R);
              check(rpc >= 1 && rpc * rb <= K1_STAGE_BYTES && (rpc + R - 1) / R <= rmax, "chunk", n, st);
            }
            check(qe <= m + 1 && p.off[m] + (int64_t)qe * rb <= (int64_t)p.bytes, "inside the tensor", n, st);
            if (m == r.z) {
              q = qe;
              break;
            }
          }
          if (m != r.z || q != r.w) m = r.z, q = r.w;  // an empty range, or one that ends with a group
        }
        check(m == n && q == 0, "last row", n, st);
      }
  std::printf("%ld checks, %ld failed\n", checks, bad);
  return bad != 0;
}
