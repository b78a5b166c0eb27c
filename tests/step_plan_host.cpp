// Prints the row plan (mm_plan.h) of every (ntheta, ns, bytes per value, V) read
// from standard input -- packed, rows, chunks, passes, cost -- and the bytes up to
// which two and more substeps of such a float32 instance go to one resident launch.
#include <cstdio>

#include "mm_plan.h"

int main() {
  int nth, ns, tsz, V;
  while (std::scanf("%d %d %d %d", &nth, &ns, &tsz, &V) == 4) {
    const mmh::RowPlan p = mmh::row_plan(nth, ns, V, tsz, 4096);
    std::printf("%d %d %d %d %.6f %zu %zu\n", (int)p.packed, p.rows, p.chunks, p.passes,
                p.passes * mmh::pass_cost(p.packed, V, tsz), mmh::resident_limit(nth, ns, 2),
                mmh::resident_limit(nth, ns, 3));
  }
  return 0;
}
