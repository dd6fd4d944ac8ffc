// The order in which the producer thread of the split product (qg_split.cu) requests its copies, and the copies
// it waits for before its block may exit: those in flight would write the shared memory of a finished block.
// Over the block's barriers as Ops, so that a host program can let any of the waits run out.
#pragma once

#ifdef __CUDACC__
#define QG_HD __host__ __device__ __forceinline__
#else
#define QG_HD inline
#endif

namespace qg {

// Unit u (64 columns of a pass): `digits` tiles of A through a ring of STAGES and one block of B into two
// buffers, B after the unit's first tile (so that this one is in flight while the first unit waits for
// the kernel before).  A wait that runs out ends the requests; every request made is waited for, oldest first
// (a buffer's barrier is then at most one phase behind the one waited for).
template <int STAGES, class Ops>
QG_HD void split_feed(Ops &ops, int units, int digits) {
  int na = 0, nb = 0;  // tiles of A and blocks of B requested
  bool ok = true;
  for (int u = 0; u < units && ok; ++u)
    for (int i = 0; i < digits && ok; ++i) {
      if (na >= STAGES && !(ok = ops.wait_a_free(na))) break;
      ops.load_a(na++, u, i);
      if (i > 0) continue;
      if (u == 0) ops.wait_inputs();
      if (u >= 2 && !(ok = ops.wait_b_free(u))) break;
      ops.load_b(u);
      nb = u + 1;
    }
  for (int q = na > STAGES ? na - STAGES : 0; q < na; ++q) ops.drain_a(q);
  for (int u = nb > 2 ? nb - 2 : 0; u < nb; ++u) ops.drain_b(u);
}

}  // namespace qg
