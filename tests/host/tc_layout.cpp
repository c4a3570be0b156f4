// Shared-memory layout of the sliced GEMM, for the host: the last byte that
// the loads of op(B)'s fragments touch, relative to its slices' first.
#include <algorithm>

#include "h2_tc_layout.h"

extern "C" int fragment_end(int S, int n) {
  int end = 0;
  for (int ct = 0; ct < (n + 7) / 8; ++ct)
    for (int ks = 0; ks < 2; ++ks)
      for (int q = 0; q < (S + 1) / 2; ++q)
        for (int lane = 0; lane < h2::tc_b_lanes(S, q); ++lane)
          end = std::max(end, (int)h2::tc_b_lane(lane, ct, ks) + q * 2 * h2::TC_SLICE + 16);
  return end;
}
extern "C" int slices_end(int S) { return S * h2::TC_SLICE; }
// bytes of the launch behind op(B)'s first slice
extern "C" int behind_b(int S, int m, int n) { return h2::tc_smem_bytes(S, m, n, false) - S * h2::TC_SLICE; }
