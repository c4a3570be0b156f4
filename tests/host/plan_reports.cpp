// Plans of a structure without any adaptive rank: one leaf, so no admissible
// block.
#include <numeric>

#include "../../paper_2403_01566_gb300/csrc/h2_build.h"
#include "../../paper_2403_01566_gb300/csrc/h2_plan.h"

namespace {
h2::MatDesc one_leaf(h2::Tree& T, h2::BlockTree& B) {
  double pts[20];
  std::iota(pts, pts + 20, 0.0);
  h2::build_cluster_tree(pts, 20, 1, 32, T);
  h2::build_block_tree(T, T, 2.0, B);
  h2::MatDesc d;
  d.rows = d.cols = &T;
  d.blocks = &B;
  d.k = 4;
  return d;
}
}  // namespace

// ranks of a product of H-matrix form, and whether its replays report
extern "C" int product_ranks(int* reports) {
  h2::Tree T;
  h2::BlockTree B;
  const h2::MatDesc d = one_leaf(T, B);
  h2::MulOptions o;
  o.hmatrix = true;
  const auto P = h2::make_product_plan(d, d, o);
  *reports = P->reports;
  return (int)P->rank_row_slot.size();
}
extern "C" int matvec_reports() {
  h2::Tree T;
  h2::BlockTree B;
  return h2::make_matvec_plan(one_leaf(T, B), 1)->reports;
}
