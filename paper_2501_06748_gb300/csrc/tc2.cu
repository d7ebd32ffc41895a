// The tensor-core element step for elements padded to 21..32 boundary nodes: every n_b x n_b
// operator in 4 x 2 tiles of 8 rows x 16 columns, every operand vector in two k-tiles.  A
// product sums, per 8 rows, the levels of both k-tiles before one recombination; the row
// exponents span all 32 rows, the column exponent all 32 entries of a shot, so the scaling
// (and the result) is that of one 32 x 32 product.
#include "tc_step.cuh"

namespace sbfwi {

int tc2_prepare(Model& md, cudaStream_t st) { return tc_prepare_tiles<2>(md, md.tc_ops, st); }

void tc2_element_launch(const ElemTcArgs& a, bool avg_accel, cudaStream_t st) {
  tc_launch_tiles<2>(a, avg_accel, st);
}

}  // namespace sbfwi
