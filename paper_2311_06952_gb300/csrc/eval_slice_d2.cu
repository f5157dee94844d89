// eval_slice_d2.cu -- the bit-sliced evaluator for depth 2 (a unit of its own so that
// the instances compile side by side).
#include "eval_slice.cuh"

namespace deoct {
namespace slc {

int launch_slice_2(deoct_ctx* ctx, int nd, const SliceArgs& sa, bool raw, int grid, cudaStream_t s) {
  return launch_slice_d<2>(ctx, nd, sa, raw, grid, s);
}

}  // namespace slc
}  // namespace deoct
