// eval_slice_d1.cu -- the bit-sliced evaluator for depth 1 (a unit of its own so that
// the instances compile side by side).
#include "eval_slice.cuh"

namespace deoct {
namespace slc {

int launch_slice_1(deoct_ctx* ctx, int nd, const SliceArgs& sa, bool raw, int grid, cudaStream_t s) {
  return launch_slice_d<1>(ctx, nd, sa, raw, grid, s);
}

}  // namespace slc
}  // namespace deoct
