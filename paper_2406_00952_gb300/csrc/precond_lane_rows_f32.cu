// FP32 spatial passes across the rows of a slice (precond_lane.cuh): pass 1 reads the FP64 input, pass 4
// works in place on the FP32 scratch.
#include "precond_lane.cuh"

namespace pcb {
namespace {
template <int M, bool EV>
struct Rows {
  static cudaError_t run(const Batch& B, Sel sel, int stage, int in_sel, int out_sel) {
    if constexpr (!EV)      // MINRES runs on Dirichlet grids
      if (stage == 1 && B.fuse_z) return lane::rows_pass<float, M, false, true, true>(B, sel, in_sel, out_sel, 0);
    return stage == 1 ? lane::rows_pass<float, M, EV, true>(B, sel, in_sel, out_sel, 0)
                      : lane::rows_pass<float, M, EV, false>(B, sel, in_sel, out_sel, 1);
  }
};

}  // namespace

cudaError_t lane_rows_f32(const Batch& B, Sel sel, int M, bool ev, int stage, int in_sel, int out_sel) {
  return ev ? lane::by_length<true, Rows>(M, B, sel, stage, in_sel, out_sel)
            : lane::by_length<false, Rows>(M, B, sel, stage, in_sel, out_sel);
}

}  // namespace pcb
