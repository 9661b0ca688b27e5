// FP64 spatial passes along the rows of a slice with a transposed result (precond_lane.cuh): passes 2
// and 5.
#include "precond_lane.cuh"

namespace pcb {
namespace {
template <int M, bool EV>
struct Cols {
  static cudaError_t run(const Batch& B, Sel sel, int stage, int in_sel, int out_sel) {
    return lane::cols_pass<double, M, EV, false>(B, sel, in_sel, out_sel, stage >= 4);
  }
};

}  // namespace

cudaError_t lane_cols_f64(const Batch& B, Sel sel, int M, bool ev, int stage, int in_sel, int out_sel) {
  return ev ? lane::by_length<true, Cols>(M, B, sel, stage, in_sel, out_sel)
            : lane::by_length<false, Cols>(M, B, sel, stage, in_sel, out_sel);
}

}  // namespace pcb
