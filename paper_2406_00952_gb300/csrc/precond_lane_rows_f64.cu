// FP64 spatial passes across the rows of a slice (precond_lane.cuh): passes 1 and 4.
#include "precond_lane.cuh"

namespace pcb {
namespace {
template <int M, bool EV>
struct Rows {
  static cudaError_t run(const Batch& B, Sel sel, int stage, int in_sel, int out_sel) {
    return lane::rows_pass<double, M, EV, false>(B, sel, in_sel, out_sel, stage >= 4);
  }
};

}  // namespace

cudaError_t lane_rows_f64(const Batch& B, Sel sel, int M, bool ev, int stage, int in_sel, int out_sel) {
  return ev ? lane::by_length<true, Rows>(M, B, sel, stage, in_sel, out_sel)
            : lane::by_length<false, Rows>(M, B, sel, stage, in_sel, out_sel);
}

}  // namespace pcb
