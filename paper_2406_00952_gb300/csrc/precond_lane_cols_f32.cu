// FP32 spatial passes along the rows of a slice with a transposed result (precond_lane.cuh): pass 2 stays
// in the FP32 scratch, pass 5 writes the FP64 output.
#include "precond_lane.cuh"

namespace pcb {
namespace {
template <int M, bool EV>
struct Cols {
  static cudaError_t run(const Batch& B, Sel sel, int stage, int in_sel, int out_sel) {
    if constexpr (!EV)      // MINRES runs on Dirichlet grids
      if (stage == 5 && B.fuse_z) return lane::cols_pass<float, M, false, true, true>(B, sel, in_sel, out_sel, 1);
    return stage == 2 ? lane::cols_pass<float, M, EV, false>(B, sel, in_sel, out_sel, 0)
                      : lane::cols_pass<float, M, EV, true>(B, sel, in_sel, out_sel, 1);
  }
};
template <int M, bool EV>
struct Dot {
  static cudaError_t run(const Batch& B, Sel sel, int sy, int sz) {
    if constexpr (EV) return cudaErrorInvalidValue;
    else lane::k_lane_dot<M><<<B.tot_ls[1], lane::spatial_threads<float, M>(), 0, B.stream>>>(
        B.G, (const Slots*)B.S, B.off_ls[1], B.count, sel, sy, sz, B.partial);
    return cudaGetLastError();
  }
};

}  // namespace

cudaError_t lane_dot_f32(const Batch& B, Sel sel, int M, int sy, int sz) {
  return lane::by_length<false, Dot>(M, B, sel, sy, sz);
}

cudaError_t lane_cols_f32(const Batch& B, Sel sel, int M, bool ev, int stage, int in_sel, int out_sel) {
  return ev ? lane::by_length<true, Cols>(M, B, sel, stage, in_sel, out_sel)
            : lane::by_length<false, Cols>(M, B, sel, stage, in_sel, out_sel);
}

}  // namespace pcb
