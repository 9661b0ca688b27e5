// FP64 time pass with one line per lane (precond_lane.cuh).
#include "precond_lane.cuh"

namespace pcb {

cudaError_t lane_time_f64(const Batch& B, Sel sel, int n, bool gz, int kind, int in_sel, int out_sel) {
  switch (n) {
    case 2: return gz ? lane::time_pass_n<double, 2, true>(B, sel, kind, in_sel, out_sel)
                  : lane::time_pass_n<double, 2, false>(B, sel, kind, in_sel, out_sel);
    case 4: return gz ? lane::time_pass_n<double, 4, true>(B, sel, kind, in_sel, out_sel)
                  : lane::time_pass_n<double, 4, false>(B, sel, kind, in_sel, out_sel);
    case 8: return gz ? lane::time_pass_n<double, 8, true>(B, sel, kind, in_sel, out_sel)
                  : lane::time_pass_n<double, 8, false>(B, sel, kind, in_sel, out_sel);
    case 16: return gz ? lane::time_pass_n<double, 16, true>(B, sel, kind, in_sel, out_sel)
                  : lane::time_pass_n<double, 16, false>(B, sel, kind, in_sel, out_sel);
    case 32: return gz ? lane::time_pass_n<double, 32, true>(B, sel, kind, in_sel, out_sel)
                  : lane::time_pass_n<double, 32, false>(B, sel, kind, in_sel, out_sel);
    case 64: return gz ? lane::time_pass_n<double, 64, true>(B, sel, kind, in_sel, out_sel)
                  : lane::time_pass_n<double, 64, false>(B, sel, kind, in_sel, out_sel);
    case 128: return gz ? lane::time_pass_n<double, 128, true>(B, sel, kind, in_sel, out_sel)
                  : lane::time_pass_n<double, 128, false>(B, sel, kind, in_sel, out_sel);
    case 256: return gz ? lane::time_pass_n<double, 256, true>(B, sel, kind, in_sel, out_sel)
                  : lane::time_pass_n<double, 256, false>(B, sel, kind, in_sel, out_sel);
    case 512: return gz ? lane::time_pass_n<double, 512, true>(B, sel, kind, in_sel, out_sel)
                  : lane::time_pass_n<double, 512, false>(B, sel, kind, in_sel, out_sel);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace pcb
