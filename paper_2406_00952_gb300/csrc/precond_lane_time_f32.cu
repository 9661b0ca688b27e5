// FP32 time pass with one line per lane (precond_lane.cuh).
#include "precond_lane.cuh"

namespace pcb {

namespace {
template <typename R>
int columns(int n, bool gz) {
  switch (n) {
#define PCB_COLUMNS(N) case N: return gz ? lane::time_lanes<R, N, true>() : lane::time_lanes<R, N, false>();
    PCB_COLUMNS(2) PCB_COLUMNS(4) PCB_COLUMNS(8) PCB_COLUMNS(16) PCB_COLUMNS(32) PCB_COLUMNS(64) PCB_COLUMNS(128)
    PCB_COLUMNS(256) PCB_COLUMNS(512) PCB_COLUMNS(1024)
#undef PCB_COLUMNS
    default: return 1;
  }
}
template <typename R>
int lines(int M) {
  switch (M) {
#define PCB_LINES(L) case L: return lane::spatial_lanes<R, L>();
    PCB_LINES(32) PCB_LINES(48) PCB_LINES(64) PCB_LINES(96) PCB_LINES(128) PCB_LINES(192) PCB_LINES(256) PCB_LINES(384)
    PCB_LINES(512) PCB_LINES(768) PCB_LINES(1024)
#undef PCB_LINES
    default: return 1;
  }
}
}  // namespace

// tile shapes for the launch counts: lines per spatial tile, columns per time tile, time tiles per block
int lane_space_lines(int M, int p) { return p ? lines<float>(M) : lines<double>(M); }
int lane_time_columns(int n, bool gz, int p) { return p ? columns<float>(n, gz) : columns<double>(n, gz); }
int lane_time_tiles(int n, int p) { return n <= (p ? 16 : 4) ? 4 : 1; }

cudaError_t lane_time_f32(const Batch& B, Sel sel, int n, bool gz, int kind, int in_sel, int out_sel) {
  switch (n) {
    case 2: return gz ? lane::time_pass_n<float, 2, true>(B, sel, kind, in_sel, out_sel)
                  : lane::time_pass_n<float, 2, false>(B, sel, kind, in_sel, out_sel);
    case 4: return gz ? lane::time_pass_n<float, 4, true>(B, sel, kind, in_sel, out_sel)
                  : lane::time_pass_n<float, 4, false>(B, sel, kind, in_sel, out_sel);
    case 8: return gz ? lane::time_pass_n<float, 8, true>(B, sel, kind, in_sel, out_sel)
                  : lane::time_pass_n<float, 8, false>(B, sel, kind, in_sel, out_sel);
    case 16: return gz ? lane::time_pass_n<float, 16, true>(B, sel, kind, in_sel, out_sel)
                  : lane::time_pass_n<float, 16, false>(B, sel, kind, in_sel, out_sel);
    case 32: return gz ? lane::time_pass_n<float, 32, true>(B, sel, kind, in_sel, out_sel)
                  : lane::time_pass_n<float, 32, false>(B, sel, kind, in_sel, out_sel);
    case 64: return gz ? lane::time_pass_n<float, 64, true>(B, sel, kind, in_sel, out_sel)
                  : lane::time_pass_n<float, 64, false>(B, sel, kind, in_sel, out_sel);
    case 128: return gz ? lane::time_pass_n<float, 128, true>(B, sel, kind, in_sel, out_sel)
                  : lane::time_pass_n<float, 128, false>(B, sel, kind, in_sel, out_sel);
    case 256: return gz ? lane::time_pass_n<float, 256, true>(B, sel, kind, in_sel, out_sel)
                  : lane::time_pass_n<float, 256, false>(B, sel, kind, in_sel, out_sel);
    case 512: return gz ? lane::time_pass_n<float, 512, true>(B, sel, kind, in_sel, out_sel)
                  : lane::time_pass_n<float, 512, false>(B, sel, kind, in_sel, out_sel);
    case 1024: return gz ? lane::time_pass_n<float, 1024, true>(B, sel, kind, in_sel, out_sel)
                  : lane::time_pass_n<float, 1024, false>(B, sel, kind, in_sel, out_sel);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace pcb
