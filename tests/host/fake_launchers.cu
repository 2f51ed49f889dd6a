// The kernel launchers that csrc/api.cu calls, without kernels: each counts a launch with the fake runtime.
#include "../../paper_2309_08068_gb300/csrc/lbm_internal.cuh"

extern "C" int fake_launched(cudaStream_t s, int kind);  // kind 0 single step, 1 ring, 2 tiled, 3 line, -1 other
static int launched(cudaStream_t s, int kind = -1) { return fake_launched(s, kind); }

namespace lbm {
int mm_launch_step(const StepArgs&, cudaStream_t s) { return launched(s, 0); }
int hv_launch_step(const StepArgs&, cudaStream_t s) { return launched(s, 0); }
int mm_launch_fused2(const StepArgs&, const StepArgs&, const FusedArgs&, cudaStream_t s) { return launched(s, 1); }
int hv_launch_fused2(const StepArgs&, const StepArgs&, const FusedArgs&, cudaStream_t s) { return launched(s, 1); }
int mm_launch_tile2(const StepArgs&, const StepArgs&, const TileArgs&, cudaStream_t s) { return launched(s, 2); }
int hv_launch_tile2(const StepArgs&, const StepArgs&, const TileArgs&, cudaStream_t s) { return launched(s, 2); }
int launch_line(bool, const LineArgs&, cudaStream_t s) { return launched(s, 3); }
int mm_launch_init(const StepArgs&, const float*, const float*, cudaStream_t s) { return launched(s); }
int hv_launch_init(const StepArgs&, const float*, const float*, cudaStream_t s) { return launched(s); }
int mm_launch_fields(const StepArgs&, FieldsOut, cudaStream_t s) { return launched(s); }
int hv_launch_fields(const StepArgs&, FieldsOut, cudaStream_t s) { return launched(s); }
int mm_launch_get(const StepArgs&, float*, cudaStream_t s) { return launched(s); }
int hv_launch_get(const StepArgs&, float*, cudaStream_t s) { return launched(s); }
int mm_launch_set(const StepArgs&, const float*, cudaStream_t s) { return launched(s); }
int hv_launch_set(const StepArgs&, const float*, cudaStream_t s) { return launched(s); }
int mm_launch_reduce(const StepArgs&, double*, int, double*, cudaStream_t s) { return launched(s); }
int hv_launch_reduce(const StepArgs&, double*, int, double*, cudaStream_t s) { return launched(s); }
int mm_launch_batch_step(const BatchLaunch&, int, int, int, cudaStream_t s) { return launched(s); }
int hv_launch_batch_step(const BatchLaunch&, int, int, int, cudaStream_t s) { return launched(s); }
int mm_launch_record_step(const StepArgs&, cudaStream_t s) { return launched(s); }
int hv_launch_record_step(const StepArgs&, cudaStream_t s) { return launched(s); }
int mm_launch_record_tile2(const StepArgs&, const StepArgs&, const TileArgs&, cudaStream_t s) { return launched(s); }
int mm_launch_adjoint(const AdjointArgs&, cudaStream_t s) { return launched(s); }
int hv_launch_adjoint(const AdjointArgs&, cudaStream_t s) { return launched(s); }
int mm_launch_adjoint_terminal(const AdjointArgs&, int, cudaStream_t s) { return launched(s); }
int hv_launch_adjoint_terminal(const AdjointArgs&, int, cudaStream_t s) { return launched(s); }
int mm_tile2_occupancy(int, int) { return 2; }
int hv_tile2_occupancy(int, int) { return 2; }
int mm_fused2_occupancy(int, int) { return 1; }
int hv_fused2_occupancy(int, int) { return 1; }
int mm_batch_occupancy(int, int, bool) { return 3; }
int hv_batch_occupancy(int, int) { return 4; }
int mm_halo_dirs(int, int* d) { d[0] = 0; return 1; }
int hv_halo_dirs(int, int* d) { d[0] = 0; return 1; }
}  // namespace lbm
