// The sweep kernels of bf16 tensors.
#define LOT_SWEEP_PART
#include "lot_sweep.cu"

namespace lot {
namespace sweep {

cudaError_t launch_bf16(const SweepPlan &P, const SweepArgs &a, cudaStream_t st) { return launch_rp<__nv_bfloat16, false>(P, a, st); }

} // namespace sweep
} // namespace lot
