// The sweep kernels of bf16 tensors that keep the weights of every iteration (backward).
#define LOT_SWEEP_PART
#include "lot_sweep.cu"

namespace lot {
namespace sweep {

cudaError_t launch_keep(const SweepPlan &P, const SweepArgs &a, cudaStream_t st) { return launch_rp<__nv_bfloat16, true>(P, a, st); }

} // namespace sweep
} // namespace lot
