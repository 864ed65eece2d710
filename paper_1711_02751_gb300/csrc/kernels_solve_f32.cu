// The one-launch trace solve with FP32 cycles (the mixed form on the assembled trace matrix).
#include "kernels_solve.inl"

namespace hdgdg {

cudaError_t launch_solve_f32(int P, const SolveArgs& a, cudaStream_t s) { return solve_dispatch<float>(P, a, s); }

}  // namespace hdgdg
