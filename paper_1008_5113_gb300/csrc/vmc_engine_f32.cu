// vmc_engine_f32.cu -- the engine's kernels and launchers in the FP32 working precision.
// Compiled once per VMC_PART (build.py), so that the kernels compile in parallel.
#include "vmc_engine_impl.cuh"

namespace vmc {

#if VMC_PART == 0
template int kernel_static_smem_T<float>();
template cudaError_t launch_ratio_T<float>(const LaunchCfg&, const Walker*, int, const Params&, int, const double*,
                                         int);
template cudaError_t launch_accept_T<float>(const LaunchCfg&, const Walker*, int, const Params&);
#elif VMC_PART == 1
template cudaError_t launch_sweep_T<float>(const LaunchCfg&, const Walker*, int, int, const Params&, int, long long,
                                         double, const uint64_t*, uint8_t*, double*);
#elif VMC_PART == 2
template cudaError_t launch_sweep_pair_T<float, 1>(const LaunchCfg&, const Walker*, int, int, const Params&, int,
                                              long long, double, const uint64_t*, uint8_t*, double*, int);
#elif VMC_PART == 6
template cudaError_t launch_sweep_pair_T<float, 2>(const LaunchCfg&, const Walker*, int, int, const Params&, int,
                                              long long, double, const uint64_t*, uint8_t*, double*, int);
#elif VMC_PART == 3
template cudaError_t prepare_step_kernels_T<float>(const LaunchCfg&);
template cudaError_t launch_step_T<float>(const LaunchCfg&, const Walker*, int, int, const Params&, int, int, int,
                                        long long, double, const uint64_t*, uint8_t*, double*, const long long*);
#elif VMC_PART == 4
template cudaError_t launch_kinetic_T<float>(const LaunchCfg&, const Walker*, int, const Params&, double*);
#elif VMC_PART == 5
template cudaError_t launch_setup_T<float>(const LaunchCfg&, const Walker*, int, int, const Params&);
template cudaError_t launch_refactor_T<float>(const LaunchCfg&, const Walker*, int, const Params&, int);
template cudaError_t launch_apply_precond_T<float>(const LaunchCfg&, const Walker*, int, const Params&);
template cudaError_t launch_bench_T<float>(const LaunchCfg&, const Walker*, int, const Params&, int, int);
#endif

}  // namespace vmc
