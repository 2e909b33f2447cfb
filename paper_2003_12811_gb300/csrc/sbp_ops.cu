// The kernels of one precision (SBP_T) and order (SBP_O): compiled once for each pair, side by side, with the same
// result in every build (nvcc's own parallel compilation, --split-compile, cuts the device code differently from
// run to run: k_strip_tile<float, 6> then had 448 bytes of spill loads in one build and 648 in the next).
#include "sbp_launch.cuh"

namespace sbphost {

template int launch_operator<SBP_T, SBP_O>(sbp_handle*, const StepArgs&, int, cudaStream_t, bool);
template int launch_wide<SBP_T, SBP_O>(sbp_handle*, const StepArgs&, int, cudaStream_t);
template void layer_launch<SBP_T, SBP_O>(sbp_handle*, const StepArgs&, int, cudaStream_t, bool);
template void set_smem_attr<SBP_T, SBP_O>();
template void launch_noalloc<SBP_T, SBP_O>(sbp_handle*, const BlockDev*, int, BlockDev*, FaceRef*, const StepArgs&, cudaStream_t);
template void launch_grad<SBP_T, SBP_O>(sbp_handle*, const GradDev*, const std::vector<GradDev>&, int, double, cudaStream_t);
#ifdef SBP_BATCH
template int batch_ctas_per_sm<SBP_O>();
template void batch_step_launch<SBP_O>(int, BatchHead*, int*, cudaStream_t);
#endif

}  // namespace sbphost
