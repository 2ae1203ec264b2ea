// drt_k_redo_out.cu -- the redo (two-float numbers, or FP64) of the FP32-bulk path-steps that FP32 cannot resolve, written in
// place into the caller's per-path-step outputs and records.
#include "drt_launch.cuh"
#include "drt_physics_ff.cuh"

namespace drt {

// redo of the queued path-steps: a fixed grid strides over the device-side count, one warp per block (see for_redo_runs)
template <bool DUAL>
__global__ void __launch_bounds__(32)
k_redo(const __grid_constant__ LinkDev L, const __grid_constant__ TimeGridD tg, const __grid_constant__ FreqGridD fg,
       const OutD out, const RedoList redo, const double *__restrict__ warm, bool two) {
    for_redo_runs(redo, blockIdx.x, gridDim.x, threadIdx.x, [&](int, int4 it) {
        path_step_redo<DUAL>(L, tg, fg, it.y, it.z, out, warm, nullptr, two);
    });
}

#ifdef DRT_REDO_DUAL   // drt_k_redo_out_dual.cu: with the rates the Doppler output needs
cudaError_t launch_redo_dual(const LinkDev &L, const TimeGridD &tg, const FreqGridD &fg, const OutD &out, void *redo,
                             const double *warm, cudaStream_t s, bool two) {
    k_redo<true><<<152 * 16, 32, 0, s>>>(L, tg, fg, out, redo_list(redo, L, tg), warm, two);
    return cudaGetLastError();
}
#else
cudaError_t launch_redo_dual(const LinkDev &L, const TimeGridD &tg, const FreqGridD &fg, const OutD &out, void *redo,
                             const double *warm, cudaStream_t s, bool two);

cudaError_t launch_redo(const LinkDev &L, const TimeGridD &tg, const FreqGridD &fg, const OutD &out, void *redo,
                        const double *warm, cudaStream_t s, bool two) {
    if (L.n_paths == 0 || tg.n_steps == 0) return cudaSuccess;
    if (out.doppler) return launch_redo_dual(L, tg, fg, out, redo, warm, s, two);
    k_redo<false><<<152 * 16, 32, 0, s>>>(L, tg, fg, out, redo_list(redo, L, tg), warm, two);
    return cudaGetLastError();
}
#endif

}  // namespace drt
