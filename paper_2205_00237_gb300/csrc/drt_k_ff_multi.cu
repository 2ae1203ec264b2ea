// drt_k_ff_multi.cu -- the two-float records of the chains with several diffractions in a segment (Newton from the warm starts) and
// of the 4-vertex chains, one launch per length.
#include "drt_launch.cuh"
#include "drt_physics_ff.cuh"

namespace drt {

cudaError_t launch_extrapolate_ff_generic(const LinkDev &L, const TimeGridD &tg, const FreqGridD &fg, const void *mem,
                                          const RecD &rec, const double *warm, cudaStream_t s) {
    const PoseQ *pose = reinterpret_cast<const PoseQ *>(mem);
    const PointQ *term = reinterpret_cast<const PointQ *>(pose + (size_t)L.n_bodies * tg.n_steps);
    if (tg.n_steps == 0) return cudaSuccess;
    return for_generic_ranges(L, 0, L.n_paths, true, [&](int kind, int a, int b) {
            if (kind == 2) run_extrapolate_ff<2, true>(L, tg, fg, pose, term, rec, a, b, warm, s);
        else if (kind == 3) run_extrapolate_ff<3, true>(L, tg, fg, pose, term, rec, a, b, warm, s);
        else run_extrapolate_ff<4, true>(L, tg, fg, pose, term, rec, a, b, warm, s);
        return cudaGetLastError();
    });
}

}  // namespace drt
