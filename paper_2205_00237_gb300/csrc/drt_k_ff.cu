// drt_k_ff.cu -- the synthesis records of the FP64 form in two-float numbers: poses per step and the extrapolation of the chains
// with at most one diffraction between point sources, one launch per length (block mapping of drt_k_fp64.cu).  The multi-diffraction
// and 4-vertex chains are in drt_k_ff_multi.cu.
#include "drt_launch.cuh"
#include "drt_physics_ff.cuh"

namespace drt {

// rows [body][step] of poses, then [terminal][step] of positions
__global__ void __launch_bounds__(128)
k_pose_ff(const BodyQ *__restrict__ bodies, int n_bodies, TermD tx, TermD rx, double t_start, double dt, int n_steps,
          PoseQ *__restrict__ pose, PointQ *__restrict__ term) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (n_bodies + 2) * n_steps) return;
    const int b = i / n_steps, ti = i - b * n_steps;
    const double t = t_start + ti * dt;
    if (b < n_bodies) {
        body_pose_ff(bodies[b], from_double(t), pose[i]);
    } else {
        const v3<double> r = val(terminal<double>(b == n_bodies ? tx : rx, t));
        term[i - n_bodies * n_steps] = PointQ{{from_double(r.x), from_double(r.y), from_double(r.z)}};
    }
}

size_t pose_ff_bytes(const LinkDev &L, const TimeGridD &tg) {
    return (size_t)tg.n_steps * (L.n_bodies * sizeof(PoseQ) + 2 * sizeof(PointQ));
}

cudaError_t launch_pose_ff(const LinkDev &L, const TimeGridD &tg, void *mem, cudaStream_t s) {
    const int n = (L.n_bodies + 2) * tg.n_steps;
    if (tg.n_steps == 0) return cudaSuccess;
    PoseQ *pose = reinterpret_cast<PoseQ *>(mem);
    k_pose_ff<<<(n + 127) / 128, 128, 0, s>>>(L.bodiesQ, L.n_bodies, L.tx, L.rx, tg.t_start, tg.dt, tg.n_steps, pose,
                                              reinterpret_cast<PointQ *>(pose + (size_t)L.n_bodies * tg.n_steps));
    return cudaGetLastError();
}

cudaError_t launch_extrapolate_ff(const LinkDev &L, const TimeGridD &tg, const FreqGridD &fg, const void *mem,
                                  const RecD &rec, int n, const double *warm, cudaStream_t s) {
    const PoseQ *pose = reinterpret_cast<const PoseQ *>(mem);
    const PointQ *term = reinterpret_cast<const PointQ *>(pose + (size_t)L.n_bodies * tg.n_steps);
    const int a = L.len_start[n], b = L.len_start[n + 1];
    if (b <= a || tg.n_steps == 0) return cudaSuccess;
    switch (n) {
    case 0: run_extrapolate_ff<0, false>(L, tg, fg, pose, term, rec, a, b, warm, s); break;
    case 1: run_extrapolate_ff<1, false>(L, tg, fg, pose, term, rec, a, b, warm, s); break;
    case 2: run_extrapolate_ff<2, false>(L, tg, fg, pose, term, rec, a, b, warm, s); break;
    default: run_extrapolate_ff<3, false>(L, tg, fg, pose, term, rec, a, b, warm, s); break;
    }
    return cudaGetLastError();
}

}  // namespace drt
