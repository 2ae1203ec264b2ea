// drt_k_base.cu -- the FP32-bulk form's anchors, in two-float numbers or FP64: body poses at the chunk bases and, per (path,
// chunk), the path length, segment vectors and phase seeds the FP32 deltas build on.
#include "drt_launch.cuh"
#include "drt_physics_ff.cuh"

namespace drt {

// one block per path, one thread per chunk: lanes share the chain signature; body poses at the
// chunk bases come from an FP64 pose table [body][chunk] built first
constexpr int BASE_T = 64;
__global__ void __launch_bounds__(BASE_T)
k_base_fp64(const LinkDev L, const TimeGridD tg, const FreqGridD fg, const double *__restrict__ pose64,
            BaseRec *__restrict__ base, const double *__restrict__ warm, int p0) {
    int p = p0 + blockIdx.x;
    int c = blockIdx.y * BASE_T + threadIdx.x;
    if (p >= L.n_paths || c >= n_chunks_of(tg)) return;
    path_base_fp64(L, tg, fg, pose64, p, c, base, warm);
}

// the same in two-float numbers, on a table of PoseQ rows
__global__ void __launch_bounds__(BASE_T)
k_base_ff(const __grid_constant__ LinkDev L, const __grid_constant__ TimeGridD tg, const __grid_constant__ FreqGridD fg,
          const PoseQ *__restrict__ pose, BaseRec *__restrict__ base, const double *__restrict__ warm, int p0) {
    const int p = p0 + blockIdx.x;
    const int c = blockIdx.y * BASE_T + threadIdx.x;
    if (p >= L.n_paths || c >= n_chunks_of(tg)) return;
    path_base_ff(L, tg, fg, pose, p, c, base, warm);
}
__global__ void __launch_bounds__(BASE_T)
k_base_pose_ff(const BodyQ *__restrict__ bodies, int n_bodies, double t_start, double dt, int n_rows, PoseQ *__restrict__ pose) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_bodies * n_rows) return;
    body_pose_ff(bodies[i / n_rows], from_double(t_start + (i % n_rows) * dt), pose[i]);
}

cudaError_t launch_base_pose64(const LinkDev &L, const TimeGridD &tg, double *pose64, cudaStream_t s, bool two) {
    if (L.n_paths == 0 || tg.n_steps == 0) return cudaSuccess;
    TimeGridD tc = make_tgrid(tg.t_start, tg.dt * tg.chunk, n_chunks_of(tg), 1);   // chunk bases
    if (!two) return launch_pose(L, tc, pose64, s);
    static_assert(sizeof(PoseQ) <= POSE_W * sizeof(double), "the rows fit the FP64 table");
    k_base_pose_ff<<<(L.n_bodies * tc.n_steps + BASE_T - 1) / BASE_T, BASE_T, 0, s>>>(
        L.bodiesQ, L.n_bodies, tc.t_start, tc.dt, tc.n_steps, reinterpret_cast<PoseQ *>(pose64));
    return cudaGetLastError();
}

// anchors of paths [p0, p1); the multi-diffraction paths [n_bulk, n_paths) read the warm starts
cudaError_t launch_base_paths(const LinkDev &L, const TimeGridD &tg, const FreqGridD &fg, const double *pose64,
                              void *base, const double *warm, int p0, int p1, cudaStream_t s, bool two) {
    if (p1 <= p0 || tg.n_steps == 0) return cudaSuccess;
    dim3 grid(p1 - p0, (n_chunks_of(tg) + BASE_T - 1) / BASE_T);
    BaseRec *b = reinterpret_cast<BaseRec *>(base);
    if (two) k_base_ff<<<grid, BASE_T, 0, s>>>(L, tg, fg, reinterpret_cast<const PoseQ *>(pose64), b, warm, p0);
    else k_base_fp64<<<grid, BASE_T, 0, s>>>(L, tg, fg, pose64, b, warm, p0);
    return cudaGetLastError();
}

}  // namespace drt
