// drt_k_batch_prep.cu -- stages 0-3 of a batch plan: FP32 base poses, FP64 chunk-base poses,
// multi-diffraction warm starts and FP64 chunk anchors, each a persistent launch over its
// (link, item) list.
#include "drt_batch.cuh"
#include "drt_physics_ff.cuh"

namespace drt {

// stages 0-3: block-wide claims of blockDim.x consecutive items.  TWO: stages 1-3 of the links that two-float numbers apply to (PoseQ
// rows), else of the others; a batch that has both runs both over all items, so that what a link gets does not depend on which
// others are in its batch.  The two-float anchors at 4 blocks per SM (128 registers; 0.65 -> 0.52 ms of a 128-link batch against
// 2 blocks without spills)
template <int STAGE, bool TWO>
__global__ void __launch_bounds__(128, TWO && STAGE == ST_BASE ? 4 : 1) k_stage(const BatchDev B) {
    __shared__ long long s_start;
    const long long total = B.n_items;
    for (;;) {
        if (threadIdx.x == 0) s_start = (long long)atomicAdd(B.counter, (unsigned long long)blockDim.x);
        __syncthreads();
        long long q = s_start + threadIdx.x;
        bool done = s_start >= total;
        __syncthreads();
        if (done) break;
        if (q >= total) continue;
        const long long it = B.it_base + q;
        int li = find_link(B, STAGE, it);
        const BatchLink &BL = B.links[li];
        if (STAGE != ST_POSEB && (BL.two != 0) != TWO) continue;
        long long local = it - BL.it0[STAGE];
        int nch = chunks_of(BL.tg);
        if (STAGE == ST_POSEB) {
            int b = (int)(local / nch), c = (int)(local - (long long)b * nch);
            double tb = BL.tg.t_start + (double)c * BL.tg.chunk * BL.tg.dt;
            if (b < BL.L.n_bodies) body_pose_base(BL.L.bodies[b], tb, BL.poseb[local]);
            else terminal_base(b == BL.L.n_bodies ? BL.L.tx : BL.L.rx, tb, BL.poseb[local]);
        } else if (STAGE == ST_POSE64) {
            int b = (int)(local / nch), c = (int)(local - (long long)b * nch);
            const double tb = BL.tg.t_start + (double)c * BL.tg.chunk * BL.tg.dt;
            if constexpr (TWO) body_pose_ff(BL.L.bodiesQ[b], from_double(tb), reinterpret_cast<PoseQ *>(BL.pose64)[local]);
            else body_pose_row(BL.L.bodies[b], tb, BL.pose64 + local * POSE_W);
        } else if (STAGE == ST_WARM) {   // rows 0..nch
            int p = BL.L.n_bulk + (int)(local / (nch + 1)), c = (int)(local % (nch + 1));
            if constexpr (TWO) path_warm_ff(BL.L, BL.tg, p, c, BL.warm);
            else path_warm_fp64(BL.L, BL.tg, p, c, BL.warm);
        } else {
            int p = (int)(local / nch), c = (int)(local % nch);
            if constexpr (TWO)
                path_base_ff(BL.L, BL.tg, BL.fg, reinterpret_cast<const PoseQ *>(BL.pose64), p, c, BL.base, BL.warm);
            else path_base_fp64(BL.L, BL.tg, BL.fg, BL.pose64, p, c, BL.base, BL.warm);
        }
    }
}

template <bool TWO> static void launch_stage(int stage, const BatchDev &B, int grid, cudaStream_t s) {
    switch (stage) {
    case ST_POSEB: k_stage<ST_POSEB, false><<<grid, 128, 0, s>>>(B); break;
    case ST_POSE64: k_stage<ST_POSE64, TWO><<<grid, 128, 0, s>>>(B); break;
    case ST_WARM: k_stage<ST_WARM, TWO><<<grid, 128, 0, s>>>(B); break;
    default: k_stage<ST_BASE, TWO><<<grid, 128, 0, s>>>(B); break;
    }
}
cudaError_t launch_batch_stage(int stage, bool two, const BatchDev &B, int grid, cudaStream_t s) {
    if (two) launch_stage<true>(stage, B, grid, s);
    else launch_stage<false>(stage, B, grid, s);
    return cudaGetLastError();
}

}  // namespace drt
