// drt_k_batch_redo.cu -- the redo at the end of a batch wave: each queued path-step recomputed in two-float
// numbers (or FP64) and its contribution added to H.  Compiled twice: values only, and (drt_k_batch_redo_dual.cu,
// DRT_BATCH_REDO_DUAL) with the rates the Doppler output needs.
#include "drt_batch.cuh"
#include "drt_physics_ff.cuh"

namespace drt {

// The lanes' steps (link li, path p, step ti; `on`: the lane has one) recomputed, then added to H by the whole warp, one after
// another: lane l takes the bins l, l + 32, .. (with a lane per step, 32 rows were written at once and the lanes without a step
// idled through it).  second: the step's carrier partner instead, where it shares the geometry.
template <bool DUAL>
__device__ void redo_add_warp(const BatchDev &B, int4 itm, bool on, bool second) {
    int li = itm.x;
    if (second) {
        li = on ? B.links[itm.x].partner : -1;
        on = on && li >= 0 && itm.y >= B.links[itm.x].pair_p0;
    }
    double r[3] = {0.0, 0.0, 0.0};
    if (on) {
        const BatchLink &BL = B.links[li];
        path_step_redo<DUAL>(BL.L, BL.tg, BL.fg, itm.y, itm.z, BL.out, BL.warm, r, BL.two != 0);
    }
    __syncwarp();
    const int lane = threadIdx.x;
    for (unsigned left = __ballot_sync(0xffffffffu, r[0] != 0.0 || r[1] != 0.0); left; left &= left - 1) {
        const int l = __ffs(left) - 1;
        const float ar = (float)__shfl_sync(0xffffffffu, r[0], l), ai = (float)__shfl_sync(0xffffffffu, r[1], l);
        const double tau = __shfl_sync(0xffffffffu, r[2], l);
        const int step = __shfl_sync(0xffffffffu, itm.z, l);
        const BatchLink &BL = B.links[__shfl_sync(0xffffffffu, li, l)];
        // a exp(-j 2 pi f_k tau): FP64-reduced seed at the lane's bin of every 512, between them at most 15 FP32 rotations by 32 bins
        // (each adds the rounding of its angle: one seed for 4096 bins was 2e-5 off at the last ones)
        const double f0 = BL.fg.f0, df = BL.fg.df, xs = 32 * df * tau;
        const int F = BL.fg.n_bins;
        float2 *row = BL.H + (size_t)step * F;
        float ws, wc;
        sincospif(2.f * (float)(xs - floor(xs)), &ws, &wc);
        for (int k0 = lane; k0 < F; k0 += 512) {
            const double x = (f0 + k0 * df) * tau;
            float sn, cs;
            sincospif(2.f * (float)(x - floor(x)), &sn, &cs);
            float zr = fmaf(ar, cs, ai * sn), zi = fmaf(ai, cs, -ar * sn);
            for (int k = k0; k < F && k < k0 + 512; k += 32) {
                atomicAdd(row + k, make_float2(zr, zi));
                const float nr = fmaf(zr, wc, zi * ws);
                zi = fmaf(zi, wc, -zr * ws);
                zr = nr;
            }
        }
    }
}

template <bool DUAL>
__global__ void __launch_bounds__(32) k_batch_redo(const BatchDev B) {   // one warp per block, spread over SMs
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {   // the run's total; a wave whose count exceeds the list
        unsigned long long *hdr = reinterpret_cast<unsigned long long *>(B.redo.count);   // marks the run
        atomicAdd(hdr + 1, (unsigned long long)*B.redo.count);
        if (*B.redo.count > B.redo.cap) atomicOr(hdr + 2, 1ull);
    }
    // Grid row y takes the chains of y vertices, so that warps that run at the same time run the same code.  Few queued steps: a run
    // (steps of one path, see for_redo_runs) per warp, the shortest latency.  Many: 32 list places per warp, whose chains'
    // branches run in turn but which keep the lanes filled (126 000 steps of a 128-link batch: 0.8 ms against 1.4 ms by runs).
    const int count = *B.redo.count, n = count < B.redo.cap ? count : B.redo.cap, lane = threadIdx.x, y = blockIdx.y;
    const bool packed = n > 64 * (int)gridDim.x;
    const int stride = packed ? 32 * (int)gridDim.x : redo_stride(gridDim.x), first = (packed ? 32 : 1) * (int)blockIdx.x;
    for (int k = first < stride ? first : n; k < n; k += stride) {
        int4 itm = make_int4(-1, 0, 0, 0);
        bool on = k + lane < n;
        if (!packed) {
            const int run = B.redo.items[k].w;
            if (run & 255) continue;   // inside another's run
            on = on && lane < (run >> 8);
        }
        if (on) itm = B.redo.items[k + lane];
        on = on && chain_length(B.links[itm.x].L, itm.y) == y;
        if (!__any_sync(0xffffffffu, on)) continue;
        redo_add_warp<DUAL>(B, itm, on, false);
        if (__any_sync(0xffffffffu, on && B.links[itm.x].partner >= 0)) redo_add_warp<DUAL>(B, itm, on, true);
    }
}

#ifdef DRT_BATCH_REDO_DUAL
cudaError_t launch_batch_redo_dual(const BatchDev &B, int grid, cudaStream_t s) {
    k_batch_redo<true><<<dim3(grid, MAXI + 1), 32, 0, s>>>(B);
    return cudaGetLastError();
}
#else
cudaError_t launch_batch_redo_dual(const BatchDev &B, int grid, cudaStream_t s);

// dual: some entry asks for the Doppler shift (the redo then carries rates)
cudaError_t launch_batch_redo(bool dual, const BatchDev &B, int grid, cudaStream_t s) {
    if (dual) return launch_batch_redo_dual(B, grid, s);
    k_batch_redo<false><<<dim3(grid, MAXI + 1), 32, 0, s>>>(B);
    return cudaGetLastError();
}
#endif

}  // namespace drt
