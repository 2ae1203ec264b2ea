// drt_physics_ff.cuh -- one (path, time-step) of the FP64 form's H synthesis in two-float numbers (drt_ff.cuh).
//
// The records that the synthesis reads are FP32 (amplitude, phase seed and phase step in turns), so the geometry only has to
// carry the path length to ~1e-10 m and the decisions exactly.  Two-float arithmetic does the first with 47 bits; a step that it
// cannot decide (a validity margin within 2^-36 of the coordinates, a virtual terminal on an edge line, a boundary of the
// transition function, a Newton solve that did not converge, anything not finite) is computed in FP64 by the lane that met it.
#pragma once
#include "drt_launch.cuh"

namespace drt {

// per (body, step): rotation rows and rotation centre; per (terminal, step): position
struct PoseQ { ff R[9], O[3]; };      // 96 B
struct PointQ { ff r[3], pad; };      // 32 B

DRT_HD v3<ff> vq(const ff *a) { return V3<ff>(a[0], a[1], a[2]); }
DRT_NOINL1 v3<ff> rotq(const PoseQ &P, v3<ff> x) {
    return V3<ff>(dot(vq(P.R), x), dot(vq(P.R + 3), x), dot(vq(P.R + 6), x));
}

// the rotation by theta(t) = w0 t + wdot t^2 / 2 about k (Rodrigues) and O(t) = o + v t + a t^2 / 2
DRT_HD void body_pose_ff(const BodyQ &B, ff t, PoseQ &q) {
    const ff t2 = halve(t * t);
    ff th = fma(B.w0, t, B.wdot * t2);
    // whole turns off: n (2 pi) in three parts
    const float n = rintf(th.h * 0.15915494309189535f);
    const ff p = ff(2 * PI) * n;
    th = (th - p) - ff(n * -6.860498e-15f);   // 2 pi less its two-float constant
    ff s, c;
    sincos_ff(th, s, c);
    const ff C1 = ff(1.f) - c, kx = B.k[0], ky = B.k[1], kz = B.k[2];
    const ff xy = kx * ky * C1, xz = kx * kz * C1, yz = ky * kz * C1;
    q.R[0] = fma(kx * kx, C1, c);
    q.R[1] = xy - kz * s;
    q.R[2] = xz + ky * s;
    q.R[3] = xy + kz * s;
    q.R[4] = fma(ky * ky, C1, c);
    q.R[5] = yz - kx * s;
    q.R[6] = xz - ky * s;
    q.R[7] = yz + kx * s;
    q.R[8] = fma(kz * kz, C1, c);
    for (int j = 0; j < 3; ++j) q.O[j] = fma(B.a[j], t2, fma(B.v[j], t, B.o[j]));
}

DRT_HD Prim<ff> load_prim_ff(const LinkDev &L, const PoseQ *pose, int n_steps, int ti, int type, int idx) {
    Prim<ff> q;
    q.type = type;
    q.idx = idx;
    int body;
    if (type == T_R) {
        const FaceQ &f = L.facesQ[idx];
        q.p = vq(f.c);
        q.a = vq(f.n);
        q.b = vq(f.u);
        q.h1 = f.hu;
        q.h2 = f.hw;
        q.mat = f.mat;
        body = f.body;
    } else if (type == T_D) {
        const EdgeQ &e = L.edgesQ[idx];
        q.p = vq(e.a);
        q.a = vq(e.e);
        q.b = vq(e.t0);
        q.c = vq(e.n0);
        q.h1 = e.len;
        q.h2 = e.wn;
        q.h3 = e.snp;
        q.h4 = e.cnp;
        q.mat = e.mat;
        body = e.body;
    } else {
        const TileQ &tl = L.tilesQ[idx];
        q.p = vq(tl.c);
        q.a = vq(tl.n);
        q.mat = tl.mat;
        body = tl.body;
    }
    if (body >= 0) {
        const PoseQ &P = pose[(size_t)body * n_steps + ti];
        q.p = vq(P.O) + rotq(P, q.p);
        q.a = rotq(P, q.a);
        if (type != T_S) q.b = rotq(P, q.b);
        if (type == T_D) q.c = rotq(P, q.c);
    }
    return q;
}

// amplitude 0 and all-zero phases for a path that does not exist; phases in turns from the path length d
DRT_HD void write_record_ff(const RecD &r, size_t ri, const FreqGridD &fg, ff d, cx<ff> a) {
    const ff x = d * fg.f0c_q, y = d * fg.dfc_q;
    float ph = (x.h - floorf(x.h)) + x.l;      // the leading part's fraction is exact
    const float st = y.h - floorf(y.h);
    const float hi = rintf((st + y.l) * 4096.f) * (1.f / 4096.f);   // 12 leading bits, so that k hi is exact
    r.rec_a[ri] = make_float4(a.re.h, a.im.h, ph, hi);
    r.rec_b[ri] = (st - hi) + y.l;
}

// the FP64 step for what two-float numbers cannot decide (out of line: rare)
template <int N, bool MULTI>
DRT_NOINL void path_step_ff_fallback(const LinkDev &L, const TimeGridD &tg, const FreqGridD &fg, int p, int ti,
                                     const RecD &rec, const double *warm) {
    const double t = tg.t_start + ti * tg.dt;
    const OutD none{};
    path_step_fp64_core<N, MULTI, false, double>(
        L, tg, fg, p, ti, none, rec, false,
        [&](int ty, int idx) { return val_prim(load_prim_direct<double>(L, t, ty, idx)); }, warm);
}

// Instruction fetch bounds this form as much as issue: a step is ~6000 instructions, and inlined at every vertex they gave 7 to 11
// no-instruction stalls per issue (28 % of the issue slots used).  With the arithmetic's helpers out of line (one copy each) and
// neighbouring blocks on neighbouring paths it is 2 to 3 (48 %).  Measured and left out: a barrier per stage, in blocks of 128 or one
// of 384 threads per SM (1.0 stalls, but the same or a longer time); an order that gives each SM its own stretch of paths (25 to
// 50 % slower: the SMs share instruction-cache lines).
template <int N>
DRT_HD cx<ff> amplitude_ff(const LinkDev &L, const Prim<ff> *pr, const v3<ff> *seg, const FreqGridD &fg) {
    v3<ff> kd[N + 2];
    ff Lfac[N + 1], sp_num, sp_den;
    field_spread<N>(pr, N, seg, kd, Lfac, sp_num, sp_den);
    const FieldK<ff> fk = field_k<ff>(fg);
    c3<ff> E = cscale(vertical_pol(kd[1]), C<ff>(ff(1.f), ff(0.f)));
#pragma unroll
    for (int i = 1; i <= N; ++i) {
        const Prim<ff> &q = pr[i - 1];
        const v3<ff> kin = kd[i], kout = kd[i + 1];
        if (q.type == T_R) {
            E = refl_field_out(E, kin, kout, q.a, matv<ff>(L.mats[q.mat]), fk.ieps);
        } else if (q.type == T_D) {
            E = diff_field_out(E, kin, kout, q.a, q.b, q.c, q.h2, q.h3, q.h4, Lfac[i], fk.k, fk.isk,
                               matv<ff>(L.mats[q.mat]), fk.ieps);
        } else {
            E = tile_field_out(E, kin, kout, q.a, tilev<ff>(L, q.idx));
        }
    }
    return cdot(E, vertical_pol(kd[N + 1])) * (fk.lam * sqrt(sp_num / sp_den));
}

template <int N, bool MULTI>
DRT_HD void path_step_ff(const LinkDev &L, const TimeGridD &tg, const FreqGridD &fg, const PoseQ *pose,
                         const PointQ *term, int p, int ti, const RecD &rec, const double *warm) {
    const uint32_t code = L.ptypes[p];
    const int4 pi = L.pprims[p];
    const int prim[MAXI] = {pi.x, pi.y, pi.z, pi.w};
    const size_t ri = (size_t)ti * L.n_paths + p;
    Prim<ff> pr[N > 0 ? N : 1];
#pragma unroll
    for (int j = 0; j < N; ++j) pr[j] = load_prim_ff(L, pose, tg.n_steps, ti, (code >> (8 * j)) & 0xff, prim[j]);
    v3<ff> V[N + 2];
    V[0] = vq(term[ti].r);
    V[N + 1] = vq(term[tg.n_steps + ti].r);
    uint32_t fl = 0;
    if (MULTI && p >= L.n_bulk) {
        WarmStart32 ws;
        warm_start_at32(L, tg, warm, p, ti, ws);
        solve_geometry<N, MULTI>(pr, V, ws.s, fl, ws.ds, ws.rate);
    } else {
        solve_geometry<N, MULTI>(pr, V, L.ps0 + (size_t)p * MAXI, fl);
    }
    v3<ff> seg[N + 2];
    ff d = ff(0.f);
#pragma unroll
    for (int i = 1; i <= N + 1; ++i) {
        seg[i] = V[i] - V[i - 1];
        d = d + norm(seg[i]);
    }
    fl |= validity<N>(pr, N, V);
    bool sure = !(fl & (F_REDO64 | F_NOCONV | F_DEGEN)) && isfinite(d.h);
    if (sure && !fl) {
        const cx<ff> a = amplitude_ff<N>(L, pr, seg, fg);
        sure = isfinite(a.re.h) && isfinite(a.im.h);
        if (sure) write_record_ff(rec, ri, fg, d, a);
    } else if (sure) {   // an invalid path-step contributes nothing
        rec.rec_a[ri] = make_float4(0.f, 0.f, 0.f, 0.f);
        rec.rec_b[ri] = 0.f;
    }
    if (!sure) path_step_ff_fallback<N, MULTI>(L, tg, fg, p, ti, rec, warm);
}

// A block covers consecutive (path, 32 steps) warps in path-major order, so neighbouring blocks, which run at the same time, are
// on paths of the same signature
template <int N, bool MULTI> struct FFBlock { static constexpr int v = 128, per_sm = N <= 1 ? 5 : N == 2 && !MULTI ? 4 : 3; };
template <int N, bool MULTI> unsigned ff_grid(const TimeGridD &tg, int paths) {
    const unsigned warps = (unsigned)paths * ((tg.n_steps + 31) / 32), per = FFBlock<N, MULTI>::v / 32;
    return (warps + per - 1) / per;
}
template <int N, bool MULTI>
__global__ void __launch_bounds__(FFBlock<N, MULTI>::v, FFBlock<N, MULTI>::per_sm)
k_extrapolate_ff(const __grid_constant__ LinkDev L, const __grid_constant__ TimeGridD tg,
                 const __grid_constant__ FreqGridD fg, const PoseQ *__restrict__ pose, const PointQ *__restrict__ term,
                 const RecD rec, int p0, int p1, const double *__restrict__ warm) {
    const unsigned w = blockIdx.x * (FFBlock<N, MULTI>::v / 32) + threadIdx.x / 32, nt = (tg.n_steps + 31) / 32;
    const int p = p0 + (int)(w / nt), ti = (int)(w % nt) * 32 + (threadIdx.x & 31);
    if (p >= p1 || ti >= tg.n_steps) return;
    path_step_ff<N, MULTI>(L, tg, fg, pose, term, p, ti, rec, warm);
}

template <int N, bool MULTI>
void run_extrapolate_ff(const LinkDev &L, const TimeGridD &tg, const FreqGridD &fg, const PoseQ *pose, const PointQ *term,
                        const RecD &rec, int p0, int p1, const double *warm, cudaStream_t s) {
    k_extrapolate_ff<N, MULTI><<<ff_grid<N, MULTI>(tg, p1 - p0), FFBlock<N, MULTI>::v, 0, s>>>(L, tg, fg, pose, term, rec,
                                                                                              p0, p1, warm);
}

}  // namespace drt
