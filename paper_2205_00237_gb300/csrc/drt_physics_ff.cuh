// drt_physics_ff.cuh -- one (path, time-step) of the FP64 form's H synthesis in two-float numbers (drt_ff.cuh).
//
// The records that the synthesis reads are FP32 (amplitude, phase seed and phase step in turns), so the geometry only has to
// carry the path length to ~1e-10 m and the decisions exactly.  Two-float arithmetic does the first with 47 bits; a step that it
// cannot decide (a validity margin within 2^-36 of the coordinates, more near grazing, a virtual terminal on an edge line, a boundary
// of the transition function, a Newton solve that did not converge, anything not finite) is computed in FP64 by the lane that met it.
// Canyon call (512 paths x 2000 steps x 512 bins) 1.93 -> 0.54 ms against the FP64 kernels, 3 paths x 1000 steps 54 -> 33 us.
#pragma once
#include "drt_launch.cuh"

namespace drt {

// per (body, step): rotation rows and rotation centre; per (terminal, step): position
struct PoseQ { ff R[9], O[3]; };      // 96 B
struct PointQ { ff r[3]; };           // 24 B: with it a row is no larger than the FP64 table's

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

// the primitive as stored: placed in the world when its body is at rest (returns -1), else relative to the rotation centre of
// the body returned
DRT_HD int load_prim_rest(const LinkDev &L, int type, int idx, Prim<ff> &q) {
    q.type = type;
    q.idx = idx;
    if (type == T_R) {
        const FaceQ &f = L.facesQ[idx];
        q.p = vq(f.c);
        q.a = vq(f.n);
        q.b = vq(f.u);
        q.h1 = f.hu;
        q.h2 = f.hw;
        q.mat = f.mat;
        return f.body;
    }
    if (type == T_D) {
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
        return e.body;
    }
    const TileQ &tl = L.tilesQ[idx];
    q.p = vq(tl.c);
    q.a = vq(tl.n);
    q.mat = tl.mat;
    return tl.body;
}
DRT_HD void pose_prim(const PoseQ &P, Prim<ff> &q) {
    q.p = vq(P.O) + rotq(P, q.p);
    q.a = rotq(P, q.a);
    if (q.type != T_S) q.b = rotq(P, q.b);
    if (q.type == T_D) q.c = rotq(P, q.c);
}
// posed from a table of rows [body][row]
DRT_HD Prim<ff> load_prim_ff(const LinkDev &L, const PoseQ *pose, int n_rows, int row, int type, int idx) {
    Prim<ff> q;
    const int body = load_prim_rest(L, type, idx, q);
    if (body >= 0) pose_prim(pose[(size_t)body * n_rows + row], q);
    return q;
}
// posed from the body's kinematics at t
DRT_HD Prim<ff> load_prim_ff_direct(const LinkDev &L, ff t, int type, int idx) {
    Prim<ff> q;
    const int body = load_prim_rest(L, type, idx, q);
    if (body >= 0) {
        PoseQ P;
        body_pose_ff(L.bodiesQ[body], t, P);
        pose_prim(P, q);
    }
    return q;
}
// the same with rates
DRT_HD Prim<dl<ff>> load_prim_ff_dual(const LinkDev &L, ff t, int type, int idx) {
    Prim<ff> q;
    const int body = load_prim_rest(L, type, idx, q);
    v3<ff> dp = V3<ff>(ff(0.f), ff(0.f), ff(0.f)), da = dp;
    if (body >= 0) {
        const BodyQ &B = L.bodiesQ[body];
        PoseQ P;
        body_pose_ff(B, t, P);
        pose_prim(P, q);
        const v3<ff> w = vq(B.k) * fma(B.wdot, t, B.w0);
        dp = axpy(vq(B.v), vq(B.a), t) + cross(w, q.p - vq(P.O));
        da = cross(w, q.a);
    }
    Prim<dl<ff>> r;
    r.type = q.type;
    r.mat = q.mat;
    r.idx = q.idx;
    r.p = dual(q.p, dp);
    r.a = dual(q.a, da);
    r.b = q.b;
    r.c = q.c;
    r.h1 = q.h1;
    r.h2 = q.h2;
    r.h3 = q.h3;
    r.h4 = q.h4;
    return r;
}
DRT_HD Prim<ff> val_prim(const Prim<dl<ff>> &q) {
    Prim<ff> r;
    r.type = q.type;
    r.mat = q.mat;
    r.idx = q.idx;
    r.p = val(q.p);
    r.a = val(q.a);
    r.b = q.b;
    r.c = q.c;
    r.h1 = q.h1;
    r.h2 = q.h2;
    r.h3 = q.h3;
    r.h4 = q.h4;
    return r;
}
DRT_HD v3<float> f32v(v3<ff> a) { return V3<float>(a.x.h, a.y.h, a.z.h); }
DRT_HD Prim<float> f32_prim(const Prim<dl<ff>> &q) {   // the Newton solve reads no more than this
    Prim<float> r;
    r.type = q.type;
    r.p = f32v(val(q.p));
    r.a = f32v(val(q.a));
    return r;
}
DRT_HD v3<dl<ff>> terminal_dual_ff(const TermQ &m, ff t) {
    const v3<ff> v = vq(m.v), a = vq(m.a);
    return dual(axpy(axpy(vq(m.r), v, t), a, halve(t * t)), axpy(v, a, t));
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
// neighbouring blocks on neighbouring paths it is 2 to 3 (41 to 59 % from one to three vertices).  Measured and left out: a barrier per stage, in blocks of 128 or one
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
    fl |= validity<N>(pr, N, V, tg.far);
    bool sure = !(fl & F_NOCONV) && (!(fl & (F_REDO64 | F_DEGEN)) || (fl & F_CLEAR)) && isfinite(d.h);
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

// ------------------------------------------------------------------------------------------------
// The FP64 parts of the FP32-bulk form in two-float numbers: warm starts, anchors at the chunk bases, and the redo of the steps FP32
// cannot resolve.  They are short dependent chains (a few solves per path), so what they cost is latency: 65 cycles per FP64
// instruction, a few per FP32 one.  Canyon: anchors 33 + 23 -> 15 + 22 us, warm starts 77 -> 31, redo 135 -> 59.

// The three-stage solve of solve_edge_params (drt_physics.cuh): FP32 values, two-float values, one dual-number step for the rates.  False
// where it did not converge (the caller runs the FP64 solve).  The rates only place Newton starts between the chunk bases and predict
// them from t = 0, so FP32 dual numbers give them (an error of 1e-5 of 10 m/s is 1e-6 m over a chunk, the size of the FP32
// rounding of the coordinates; a two-float step took half of the solve's latency) unless FP32 does not resolve the step.
template <int N>
DRT_HD bool solve_edge_params_ff(const LinkDev &L, int p, double t, const double *sin, double *sv, double *sd) {
    const uint32_t code = L.ptypes[p];
    const int4 pi = L.pprims[p];
    const int prim[MAXI] = {pi.x, pi.y, pi.z, pi.w};
    const ff tq = from_double(t);
    Prim<dl<ff>> pr[N];
#pragma unroll
    for (int j = 0; j < N; ++j) pr[j] = load_prim_ff_dual(L, tq, (code >> (8 * j)) & 0xff, prim[j]);
    v3<dl<ff>> V[N + 2];
    V[0] = terminal_dual_ff(L.txq, tq);
    V[N + 1] = terminal_dual_ff(L.rxq, tq);
    bool nv[N + 1];   // the unknowns: diffractions of a stretch with several of them
    int cf[N + 1], c = 0, run = -1;
#pragma unroll
    for (int i = 1; i <= N; ++i) {
        c = pr[i - 1].type == T_S ? 0 : c + (pr[i - 1].type == T_D ? 1 : 0);
        cf[i] = c;
    }
#pragma unroll
    for (int i = N; i >= 1; --i) {
        if (pr[i - 1].type == T_S) run = -1;
        else if (run < 0) run = cf[i];
        nv[i] = pr[i - 1].type == T_D && run >= 2;
    }
    place_tiles<N>(pr, V);
    double s1[MAXI];
#pragma unroll
    for (int j = 0; j < MAXI; ++j) s1[j] = sin[j];
    {
        Prim<float> pf[N];
        v3<float> Vf[N + 2];
        uint32_t ff_ = 0;
#pragma unroll
        for (int j = 0; j < N; ++j) pf[j] = f32_prim(pr[j]);
#pragma unroll
        for (int i = 0; i <= N + 1; ++i) Vf[i] = f32v(val(V[i]));
        newton_diffractions<N>(pf, Vf, nv, s1, (const double *)nullptr, (const double *)nullptr, ff_);
        if (!(ff_ & F_NOCONV))
#pragma unroll
            for (int j = 0; j < N; ++j)
                if (nv[j + 1]) s1[j] = (double)dot(Vf[j + 1] - pf[j].p, pf[j].a);
    }
    uint32_t fl = 0;
    {
        Prim<ff> pd[N];
        v3<ff> Vd[N + 2];
#pragma unroll
        for (int j = 0; j < N; ++j) pd[j] = val_prim(pr[j]);
#pragma unroll
        for (int i = 0; i <= N + 1; ++i) Vd[i] = val(V[i]);
        newton_diffractions<N>(pd, Vd, nv, s1, (const double *)nullptr, (const double *)nullptr, fl);
#pragma unroll
        for (int j = 0; j < N; ++j)
            if (nv[j + 1]) s1[j] = to_double(dot(Vd[j + 1] - pd[j].p, pd[j].a));
    }
    {
        Prim<dl<float>> pf[N];
        v3<dl<float>> Vf[N + 2];
#pragma unroll
        for (int j = 0; j < N; ++j) {
            pf[j].type = pr[j].type;
            pf[j].p = dual(f32v(val(pr[j].p)), f32v(der(pr[j].p)));
            pf[j].a = dual(f32v(val(pr[j].a)), f32v(der(pr[j].a)));
        }
#pragma unroll
        for (int i = 0; i <= N + 1; ++i) Vf[i] = dual(f32v(val(V[i])), f32v(der(V[i])));
        uint32_t f32 = 0;   // one step from the root gives the rates; its value part is the FP32 rounding
        newton_diffractions<N, 1>(pf, Vf, nv, s1, (const double *)nullptr, (const double *)nullptr, f32);
        bool ok = !(fl & F_NOCONV);
#pragma unroll
        for (int j = 0; j < MAXI; ++j) {
            sv[j] = s1[j];
            sd[j] = 0.0;
            if (j < N && nv[j + 1 < N + 1 ? j + 1 : N]) {
                const dl<float> sj = dot(Vf[j + 1 < N + 1 ? j + 1 : N] - pf[j < N ? j : 0].p, pf[j < N ? j : 0].a);
                sd[j] = sj.d;
                ok = ok && isfinite(sj.d) && fabsf(sj.v - (float)s1[j]) < 1e-3f;
            }
        }
        if (ok) return true;   // else (FP32 does not settle: near grazing) the step below
    }
    newton_diffractions<N>(pr, V, nv, s1, (const double *)nullptr, (const double *)nullptr, fl);
    bool ok = !(fl & F_NOCONV);
    // the diffractions alone in their stretch: on their Keller cones
    bool single = false;
#pragma unroll
    for (int i = 1; i <= N; ++i) single = single || (pr[i - 1].type == T_D && !nv[i]);
    if (single) place_keller<N>(pr, V, fl, nv);
#pragma unroll
    for (int j = 0; j < MAXI; ++j) {
        sv[j] = sin[j];
        sd[j] = 0.0;
        if (j < N && pr[j].type == T_D) {
            const dl<ff> sj = dot(V[j + 1] - pr[j].p, pr[j].a);
            ok = ok && isfinite(sj.v.h) && isfinite(sj.d.h);
            sv[j] = to_double(sj.v);
            sd[j] = to_double(sj.d);
        }
    }
    return ok;
}
template <int N> DRT_NOINL void solve_edge_params_fp64(const LinkDev &L, int p, double t, const double *sin, double *sv, double *sd) {
    solve_edge_params<N>(L, p, t, sin, sv, sd, [&](int ty, int idx) { return load_prim_direct<double>(L, t, ty, idx); });
}
DRT_HD void edge_params_ff(const LinkDev &L, int p, double t, const double *sin, double *sv, double *sd) {
    with_length<2>(chain_length(L, p), [&](auto NC) {
        constexpr int N = decltype(NC)::value;
        double start[MAXI];
        for (int j = 0; j < MAXI; ++j) start[j] = sin[j];
        if (!solve_edge_params_ff<N>(L, p, t, start, sv, sd)) solve_edge_params_fp64<N>(L, p, t, start, sv, sd);
    });
}
// path_t0par_fp64 and path_warm_fp64 (drt_physics.cuh) on it; the former's rates serve a linear predictor
DRT_HD void path_t0par_ff(const LinkDev &L, int p, double *out) {
    edge_params_ff(L, p, 0.0, L.ps0 + (size_t)p * MAXI, out, out + MAXI);
}
DRT_HD void path_warm_ff(const LinkDev &L, const TimeGridD &tg, int p, int row, double *warm) {
    const double t = tg.t_start + (double)row * tg.chunk * tg.dt;
    const double *q = L.t0par + (size_t)(p - L.n_bulk) * (2 * MAXI);
    double start[MAXI];
    for (int j = 0; j < MAXI; ++j) start[j] = q[j] + q[MAXI + j] * t;
    double *w = warm + ((size_t)row * (L.n_paths - L.n_bulk) + (p - L.n_bulk)) * (2 * MAXI);
    edge_params_ff(L, p, t, start, w, w + MAXI);
}

// path_base_fp64 (drt_physics.cuh): anchors of a (path, chunk) from the poses at the chunk bases [body][chunk]
template <int N> DRT_NOINL void path_base_ff_fallback(const LinkDev &L, const TimeGridD &tg, const FreqGridD &fg, int p, int chunk,
                                                      BaseRec *out, const double *warm) {
    const double tb = tg.t_start + (double)chunk * tg.chunk * tg.dt;
    path_base_fp64_core<N>(L, tg, fg, p, chunk, out, warm,
                           [&](int ty, int idx) { return val_prim(load_prim_direct<double>(L, tb, ty, idx)); });
}
template <int N = -1>
DRT_HD void path_base_ff(const LinkDev &L, const TimeGridD &tg, const FreqGridD &fg, const PoseQ *pose, int p, int chunk,
                         BaseRec *out, const double *warm) {
    if constexpr (N < 0) {
        with_length(chain_length(L, p), [&](auto NC) {
            path_base_ff<decltype(NC)::value>(L, tg, fg, pose, p, chunk, out, warm);
        });
    } else {
        const ff tb = from_double(tg.t_start + (double)chunk * tg.chunk * tg.dt);
        const int n_chunks = (tg.n_steps + tg.chunk - 1) / tg.chunk;
        const uint32_t code = L.ptypes[p];
        const int4 pi = L.pprims[p];
        const int prim[MAXI] = {pi.x, pi.y, pi.z, pi.w};
        Prim<ff> pr[N > 0 ? N : 1];
#pragma unroll
        for (int j = 0; j < N; ++j) pr[j] = load_prim_ff(L, pose, n_chunks, chunk, (code >> (8 * j)) & 0xff, prim[j]);
        v3<ff> V[N + 2];
        V[0] = val(terminal_dual_ff(L.txq, tb));
        V[N + 1] = val(terminal_dual_ff(L.rxq, tb));
        uint32_t fl = 0;
        const double *s0 = L.ps0 + (size_t)p * MAXI;
        if (warm && p >= L.n_bulk) s0 = warm_row(L, warm, chunk, p);
        solve_geometry_any<N>(pr, V, s0, fl);
        BaseRec r;
        ff d = ff(0.f);
#pragma unroll
        for (int i = 0; i <= MAXI; ++i) r.seg[i][0] = r.seg[i][1] = r.seg[i][2] = 0.f;
#pragma unroll
        for (int i = 1; i <= N + 1; ++i) {
            const v3<ff> sg = V[i] - V[i - 1];
            d = d + norm(sg);
            r.seg[i - 1][0] = sg.x.h;
            r.seg[i - 1][1] = sg.y.h;
            r.seg[i - 1][2] = sg.z.h;
        }
        if ((fl & (F_REDO64 | F_NOCONV | F_DEGEN)) || !isfinite(d.h)) {
            path_base_ff_fallback<N>(L, tg, fg, p, chunk, out, warm);
            return;
        }
        const ff x = d * fg.f0c_q, y = d * fg.dfc_q;
        const float st = y.h - floorf(y.h);
        r.d = to_double(d);
        r.ph0 = (x.h - floorf(x.h)) + x.l;
        r.st_hi = rintf((st + y.l) * 4096.f) * (1.f / 4096.f);
        r.st_lo = (st - r.st_hi) + y.l;
        r.pad = 0.f;
        out[(size_t)chunk * L.n_paths + p] = r;
    }
}

// App. A Eq. doppler_freq (doppler<N>, drt_physics.cuh): sum_i log1p(-u_i) - log1p(-u_{i-1}) with u = v.k / c, to second order while every
// |u| is below 1e-5 (the third-order terms are then below 1e-10 of the first).  The points of a chain that is no ray may run faster
// than that: FP64 logarithms there.
template <int N> DRT_HD float doppler_ff(const v3<dl<ff>> *V, const v3<ff> *seg, const FreqGridD &fg) {
    ff s1 = ff(0.f);
    float s2 = 0.f, big = 0.f;
    double full = 0.0;
#pragma unroll
    for (int i = 1; i <= N + 1; ++i) {
        const v3<ff> k = unit(seg[i]);
        const ff u1 = dot(der(V[i]), k), u0 = dot(der(V[i - 1]), k);
        s1 = s1 + (u0 - u1);
        s2 += (u0.h - u1.h) * (u0.h + u1.h);
        const float m = fmaxf(fabsf(u0.h), fabsf(u1.h));
        big = fmaxf(big, m);
        if (!(m < 1e-5f * (float)C0)) full += log1p(-to_double(u1) * (1 / C0)) - log1p(-to_double(u0) * (1 / C0));
        else full += to_double(u0 - u1) * (1 / C0);
    }
    if (!(big < 1e-5f * (float)C0)) return (float)(fg.fc * expm1(full));
    const ff S = s1 * ff(1 / C0) + ff(s2 * (float)(0.5 / (C0 * C0)));
    return (fg.kq * ff(C0 / (2 * PI)) * (S + halve(S * S))).h;   // fc = k c / 2 pi
}

// Redo of one queued FP32-bulk path-step in two-float numbers: FP32 output formats and
// (Re a, Im a, tau) in rec64, a = 0 where the path does not exist.  False where two-float numbers cannot decide the step.
template <int N, bool DUAL>
DRT_HD bool path_step_redo_ff(const LinkDev &L, const TimeGridD &tg, const FreqGridD &fg, int p, int ti, const OutD &out,
                              const double *warm, double *rec64) {
    typedef std::conditional_t<DUAL, dl<ff>, ff> S;
    const ff t = from_double(tg.t_start + ti * tg.dt);
    const uint32_t code = L.ptypes[p];
    const int4 pi = L.pprims[p];
    const int prim[MAXI] = {pi.x, pi.y, pi.z, pi.w};
    Prim<S> pr[N > 0 ? N : 1];
#pragma unroll
    for (int j = 0; j < N; ++j) {
        if constexpr (DUAL) pr[j] = load_prim_ff_dual(L, t, (code >> (8 * j)) & 0xff, prim[j]);
        else pr[j] = load_prim_ff_direct(L, t, (code >> (8 * j)) & 0xff, prim[j]);
    }
    v3<S> V[N + 2];
    if constexpr (DUAL) {
        V[0] = terminal_dual_ff(L.txq, t);
        V[N + 1] = terminal_dual_ff(L.rxq, t);
    } else {
        V[0] = val(terminal_dual_ff(L.txq, t));
        V[N + 1] = val(terminal_dual_ff(L.rxq, t));
    }
    uint32_t fl = 0;
    if (warm && p >= L.n_bulk) {
        WarmStart32 ws;
        warm_start_at32(L, tg, warm, p, ti, ws);
        solve_geometry_any<N>(pr, V, ws.s, fl, ws.ds, ws.rate);
    } else {
        solve_geometry_any<N>(pr, V, L.ps0 + (size_t)p * MAXI, fl);
    }
    v3<ff> P[N + 2], seg[N + 2];
    ff d = ff(0.f);
    P[0] = val(V[0]);
#pragma unroll
    for (int i = 1; i <= N + 1; ++i) {
        P[i] = val(V[i]);
        seg[i] = P[i] - P[i - 1];
        d = d + norm(seg[i]);
    }
    fl |= validity<N>(pr, N, P, tg.far);
    if ((fl & (F_REDO64 | F_NOCONV | F_DEGEN)) || !isfinite(d.h)) return false;   // every bit is written out: all decided
    fl &= ~F_CLEAR;
    cx<ff> a = C<ff>(ff(0.f), ff(0.f));
    if (!fl || out.amp) {
        Prim<ff> pv[N > 0 ? N : 1];
        if constexpr (DUAL) {
#pragma unroll
            for (int j = 0; j < N; ++j) pv[j] = val_prim(pr[j]);
            a = amplitude_ff<N>(L, pv, seg, fg);
        } else {
            a = amplitude_ff<N>(L, pr, seg, fg);
        }
        if (!isfinite(a.re.h) || !isfinite(a.im.h)) return false;
    }
    const double tau = to_double(d) * (1 / C0);
    if (rec64) {
        rec64[0] = fl ? 0.0 : to_double(a.re);
        rec64[1] = fl ? 0.0 : to_double(a.im);
        rec64[2] = tau;
    }
    const size_t oi = (size_t)ti * L.n_paths + L.perm[p];
    if (out.tau) out.tau[oi] = tau;
    if (out.amp) {
        float *q = reinterpret_cast<float *>(out.amp) + 2 * oi;
        q[0] = a.re.h;
        q[1] = a.im.h;
    }
    if constexpr (DUAL)
        if (out.doppler) reinterpret_cast<float *>(out.doppler)[oi] = doppler_ff<N>(V, seg, fg);
    if (out.angles) {
        const v3<ff> kd = seg[1], ka = -seg[N + 1];
        auto flat = [](v3<ff> k) {   // length of the horizontal part
            const ff r2 = fma(k.x, k.x, k.y * k.y);
            return r2.h > 0.f ? sqrt(r2) : ff(0.f);
        };
        float *q = out.angles + 4 * oi;
        q[0] = atan2_ff(kd.y, kd.x);
        q[1] = atan2_ff(kd.z, flat(kd));
        q[2] = atan2_ff(ka.y, ka.x);
        q[3] = atan2_ff(ka.z, flat(ka));
    }
    if (out.flags) out.flags[oi] = (uint8_t)fl;
    if (out.points) {
        double *q = out.points + oi * (MAXI * 3);
        const double qn = nan("");
#pragma unroll
        for (int j = 0; j < MAXI; ++j) {
            q[3 * j + 0] = j < N ? to_double(P[j + 1 < N + 1 ? j + 1 : N].x) : qn;
            q[3 * j + 1] = j < N ? to_double(P[j + 1 < N + 1 ? j + 1 : N].y) : qn;
            q[3 * j + 2] = j < N ? to_double(P[j + 1 < N + 1 ? j + 1 : N].z) : qn;
        }
    }
    return true;
}
template <int N, bool DUAL>
DRT_NOINL void path_step_redo_fp64(const LinkDev &L, const TimeGridD &tg, const FreqGridD &fg, int p, int ti, const OutD &out,
                                   const double *warm, double *rec64) {
    const double t = tg.t_start + ti * tg.dt;
    const RecD nor{nullptr, nullptr};
    if constexpr (DUAL)
        path_step_fp64_core<N, true, true, dl<double>>(
            L, tg, fg, p, ti, out, nor, true, [&](int ty, int idx) { return load_prim_direct<double>(L, t, ty, idx); },
            warm, rec64);
    else
        path_step_fp64_core<N, true, true, double>(
            L, tg, fg, p, ti, out, nor, true,
            [&](int ty, int idx) { return val_prim(load_prim_direct<double>(L, t, ty, idx)); }, warm, rec64);
}
// two: two-float numbers apply to the link and grid (ff_applies), else the step is computed in FP64
template <bool DUAL>
DRT_HD void path_step_redo(const LinkDev &L, const TimeGridD &tg, const FreqGridD &fg, int p, int ti, const OutD &out,
                           const double *warm, double *rec64, bool two) {
    with_length(chain_length(L, p), [&](auto NC) {
        constexpr int N = decltype(NC)::value;
        if (!two || !path_step_redo_ff<N, DUAL>(L, tg, fg, p, ti, out, warm, rec64))
            path_step_redo_fp64<N, DUAL>(L, tg, fg, p, ti, out, warm, rec64);
    });
}

// ------------------------------------------------------------------------------------------------
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
