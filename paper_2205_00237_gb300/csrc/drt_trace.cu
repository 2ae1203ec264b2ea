// drt_trace.cu -- conventional ray tracing at one instant on the GPU (Sec. II: the ray-tracing run DRT
// starts from at t0 and repeats at every multipath-lifetime boundary, Sec. IV-B), by brute-force
// image-tree enumeration: every chain of at most two reflections / diffractions (no primitive twice
// in a row) and every single-tile scattering chain is a candidate; one thread solves a candidate with
// the extrapolation's FP64 geometry at the instant (image method, Keller cone, Newton from the edge
// midpoints for two diffractions in a segment), keeps it when its FP64 validity flags are 0 and no
// face blocks any of its segments, and appends it to the output list.
#include <algorithm>
#include <cstdint>
#include <vector>

#include "drt_launch.cuh"
#include "drt_physics_ff.cuh"

namespace drt {

// a face posed at the instant: centre, unit normal, in-plane axes, half extents
struct PosedFace { double c[3], n[3], u[3], w[3], hu, hw; };
struct PosedFaceQ { ff c[3], n[3], u[3], w[3], hu, hw; };   // the same in two-float numbers, in a table behind the first

DRT_HD void pose_face(const LinkDev &L, double t, int f, PosedFace *out_f) {
    const FaceD &F = L.faces[f];
    double P[POSE_W];
    body_pose_row(L.bodies[F.body], t, P);
    const Pose<double> q = load_pose<double>(P);
    const v3<double> c = q.O + rot(q, F.c), n = rot(q, F.n), u = rot(q, F.u), w = cross(u, n);
    PosedFace r;
    r.c[0] = c.x; r.c[1] = c.y; r.c[2] = c.z;
    r.n[0] = n.x; r.n[1] = n.y; r.n[2] = n.z;
    r.u[0] = u.x; r.u[1] = u.y; r.u[2] = u.z;
    r.w[0] = w.x; r.w[1] = w.y; r.w[2] = w.z;
    r.hu = F.hu;
    r.hw = F.hw;
    *out_f = r;
}

__global__ void k_pose_faces(const LinkDev L, double t, PosedFace *__restrict__ out, PosedFaceQ *__restrict__ outq) {
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= L.n_faces) return;
    pose_face(L, t, f, out + f);
    if (!outq) return;
    const PosedFace F = out[f];
    PosedFaceQ q;
    for (int j = 0; j < 3; ++j) {
        q.c[j] = from_double(F.c[j]);
        q.n[j] = from_double(F.n[j]);
        q.u[j] = from_double(F.u[j]);
        q.w[j] = from_double(F.w[j]);
    }
    q.hu = L.facesQ[f].hu;
    q.hw = L.facesQ[f].hw;
    outq[f] = q;
}

// Does the face block the segment A -> B?  It does when the segment crosses the face's plane
// strictly between its ends at a point inside the rectangle; a face whose plane holds A or B (within
// 1e-9 m: the face a reflection point or a tile lies on, the faces of a diffracting edge, faces coplanar
// with those) does not.
DRT_HD bool face_blocks(const PosedFace &F, v3<double> A, v3<double> B) {
    const v3<double> c = V3(F.c[0], F.c[1], F.c[2]), n = V3(F.n[0], F.n[1], F.n[2]);
    const double ha = dot(A - c, n), hb = dot(B - c, n);
    if (fabs(ha) < 1e-9 || fabs(hb) < 1e-9) return false;
    if ((ha > 0.0) == (hb > 0.0)) return false;
    const v3<double> r = A + (B - A) * (ha / (ha - hb)) - c;
    return fabs(dot(r, V3(F.u[0], F.u[1], F.u[2]))) <= F.hu && fabs(dot(r, V3(F.w[0], F.w[1], F.w[2]))) <= F.hw;
}

// one ray found: its enumeration index, chain and diffraction parameters at the instant
// (n: the vertices, and from bit 8 on how far it is decided; index -1: FP64 found that it is none)
enum { RAY_FINAL = 0, RAY_POLISH = 1, RAY_OPEN = 2 };
struct RayPoints { ff v[2][3]; float amp, pad; };   // the solved vertices of a listed candidate, and its amp (validity)
struct TracedRay { long long index; int32_t n; uint32_t types; int32_t prims[MAXI]; double s[MAXI]; };

constexpr int TRACE_T = 128;

// candidate k of the enumeration (0 = line of sight; single faces (R), edges (D), tiles (S); ordered
// pairs of faces / edges, the same primitive twice excluded) solved at t: true when it is a ray, which
// then fills *r
// the candidate's chain of N interactions (codes c[0..N-1]): solved, checked and, if it is a ray, stored
// (blocked(A, B): whether a face blocks a segment)
template <int N, class Blocked>
DRT_HD bool trace_chain(const LinkDev &L, double t, long long k, const int *code, TracedRay *r, Blocked blocked) {
    const int NP = L.n_faces + L.n_edges;
    Prim<double> pr[N > 0 ? N : 1];
    double s0[MAXI] = {0.0, 0.0, 0.0, 0.0};
    uint32_t types = 0;
    int prims[MAXI] = {0, 0, 0, 0};
#pragma unroll
    for (int j = 0; j < N; ++j) {
        const int c = code[j];
        int ty, idx;
        if (c < L.n_faces) { ty = T_R; idx = c; }
        else if (c < NP) { ty = T_D; idx = c - L.n_faces; s0[j] = 0.5 * L.edges[idx].len; }
        else { ty = T_S; idx = c - NP; }
        pr[j] = val_prim(load_prim_direct<double>(L, t, ty, idx));
        types |= (uint32_t)ty << (8 * j);
        prims[j] = idx;
    }
    v3<double> V[N + 2];
    V[0] = val(terminal<double>(L.tx, t));
    V[N + 1] = val(terminal<double>(L.rx, t));
    uint32_t fl = 0;
    solve_geometry_any<N>(pr, V, s0, fl);
    fl |= validity<N>(pr, N, V);
#pragma unroll
    for (int i = 1; i <= N; ++i)
        if (!(isfinite(V[i].x) && isfinite(V[i].y) && isfinite(V[i].z))) fl |= F_DEGEN;
    if (fl) return false;
#pragma unroll
    for (int i = 1; i <= N + 1; ++i)
        if (blocked(V[i - 1], V[i])) return false;
    r->index = k;
    r->n = N;
    r->types = types;
#pragma unroll
    for (int j = 0; j < MAXI; ++j) {
        r->prims[j] = prims[j];
        r->s[j] = 0.0;
        if (j < N)
            if (pr[j].type == T_D) r->s[j] = dot(V[j + 1] - pr[j].p, pr[j].a);
    }
    return true;
}

template <class Blocked>
DRT_HD bool trace_eval(const LinkDev &L, double t, long long k, int with_tiles, TracedRay *r, Blocked blocked) {
    const int NP = L.n_faces + L.n_edges, NT = with_tiles ? L.n_tiles : 0;
    int n = 0, code[2] = {0, 0};
    if (k > 0) {
        const long long j = k - 1;
        if (j < NP + NT) {
            code[0] = (int)j;
            n = 1;
        } else {
            const long long q = j - NP - NT;
            code[0] = (int)(q / NP);
            code[1] = (int)(q % NP);
            if (code[0] == code[1]) return false;
            n = 2;
        }
    }
    if (n == 0) return trace_chain<0>(L, t, k, code, r, blocked);
    if (n == 1) return trace_chain<1>(L, t, k, code, r, blocked);
    return trace_chain<2>(L, t, k, code, r, blocked);
}

__global__ void __launch_bounds__(TRACE_T)
k_trace(const LinkDev L, double t, long long n_cand, int with_tiles, const PosedFace *__restrict__ faces,
        TracedRay *__restrict__ out, int cap, int *__restrict__ count) {
    const long long k = blockIdx.x * (long long)TRACE_T + threadIdx.x;
    if (k >= n_cand) return;
    TracedRay r;
    if (!trace_eval(L, t, k, with_tiles, &r, [&](v3<double> A, v3<double> B) {
            for (int f = 0; f < L.n_faces; ++f)
                if (face_blocks(faces[f], A, B)) return true;
            return false;
        }))
        return;
    const int slot = atomicAdd(count, 1);
    if (slot < cap) out[slot] = r;
}

// ------------------------------------------------------------------------------------------------
// The same in three passes.  Nearly every candidate is no ray by a clear margin, and in FP64 all of them wait on the FP64 pipe, and
// the few that reach the segment-face tests on one thread's loop over the faces (1.13 ms for the canyon's 97206 candidates).  k_trace_ff
// solves and checks the candidates in two-float numbers, with margins as in path_step_ff, and lists those that may be rays;
// k_trace_block, a warp per listed candidate, spreads the (segment, face) tests over its lanes and tries what is still open in FP64;
// k_trace_polish solves the rays' diffraction parameters in FP64 from the two-float ones (one Newton step).  The list ends as k_trace's.

// 1: the face blocks the segment, 0: it does not, -1: within the margins.  The ends' heights over the face are less certain than a
// coordinate by upA and upB, their places along it by amp
DRT_NOINL1 int face_blocks_ff(const PosedFaceQ &F, v3<ff> A, v3<ff> B, float upA, float upB, float amp, float far) {
    const v3<ff> c = vq(F.c), n = vq(F.n);
    const ff ha = dot(A - c, n), hb = dot(B - c, n);
    const float fa = fabsf(ha.h), fb = fabsf(hb.h), scale = fmaxf(fmaxf(amax3(A), amax3(B)), fmaxf(amax3(c), far));
    // an end within 1e-9 m of the plane: the points of a chain lie on its own faces to ~2^-46 of the coordinates, which 2^-42 bounds
    const float tol = ff_margin_tol(scale), e = fmaxf(2.3e-13f * (scale + 1.f), 1e-10f);
    if (!(fabsf(fa - 1e-9f) > e * upA) || !(fabsf(fb - 1e-9f) > e * upB)) return -1;
    if (fa < 1e-9f || fb < 1e-9f) return 0;
    if ((ha.h > 0.f) == (hb.h > 0.f)) return 0;
    const v3<ff> r = axpy(A, B - A, ha / (ha - hb)) - c;
    const float mu = ff_within(dot(r, vq(F.u)), F.hu), mw = ff_within(dot(r, vq(F.w)), F.hw);
    // the point moves along the plane with the error of h over the segment's slope
    const v3<ff> d = B - A;
    const float lim = tol * fmaxf(1.f, amp * (1.f / 64.f)) * (1.f + (fabsf(d.x.h) + fabsf(d.y.h) + fabsf(d.z.h)) / (fa + fb));
    if (mu < -lim || mw < -lim) return 0;
    return mu > lim && mw > lim ? 1 : -1;
}

// how much less certain than a coordinate the height over a face of normal n is at a vertex on the primitive q, which may lie amp
// coordinate errors from its place along its face or edge
DRT_HD float height_amp(const Prim<ff> &q, v3<float> n, float amp) {
    const v3<float> a = f32v(q.a);
    const v3<float> x = cross(a, n);
    return 1.f + amp * (q.type == T_D ? fabsf(dot(a, n)) : sqrtf(dot(x, x)));
}

// the faces, then the edges, posed
__global__ void __launch_bounds__(128)
k_pose_prims(const __grid_constant__ LinkDev L, double t, Prim<ff> *__restrict__ prims) {
    const int i = blockIdx.x * 128 + threadIdx.x;
    if (i >= L.n_faces + L.n_edges) return;
    prims[i] = load_prim_ff_direct(L, from_double(t), i < L.n_faces ? T_R : T_D, i < L.n_faces ? i : i - L.n_faces);
}

// Two edges whose lines meet in a point C (a corner of a box or of a facade): the shortest path over both runs through C when the length
// has its minimum at that kink, where the Newton solve does not converge or ends on a path without a middle segment; either way the
// chain is no ray.  The minimum is there when the pulls of the outer segments along the edges can be balanced by a vector z of length
// below 1 (the subgradient of the middle segment's length): z.e1 = -p, z.e2 = -q with p = u.e1, q = w.e2 for the unit directions u
// from A to C and w from C to B.  The length is convex, so a kink minimum with |z| clear of 1 is its only stationary point.
DRT_HD bool corner_path(const Prim<ff> &E1, const Prim<ff> &E2, v3<ff> A, v3<ff> B) {
    const v3<ff> x = cross(E1.a, E2.a), d = E2.p - E1.p;
    const ff xx = dot(x, x), gap = dot(d, x);
    // the lines meet within 5e-11 m: with |z|^2 < 0.99 the middle segment of the shortest path is then below 5e-10 m, no segment
    if (!(xx.h > 1e-4f) || !(gap.h * gap.h < 2.5e-21f * xx.h)) return false;
    const v3<ff> C = axpy(E1.p, E1.a, dot(cross(d, E2.a), x) / xx);
    const v3<float> e1 = f32v(E1.a), e2 = f32v(E2.a), ac = f32v(C - A), cb = f32v(B - C);
    if (!(dot(ac, ac) > 0.01f) || !(dot(cb, cb) > 0.01f)) return false;
    const v3<float> u = unit(ac), w = unit(cb);
    const float c = dot(e1, e2), p = dot(u, e1), q = dot(w, e2), det = 1.f - c * c;
    const float a = (c * q - p) / det, b = (c * p - q) / det;   // z = a e1 + b e2
    return -(a * p + b * q) < 0.99f;                            // |z|^2
}

// A pair solved in FP32 first: whether the solve fails a test with every margin (the failed one's too) clear of the FP32 error, so that the
// chain is none.  A coordinate's error moves a point by the amplification of vertex_margins at each vertex; the points' errors were at most
// 0.08 of that product times 2e-6 of the coordinates (2e6 random pairs), so an eighth of it, and 1000 in any case, bounds the margins.
struct Fp32Check { bool none; float margin, amp; };
DRT_HD Fp32Check fp32_first(const Prim<ff> *pr, const v3<ff> *V, const double *s0, Prim<float> *pf, v3<float> *Vf, uint32_t &f0) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        pf[j].type = pr[j].type;
        pf[j].p = f32v(pr[j].p);
        pf[j].a = f32v(pr[j].a);
        pf[j].b = f32v(pr[j].b);
        pf[j].c = f32v(pr[j].c);
        pf[j].h1 = pr[j].h1.h;
        pf[j].h2 = pr[j].h2.h;
        pf[j].h3 = pr[j].h3.h;
        pf[j].h4 = pr[j].h4.h;
    }
    Vf[0] = f32v(V[0]);
    Vf[3] = f32v(V[3]);
    uint32_t bad = 0;
    solve_geometry_any<2>(pf, Vf, s0, f0);
    float margin = 1e30f, amp = 1.f;
    bool fine = true;
#pragma unroll
    for (int i = 1; i <= 2; ++i) {
        const Prim<float> &q = pf[i - 1];
        const VertexCheck<float> v = vertex_validity_inl(q.type, q.p, q.a, q.b, q.c, q.h1, q.h2, q.h3, q.h4, Vf[i - 1], Vf[i], Vf[i + 1]);
        bad |= v.fl;
        margin = fminf(margin, v.m);
        fine = fine && isfinite(Vf[i].x) && isfinite(Vf[i].y) && isfinite(Vf[i].z) && v.m > 1000.f;
        // of a leg and its part along the normal or the edge: leg / height, or (leg / distance from the edge line)^2
        const v3<float> dm = Vf[i - 1] - Vf[i], dp = Vf[i + 1] - Vf[i];
        const float hm = dot(dm, q.a), hp = dot(dp, q.a), lm = dot(dm, dm), lp = dot(dp, dp);
        if (q.type == T_R) amp *= 1.f + sqrtf(2.f * (lm + lp)) / (fabsf(hm) + fabsf(hp));
        else amp *= 1.f / fmaxf(1.f - fmaxf(hm * hm / lm, hp * hp / lp), 0.f);
    }
    return Fp32Check{fine && bad && margin > 1000.f && margin > 0.125f * amp && !(f0 & (F_NOCONV | F_REDO64 | F_DEGEN)), margin, amp};
}

template <int N>
DRT_HD int trace_chain_ff(const LinkDev &L, double t, float far, const int *code, const Prim<ff> *prims, TracedRay *r,
                          RayPoints *v) {
    const int NP = L.n_faces + L.n_edges;
    const ff tq = from_double(t);
    Prim<ff> pr[N > 0 ? N : 1];
    double s0[MAXI] = {0.0, 0.0, 0.0, 0.0};
    uint32_t types = 0;
    bool any_d = false;
    r->n = N;
#pragma unroll
    for (int j = 0; j < MAXI; ++j) {
        r->prims[j] = 0;
        r->s[j] = 0.0;
    }
#pragma unroll
    for (int j = 0; j < N; ++j) {
        const int c = code[j];
        int ty, idx;
        if (c < L.n_faces) { ty = T_R; idx = c; }
        else if (c < NP) { ty = T_D; idx = c - L.n_faces; s0[j] = 0.5 * L.edges[idx].len; }
        else { ty = T_S; idx = c - NP; }
        if (ty == T_S) pr[j] = load_prim_ff_direct(L, tq, ty, idx);
        else pr[j] = prims[c];
        types |= (uint32_t)ty << (8 * j);
        r->prims[j] = idx;
        any_d = any_d || ty == T_D;
    }
    r->types = types;
    v3<ff> V[N + 2];
    V[0] = val(terminal_dual_ff(L.txq, tq));
    V[N + 1] = val(terminal_dual_ff(L.rxq, tq));
    uint32_t fl = 0;
    if constexpr (N == 2) {
        if (pr[0].type == T_D && pr[1].type == T_D && corner_path(pr[0], pr[1], V[0], V[3])) return -1;
        Prim<float> pf[2];
        v3<float> Vf[4];
        uint32_t f0 = 0;
        if (fp32_first(pr, V, s0, pf, Vf, f0).none) return -1;
        if (!(f0 & F_NOCONV))   // the two-float Newton solve starts from the FP32 one's
#pragma unroll
            for (int j = 0; j < 2; ++j)
                if (pf[j].type == T_D) s0[j] = (double)dot(Vf[j + 1] - pf[j].p, pf[j].a);
    }
    solve_geometry_any<N>(pr, V, s0, fl);
    fl |= validity<N>(pr, N, V, far, &v->amp);
    if (fl & F_NOCONV) return RAY_OPEN;
#pragma unroll
    for (int i = 1; i <= N; ++i)
        if (!(isfinite(V[i].x.h) && isfinite(V[i].y.h) && isfinite(V[i].z.h))) return RAY_OPEN;
    if (fl & F_CLEAR) return -1;
    if (fl & (F_REDO64 | F_DEGEN)) return RAY_OPEN;
    if (fl) return -1;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        v->v[j][0] = V[j + 1].x;
        v->v[j][1] = V[j + 1].y;
        v->v[j][2] = V[j + 1].z;
        if (pr[j].type == T_D) r->s[j] = to_double(dot(V[j + 1] - pr[j].p, pr[j].a));
    }
    return any_d ? RAY_POLISH : RAY_FINAL;
}

__global__ void __launch_bounds__(TRACE_T)
k_trace_ff(const __grid_constant__ LinkDev L, double t, float far, long long n_cand, int with_tiles, const Prim<ff> *__restrict__ prims,
           TracedRay *__restrict__ out, RayPoints *__restrict__ points, int cap, int *__restrict__ count) {
    const long long k = blockIdx.x * (long long)TRACE_T + threadIdx.x;
    if (k >= n_cand) return;
    const int NP = L.n_faces + L.n_edges, NT = with_tiles ? L.n_tiles : 0;
    TracedRay r;
    RayPoints v{};
    int code[2] = {0, 0}, state;
    if (k == 0) {
        state = trace_chain_ff<0>(L, t, far, code, prims, &r, &v);
    } else if (k - 1 < NP + NT) {
        code[0] = (int)(k - 1);
        state = trace_chain_ff<1>(L, t, far, code, prims, &r, &v);
    } else {
        const long long q = k - 1 - NP - NT;
        code[0] = (int)(q / NP);
        code[1] = (int)(q % NP);
        if (code[0] == code[1]) return;
        state = trace_chain_ff<2>(L, t, far, code, prims, &r, &v);
    }
    if (state < 0) return;
    r.index = k;
    r.n |= state << 8;
    const int slot = atomicAdd(count, 1);
    if (slot >= cap) return;
    out[slot] = r;
    points[slot] = v;
}

__global__ void __launch_bounds__(128)
k_trace_block(const __grid_constant__ LinkDev L, double t, float far, int with_tiles, const PosedFace *__restrict__ faces,
              const PosedFaceQ *__restrict__ facesq, const Prim<ff> *__restrict__ prims, TracedRay *__restrict__ out, const RayPoints *__restrict__ points, int cap,
              const int *__restrict__ count) {
    const int n = min(*count, cap), lane = threadIdx.x & 31;
    const ff tq = from_double(t);
    for (int k = blockIdx.x * 4 + (threadIdx.x >> 5); k < n; k += gridDim.x * 4) {   // warp-uniform
        TracedRay *r = out + k;
        if (r->n >> 8 != RAY_OPEN) {
            const int N = r->n & 255;
            const RayPoints &v = points[k];
            const v3<ff> tx = val(terminal_dual_ff(L.txq, tq)), rx = val(terminal_dual_ff(L.rxq, tq));
            bool hit = false, open = false;
            for (int q = lane; q < (N + 1) * L.n_faces; q += 32) {
                const int i = q / L.n_faces, f = q - i * L.n_faces;
                const v3<ff> A = i == 0 ? tx : vq(v.v[i - 1]), B = i == N ? rx : vq(v.v[i]);
                // (terminals and tiles are where they are; for nearly every face the most that a height can be off is enough)
                int b = face_blocks_ff(facesq[f], A, B, i == 0 ? 1.f : 1.f + v.amp, i == N ? 1.f : 1.f + v.amp, v.amp, far);
                if (b < 0) {
                    const v3<float> n = f32v(vq(facesq[f].n));
                    auto up = [&](int j) {   // of vertex j + 1
                        const int ty = (r->types >> (8 * j)) & 0xff;
                        return ty == T_S ? 1.f : height_amp(prims[r->prims[j] + (ty == T_D ? L.n_faces : 0)], n, v.amp);
                    };
                    b = face_blocks_ff(facesq[f], A, B, i == 0 ? 1.f : up(i - 1), i == N ? 1.f : up(i), v.amp, far);
                }
                hit = hit || b > 0;
                open = open || b < 0;
            }
            hit = __any_sync(0xffffffffu, hit);
            open = __any_sync(0xffffffffu, open);
            if (hit) {
                if (lane == 0) r->index = -1;
                continue;
            }
            if (!open) continue;
        }
        TracedRay q;
        const bool ray = trace_eval(L, t, r->index, with_tiles, &q, [&](v3<double> A, v3<double> B) {
            bool hit = false;
            for (int f = lane; f < L.n_faces; f += 32) hit = hit || face_blocks(faces[f], A, B);
            return __any_sync(0xffffffffu, hit) != 0;
        });
        __syncwarp();   // every lane has read the entry
        if (lane == 0) {
            if (ray) *r = q;
            else r->index = -1;
        }
    }
}

// the diffraction parameters of a ray in FP64, from the two-float ones
template <int N> DRT_HD void polish_ray(const LinkDev &L, double t, TracedRay *r) {
    Prim<double> pr[N];
    double s0[MAXI] = {r->s[0], r->s[1], 0.0, 0.0};
#pragma unroll
    for (int j = 0; j < N; ++j) pr[j] = val_prim(load_prim_direct<double>(L, t, (r->types >> (8 * j)) & 0xff, r->prims[j]));
    v3<double> V[N + 2];
    V[0] = val(terminal<double>(L.tx, t));
    V[N + 1] = val(terminal<double>(L.rx, t));
    uint32_t fl = 0;
    solve_geometry_any<N>(pr, V, s0, fl);
#pragma unroll
    for (int j = 0; j < N; ++j)
        if (pr[j].type == T_D) r->s[j] = dot(V[j + 1] - pr[j].p, pr[j].a);
}

__global__ void __launch_bounds__(32)
k_trace_polish(const __grid_constant__ LinkDev L, double t, TracedRay *__restrict__ out, int cap, const int *__restrict__ count) {
    const int n = min(*count, cap);
    for (int k = blockIdx.x * 32 + threadIdx.x; k < n; k += gridDim.x * 32) {
        TracedRay *r = out + k;
        if (r->n >> 8 != RAY_POLISH || r->index < 0) continue;
        if ((r->n & 255) == 1) polish_ray<1>(L, t, r);
        else polish_ray<2>(L, t, r);
    }
}

long long trace_candidates(const LinkDev &L, int max_order, int with_tiles) {
    const long long NP = L.n_faces + L.n_edges, NT = with_tiles ? L.n_tiles : 0;
    return 1 + (max_order >= 1 ? NP + NT : 0) + (max_order >= 2 ? NP * NP : 0);
}

// The three passes cost 25 us more in launches, and at order 2 the solves of what stays open come on top of the two-float ones
// (560 + us against 435 for a handful of candidates); what they save is the FP64 pass's loop over the faces on one thread (per
// face 0.9 us at order 0, 2.5 at 1, 3 at 2) and, where the candidates are more than the FP64 pipes take at once, its solves.
// Measured on parts of the canyon and link scenes, FP64 | two-float us: order 0, 18 faces 90 | 102, 53 faces 118 | 101; order 1, 10
// faces 116 | 124, 17 faces 134 | 107; order 2, 31 faces and 84 edges 530 | 725, 53 and 129 (33125 candidates) 826 | 717.
bool trace_two_float(const LinkDev &L, int max_order, int with_tiles) {
    const int least = max_order == 0 ? 31 : max_order == 1 ? 11 : 41;
    return L.n_faces >= least || trace_candidates(L, max_order, with_tiles) > 16384;
}

size_t trace_ray_bytes() { return sizeof(TracedRay); }
size_t trace_face_bytes() { return sizeof(PosedFace); }
size_t trace_prim_bytes(const LinkDev &L, int cap) {   // posed faces and primitives, then the points of `cap` listed candidates
    return (size_t)L.n_faces * sizeof(PosedFaceQ) + (size_t)(L.n_faces + L.n_edges) * sizeof(Prim<ff>) + cap * sizeof(RayPoints);
}

cudaError_t launch_trace(const LinkDev &L, double t, int max_order, int with_tiles, void *faces, void *rays, int cap,
                         int *count, cudaStream_t s, void *prims_mem, double far) {
    const bool two = prims_mem != nullptr;
    cudaError_t e = cudaMemsetAsync(count, 0, sizeof(int), s);
    if (e != cudaSuccess) return e;
    PosedFace *F = reinterpret_cast<PosedFace *>(faces);
    PosedFaceQ *Q = reinterpret_cast<PosedFaceQ *>(prims_mem);
    TracedRay *out = reinterpret_cast<TracedRay *>(rays);
    if (L.n_faces > 0) k_pose_faces<<<(L.n_faces + 127) / 128, 128, 0, s>>>(L, t, F, Q);
    const long long n = trace_candidates(L, max_order, with_tiles);
    const unsigned grid = (unsigned)((n + TRACE_T - 1) / TRACE_T);
    if (two) {
        Prim<ff> *prims = reinterpret_cast<Prim<ff> *>(Q + L.n_faces);
        const int np = L.n_faces + L.n_edges;
        RayPoints *points = reinterpret_cast<RayPoints *>(prims + np);
        if (np) k_pose_prims<<<(np + 127) / 128, 128, 0, s>>>(L, t, prims);
        k_trace_ff<<<grid, TRACE_T, 0, s>>>(L, t, (float)far, n, with_tiles, prims, out, points, cap, count);
        k_trace_block<<<152 * 4, 128, 0, s>>>(L, t, (float)far, with_tiles, F, Q, prims, out, points, cap, count);
        k_trace_polish<<<152 * 8, 32, 0, s>>>(L, t, out, cap, count);
    } else {
        k_trace<<<grid, TRACE_T, 0, s>>>(L, t, n, with_tiles, F, out, cap, count);
    }
    return cudaGetLastError();
}

// the rays in a list of `count` (in any order) to host arrays in enumeration order; returns their number
int trace_unpack(const void *rays_host, int count, uint8_t *n_int, uint8_t *types, int32_t *prims, double *s0, int cap) {
    const TracedRay *R = reinterpret_cast<const TracedRay *>(rays_host);
    std::vector<int> order;
    order.reserve(count);
    for (int i = 0; i < count; ++i)
        if (R[i].index >= 0) order.push_back(i);
    const int found = (int)order.size();
    std::sort(order.begin(), order.end(), [&](int a, int b) { return R[a].index < R[b].index; });
    for (int q = 0; q < found && q < cap; ++q) {
        const TracedRay &r = R[order[q]];
        const int n = r.n & 255;
        n_int[q] = (uint8_t)n;
        for (int j = 0; j < MAXI; ++j) {
            types[q * MAXI + j] = (uint8_t)((r.types >> (8 * j)) & 0xff);
            prims[q * MAXI + j] = j < n ? r.prims[j] : -1;
            s0[q * MAXI + j] = r.s[j];
        }
    }
    return found;
}

}  // namespace drt
