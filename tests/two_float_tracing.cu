// Random candidates of the ray tracer, solved by its two-float pass (FP32 first) and in FP64, and the occlusion of their segments.
// in:  most diffractions of a chain, extent (m), shortest leg (m), smallest grazing angle (rad), distance travelled until then (m), smallest margin (m), seed,
//      chains per length
// out: candidates, decided by the two-float pass, of those rays, of those decided otherwise than in FP64, of those where FP64 has not
//      converged; (segment, face) pairs, decided in two-float numbers, of those otherwise than in FP64; candidates that FP32 discards, of
//      those whose FP32 points are further off than the bound it goes by, of those whose margin that bound reaches
#include <cstdio>

#include "drt_trace.cu"
#include "random_chains.cuh"

struct Counts { long all, decided, rays, wrong, unconverged, pairs, sure, differ, dropped, off, near; };

PosedFaceQ two_float(const PosedFace &F) {
    PosedFaceQ q;
    for (int j = 0; j < 3; ++j) {
        q.c[j] = ff_host(F.c[j]);
        q.n[j] = ff_host(F.n[j]);
        q.u[j] = ff_host(F.u[j]);
        q.w[j] = ff_host(F.w[j]);
    }
    q.hu = ff_host(F.hu);
    q.hw = ff_host(F.hw);
    return q;
}

// the chain's points in FP64
template <int N> std::vector<v3<double>> solved(const Chain<N> &x, const double *start, uint32_t &fl) {
    Prim<double> pd[N];
    for (int j = 0; j < N; ++j) pd[j] = val_prim(load_prim_direct<double>(x.L, x.t, x.types[j], x.prims[j]));
    std::vector<v3<double>> P(N + 2);
    P[0] = val(terminal<double>(x.L.tx, x.t));
    P[N + 1] = val(terminal<double>(x.L.rx, x.t));
    solve_geometry_any<N>(pd, P.data(), start, fl);
    return P;
}

template <int N> void trial(int max_d, double S, double lmin, double gmin, double far, Counts &c) {
    Chain<N> x;
    if (!x.draw(max_d, S, lmin, gmin, far, 0.0)) return;
    const LinkDev &L = x.L;
    const double t = x.t;
    const float reach = (float)ff_reach(x.H.view, t);
    std::vector<Prim<ff>> prims;
    for (int i = 0; i < L.n_faces; ++i) prims.push_back(load_prim_ff_direct(L, ff(t), T_R, i));
    for (int i = 0; i < L.n_edges; ++i) prims.push_back(load_prim_ff_direct(L, ff(t), T_D, i));
    int code[2] = {0, 0};
    for (int j = 0; j < N; ++j) code[j] = x.prims[j] + (x.types[j] == T_D ? L.n_faces : 0);
    TracedRay r{}, rd{};
    RayPoints v{};
    double start[MAXI] = {0, 0, 0, 0};
    for (int j = 0; j < N; ++j)
        if (x.types[j] == T_D) start[j] = 0.5 * L.edges[x.prims[j]].len;
    if constexpr (N == 2) {
        const Prim<ff> pr[2] = {prims[code[0]], prims[code[1]]};
        v3<ff> V[4];
        V[0] = val(terminal_dual_ff(L.txq, ff(t)));
        V[3] = val(terminal_dual_ff(L.rxq, ff(t)));
        Prim<float> pf[2];
        v3<float> Vf[4];
        uint32_t f0 = 0, fl = 0;
        const Fp32Check q = fp32_first(pr, V, start, pf, Vf, f0);
        const std::vector<v3<double>> P = solved<N>(x, start, fl);
        if (q.none && !(fl & F_NOCONV)) {
            double off = 0, scale = 0;
            for (int i = 1; i <= 2; ++i) {
                const v3<double> d = P[i] - V3<double>(Vf[i].x, Vf[i].y, Vf[i].z);
                off = std::fmax(off, std::sqrt(dot(d, d)));
            }
            for (int i = 0; i <= 3; ++i) scale = std::fmax(scale, (double)amax3(Vf[i]));
            for (int j = 0; j < 2; ++j) scale = std::fmax(scale, (double)amax3(pf[j].p));
            ++c.dropped;
            c.off += off > 0.125 * q.amp * (double)fp32_margin_tol((float)scale);
            c.near += !(q.margin > 0.125f * q.amp);
        }
    }
    const int state = trace_chain_ff<N>(L, t, reach, code, prims.data(), &r, &v);
    ++c.all;
    if (state == RAY_OPEN) return;
    ++c.decided;
    std::vector<v3<double>> P;   // the FP64 points, from the segments that the ray is made of
    const bool ray = trace_chain<N>(L, t, 1, code, &rd, [&](v3<double> A, v3<double> B) {
        if (P.empty()) P.push_back(A);
        P.push_back(B);
        return false;
    });
    c.rays += ray;
    if (ray != (state >= 0)) {
        uint32_t fl = 0;
        solved<N>(x, start, fl);
        if (fl & F_NOCONV) ++c.unconverged;
        else ++c.wrong;
        return;
    }
    if (!ray) return;
    const v3<ff> ends[2] = {val(terminal_dual_ff(L.txq, ff(t))), val(terminal_dual_ff(L.rxq, ff(t)))};
    for (int i = 0; i <= N; ++i)
        for (int f = 0; f < L.n_faces; ++f)
            for (int k = 0; k < 8; ++k) {
                PosedFace F;
                pose_face(L, t, f, &F);
                if (k) {   // a face of any slope to the segment's end, its rim close to where it is crossed
                    const V at = k & 1 ? P[i] : P[i + 1], n = k & 2 ? any_unit() : across(unit_of(P[i + 1] - P[i])), u = across(n);
                    const V w = cross(u, n), c0 = at + n * (sign() * log_uniform(NEAR, 1));
                    F.hu = uniform(1, 20);
                    F.hw = uniform(1, 20);
                    put(F.c, c0 + u * (sign() * (F.hu - sign() * log_uniform(NEAR, 1))) + w * uniform(-1, 1));
                    put(F.n, n);
                    put(F.u, u);
                    put(F.w, w);
                }
                const PosedFaceQ Q = two_float(F);
                const v3<float> n = f32v(vq(Q.n));
                auto up = [&](int j) { return height_amp(prims[code[j]], n, v.amp); };
                const int b = face_blocks_ff(Q, i == 0 ? ends[0] : vq(v.v[i - 1]), i == N ? ends[1] : vq(v.v[i]),
                                             i == 0 ? 1.f : up(i - 1), i == N ? 1.f : up(i), v.amp, reach);
                ++c.pairs;
                if (b < 0) continue;
                ++c.sure;
                c.differ += b != (int)face_blocks(F, P[i], P[i + 1]);
            }
}

int main() {
    double max_d, S, lmin, gmin, far, near, seed, n;
    while (std::scanf("%lf %lf %lf %lf %lf %lf %lf %lf", &max_d, &S, &lmin, &gmin, &far, &near, &seed, &n) == 8) {
        Counts c{};
        rng.seed((uint64_t)seed);
        NEAR = near;
        for (long k = 0; k < (long)n; ++k) {
            trial<1>((int)max_d, S, lmin, gmin, far, c);
            trial<2>((int)max_d, S, lmin, gmin, far, c);
        }
        std::printf("%ld %ld %ld %ld %ld %ld %ld %ld %ld %ld %ld\n", c.all, c.decided, c.rays, c.wrong, c.unconverged, c.pairs, c.sure,
                    c.differ, c.dropped, c.off, c.near);
    }
}
