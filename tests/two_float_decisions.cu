// Random chains decided in two-float numbers and in FP64, as H's records and redone steps decide them.
// in:  most diffractions of a chain, extent (m), shortest leg (m), smallest grazing angle (rad), distance travelled until then (m), seed,
//      chains per length
// out: chains, decided in two-float numbers, of those rays, of those decided otherwise than in FP64, of those where FP64 has not converged
#include <cstdio>

#include "random_chains.cuh"

struct Counts { long all, decided, rays, wrong, unconverged; };

template <int N> void trial(int max_d, double S, double lmin, double gmin, double far, Counts &c) {
    Chain<N> x;
    if (!x.draw(max_d, S, lmin, gmin, far, 0.3)) return;
    const LinkDev &L = x.L;
    const double t = x.t;
    Prim<double> pd[N];
    Prim<ff> pq[N];
    for (int j = 0; j < N; ++j) {
        pd[j] = val_prim(load_prim_direct<double>(L, t, x.types[j], x.prims[j]));
        pq[j] = load_prim_ff_direct(L, ff(t), x.types[j], x.prims[j]);
    }
    v3<double> Vd[N + 2];
    v3<ff> Vq[N + 2];
    Vd[0] = val(terminal<double>(L.tx, t));
    Vd[N + 1] = val(terminal<double>(L.rx, t));
    Vq[0] = val(terminal_dual_ff(L.txq, ff(t)));
    Vq[N + 1] = val(terminal_dual_ff(L.rxq, ff(t)));
    uint32_t fd = 0, fq = 0;
    solve_geometry_any<N>(pd, Vd, x.s0, fd);
    fd |= validity<N>(pd, N, Vd);
    solve_geometry_any<N>(pq, Vq, x.s0, fq);
    fq |= validity<N>(pq, N, Vq, (float)ff_reach(x.H.view, t));
    ++c.all;
    for (int i = 1; i <= N; ++i)
        if (!std::isfinite(Vq[i].x.h)) return;
    // as in the records (path_step_ff) and in redone steps, whose flags are written out
    if ((fq & F_NOCONV) || ((fq & (F_REDO64 | F_DEGEN)) && !(fq & F_CLEAR))) return;
    ++c.decided;
    c.rays += fd == 0;
    const bool open = fq & F_REDO64;
    if ((open ? !fd : (fq & ~F_CLEAR) != fd)) {
        if (fd & F_NOCONV) ++c.unconverged;
        else ++c.wrong;
    }
}

int main() {
    double max_d, S, lmin, gmin, far, seed, n;
    while (std::scanf("%lf %lf %lf %lf %lf %lf %lf", &max_d, &S, &lmin, &gmin, &far, &seed, &n) == 7) {
        Counts c{};
        rng.seed((uint64_t)seed);
        for (long k = 0; k < (long)n; ++k) {
            trial<1>((int)max_d, S, lmin, gmin, far, c);
            trial<2>((int)max_d, S, lmin, gmin, far, c);
            trial<3>((int)max_d, S, lmin, gmin, far, c);
        }
        std::printf("%ld %ld %ld %ld %ld\n", c.all, c.decided, c.rays, c.wrong, c.unconverged);
    }
}
