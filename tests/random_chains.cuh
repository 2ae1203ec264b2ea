// Random chains close to their validity boundaries and to grazing, for programs that decide them on the host.
#pragma once
#include <random>

#include "drt_physics_ff.cuh"

using namespace drt;
typedef v3<double> V;

std::mt19937_64 rng;
double uniform(double a, double b) { return a + (b - a) * (rng() >> 11) * 0x1p-53; }
double log_uniform(double a, double b) { return std::exp(uniform(std::log(a), std::log(b))); }
bool coin() { return uniform(0, 1) < 0.5; }
double sign() { return coin() ? 1 : -1; }
V unit_of(V a) { return a * (1 / std::sqrt(dot(a, a))); }
V any_unit() {
    for (;;) {
        const V v = V3<double>(uniform(-1, 1), uniform(-1, 1), uniform(-1, 1));
        if (dot(v, v) > 0.01 && dot(v, v) < 1) return unit_of(v);
    }
}
V across(V u) { return unit_of(cross(u, any_unit())); }
void put(double *d, V v) {
    d[0] = v.x;
    d[1] = v.y;
    d[2] = v.z;
}

double NEAR = 1e-13;   // smallest margin drawn (m)

// a chain of N vertices whose points are known, with a primitive laid through each, and everything on its way so that it is there at t
template <int N> struct Chain {
    PackedLink H;
    LinkDev L;
    double t, s0[MAXI] = {0, 0, 0, 0};
    uint8_t types[MAXI] = {0, 0, 0, 0};
    int32_t prims[MAXI] = {-1, -1, -1, -1};

    // max_d: most diffractions; S: extent, lmin: shortest leg (m); gmin: smallest grazing angle (rad); far: what is travelled until t (m);
    // p_tile: share of tiles.  False where a wedge normal came out more than 1e-9 off its edge's perpendicular
    bool draw(int max_d, double S, double lmin, double gmin, double far, double p_tile) {
        drt_scene s{};
        drt_body b{};
        drt_material m{};
        b.k[2] = 1;
        m.eps_r = 3;
        s.bodies = &b;
        s.materials = &m;
        s.n_bodies = s.n_materials = 1;
        std::vector<drt_face> faces;
        std::vector<drt_edge> edges;
        std::vector<drt_tile> tiles;
        const uint8_t n_int = N;
        V P = V3<double>(uniform(-S, S), uniform(-S, S), uniform(-S, S)), u = any_unit();
        t = far > 0 ? 1.0 : 0.0;
        const V way = any_unit() * far;
        put(s.tx.r, P - way);
        for (int j = 0; j < N; ++j) {
            P = P + u * log_uniform(lmin, S);
            int kind = (int)uniform(0, 2.0 + p_tile);
            if (kind == 1 && (int)edges.size() == max_d) kind = 0;
            V w;
            if (kind == 0) {
                const double g = log_uniform(gmin, 1.5);
                const V n = unit_of(across(u) * std::cos(g) - u * std::sin(g)), a1 = across(n), a2 = cross(a1, n);
                w = u - n * (2 * dot(u, n));
                drt_face f{};
                f.hu = uniform(1, 20);
                f.hw = uniform(1, 20);
                const double mu = sign() * log_uniform(NEAR, 1), mw = coin() ? uniform(0.1, f.hw) : sign() * log_uniform(NEAR, 1);
                put(f.c, P + a1 * (sign() * (f.hu - mu)) + a2 * (sign() * (f.hw - mw)) - way);
                put(f.n, n);
                put(f.u, a1);
                types[j] = DRT_T_R;
                prims[j] = (int)faces.size();
                faces.push_back(f);
            } else if (kind == 1) {
                const double g = log_uniform(gmin, 1.5);
                const V e = unit_of(u * std::cos(g) + across(u) * std::sin(g)) * sign();
                V x = u - e * dot(u, e);
                const double r = std::sqrt(dot(x, x));
                x = unit_of(x);
                x = unit_of(x - e * dot(x, e));
                const V y = cross(e, x);
                auto around = [&](double a) { return x * std::cos(a) + y * std::sin(a); };
                w = e * dot(u, e) + around(coin() ? uniform(-3, 3) : sign() * log_uniform(NEAR / S, 3)) * r;
                const double len = uniform(2, 30), mu = coin() ? uniform(0.1, len) : sign() * log_uniform(NEAR, 1);
                const V a = P - e * (coin() ? mu : len - mu) - way;
                const V n0 = unit_of(around(coin() ? uniform(0, 6.28) : sign() * log_uniform(NEAR / S, 3)));
                drt_edge d{};
                d.wedge_n = coin() ? 1.5 : uniform(1.05, 1.99);
                const double q = (d.wedge_n - 1) * M_PI;
                put(d.a, a);
                put(d.b, a + e * len);
                put(d.n0, n0);
                put(d.nn, unit_of(n0 * std::cos(q) + cross(e, n0) * std::sin(q)));
                s0[j] = dot(P - way - a, e) + sign() * log_uniform(1e-6, 1);
                types[j] = DRT_T_D;
                prims[j] = (int)edges.size();
                edges.push_back(d);
            } else {
                w = any_unit();
                drt_tile q{};
                put(q.c, P - way);
                put(q.n, coin() ? unit_of(w - u) : unit_of(across(u) - u * log_uniform(gmin, 1)));
                q.area = 4;
                q.s = 0.3;
                q.alpha_r = 2;
                types[j] = DRT_T_S;
                prims[j] = (int)tiles.size();
                tiles.push_back(q);
            }
            u = w;
        }
        put(s.rx.r, P + u * log_uniform(lmin, S) - way);
        put(s.tx.v, way);
        put(s.rx.v, way);
        put(b.v, way);
        s.faces = faces.data();
        s.edges = edges.data();
        s.tiles = tiles.data();
        s.n_faces = (int)faces.size();
        s.n_edges = (int)edges.size();
        s.n_tiles = (int)tiles.size();
        drt_path_set ps{};
        ps.n_paths = 1;
        ps.n_int = &n_int;
        ps.types = types;
        ps.prims = prims;
        ps.s0 = s0;
        if (pack_link(&s, &ps, H)) return false;
        L = H.dev;
        L.bodies = H.bodies.data();
        L.faces = H.faces.data();
        L.edges = H.edges.data();
        L.tiles = H.tiles.data();
        L.facesQ = H.facesQ.data();
        L.edgesQ = H.edgesQ.data();
        L.tilesQ = H.tilesQ.data();
        L.bodiesQ = H.bodiesQ.data();
        L.body_fixed = H.body_fixed.data();
        return true;
    }
};
