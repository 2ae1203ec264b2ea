"""The workloads that the library's speed is measured on: what a program that uses it asks of it, through its public entry
points, from one small prediction to a batch of links.

Sizes and scenes are those of the repository's own workloads (inputs.py, bench.py, the tests): the 28 GHz tiny scene of 3
paths, the 60 GHz canyon of 512 chains, the 28 GHz road links of 8 to 2048 chains, the highway of 20300 chains at two
carriers, and the request mix of the serving loop.  `seed` draws what differs from one use to the next: the kinematics of the
terminals and vehicles (the scenes' own distributions; positions at t0 stay, so the committed chains are rays there), the
chains and their order, and the instants that predictions start at.

exact() restates the method in 64 bits with plain torch (image method and back-tracking, Keller cone, Newton on the unfolded
length for several diffractions in one stretch, Fresnel / UTD / effective roughness, the direct sum for H), for all outputs
that are computed numbers.
"""
import dataclasses
import functools
import math
import os

import numpy as np
import torch

from paper_2205_00237_gb300 import drt
from paper_2205_00237_gb300 import inputs as I

GOLD = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "tests", "golden")
PREC = {"fp64": drt.FP64, "bulk": drt.FP32_BULK}
CARRIER = {"tiny": (28e9, 400e6), "link": (28e9, 400e6), "canyon": (60e9, 1e9)}
C0, EPS0 = 299792458.0, 8.8541878128e-12


def listed():
    return [
        # the smallest prediction: 3 rays over a second; launches and latency are all of it
        dict(name="tiny_fp64", kind="synth", scene="tiny", paths=3, steps=1000, dt=1e-3, bins=256, prec="fp64"),
        # one short anticipative request: a link's 32 strongest chains over 50 ms
        dict(name="request_bulk", kind="synth", scene="canyon", paths=32, steps=50, dt=1e-3, bins=512, prec="bulk"),
        # the full canyon link over a second, both precisions (the benchmark's headline, and its FP32-bulk form)
        dict(name="canyon_fp64", kind="synth", scene="canyon", paths=512, steps=2000, dt=0.5e-3, bins=512, prec="fp64"),
        dict(name="canyon_bulk", kind="synth", scene="canyon", paths=512, steps=2000, dt=0.5e-3, bins=512, prec="bulk"),
        # per-path records (delay, amplitude, Doppler, angles, flags): a localisation or channel-sounding user
        dict(name="records_fp64", kind="records", scene="canyon", paths=512, steps=2000, dt=0.5e-3, prec="fp64"),
        dict(name="records_bulk", kind="records", scene="link", paths=2048, steps=1237, dt=1e-3, prec="bulk"),
        # the power-Doppler profile of the paper's comparison: 200 ms windows, 14.34 Hz bins
        dict(name="profile_bulk", kind="profile", scene="canyon", paths=512, steps=2000, dt=0.5e-3, prec="bulk",
             per_bin=400, bins=1116, x0=-8e3, dx=14.34, what="doppler"),
        # multipath-lifetime plan, then H over its windows
        dict(name="windows_fp64", kind="windows", scene="canyon", paths=512, steps=2000, dt=0.5e-3, bins=512, prec="fp64",
             share=1e-5, min_steps=20, max_steps=300),
        # ray tracing again at every window start, and H over the rays found: the paper's whole procedure
        dict(name="retraced_bulk", kind="retraced", scene="canyon", paths=32, steps=400, dt=0.5e-3, bins=512, prec="bulk",
             windows=2),
        # many links of very different sizes in one launch sequence (8 to 2048 chains, 100 to 5000 steps)
        dict(name="batch_128", kind="batch", links=128, bins=256, mix=0),
        # one highway link at its two carriers: the largest path set, the widest frequency grid
        dict(name="highway_pair", kind="highway", link=0, steps=500, bins=1024),
        # a burst of requests into the serving loop: links of 512, 128 and 32 chains, horizons of 50 to 500 ms
        dict(name="serve_burst", kind="serve", requests=48, bins=512, mix=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["synth"] * 4 + ["records", "records", "profile", "windows", "retraced", "batch", "highway", "serve"])
    prec = rng.choice(["fp64", "bulk"])
    if kind == "batch":
        return dict(kind=kind, links=_log(rng, 8, 128), bins=_log(rng, 64, 300), mix=rng.randrange(1, 1 << 16))
    if kind == "highway":
        return dict(kind=kind, link=rng.randrange(64), steps=_log(rng, 50, 500), bins=_log(rng, 256, 1024))
    if kind == "serve":
        return dict(kind=kind, requests=_log(rng, 1, 48), bins=_log(rng, 128, 512), mix=rng.randrange(1, 1 << 16))
    scene = rng.choice(["link", "canyon"])
    paths = _log(rng, 8, 2048 if scene == "link" else 512)
    steps = min(_log(rng, 50, 5000), 4000000 // paths)
    c = dict(kind=kind, scene=scene, paths=paths, steps=steps, dt=rng.choice([0.5e-3, 1e-3]), prec=prec)
    if kind == "records":
        return c
    if kind == "profile":
        if rng.random() < 0.5:
            return dict(c, per_bin=_log(rng, 20, 400), bins=_log(rng, 100, 1116), x0=-8e3, dx=14.34, what="doppler")
        return dict(c, per_bin=_log(rng, 20, 400), bins=_log(rng, 100, 2000), x0=0.0, dx=1e-9, what="delay")
    c["bins"] = _log(rng, 64, 1024)
    if kind == "windows":
        return dict(c, share=10.0 ** rng.uniform(-6, -3), min_steps=rng.randrange(1, 40), max_steps=rng.randrange(60, 400))
    if kind == "retraced":
        return dict(c, paths=32, steps=min(steps, 600), windows=rng.randrange(1, 4))
    return c


# ------------------------------------------------------------------------------------------------
# inputs

@functools.lru_cache(maxsize=8)
def _base(name, k):
    """Scene k of a workload as it stands at t0, and its committed chains.  Left out: the one chain in a thousand that joins a
    tile and an edge of the same facade.  The tile lies in the plane of the edge's wedge face, at distance 0 from the boundary
    that decides whether the chain is a ray, so the last bit of any arithmetic decides it, and an error of H could not be
    told from such a decision."""
    scene = {"tiny": I.scene_tiny, "link": I.scene_link, "canyon": I.scene_canyon}[name](k)
    paths = I.PathSet.from_npz(os.path.join(GOLD, "pathset_%s_seed%d.npz" % (name, k)))
    keep = np.ones(paths.n_paths, bool)
    for j in range(paths.types.shape[1] - 1):
        for s, d in ((j, j + 1), (j + 1, j)):
            p = np.nonzero((paths.types[:, s] == I.T_S) & (paths.types[:, d] == I.T_D))[0]
            tile, edge = scene.tiles[paths.prims[p, s]], scene.edges[paths.prims[p, d]]
            for n in ("n0", "nn"):
                keep[p[np.abs(((tile["c"] - edge["a"]) * edge[n]).sum(1)) < 1e-6]] = False
    return scene, paths.subset(np.nonzero(keep)[0])


@functools.lru_cache(maxsize=1)
def _highway_rd():
    return I.PathSet.from_npz(os.path.join(GOLD, "pathset_highway_rd_seed0.npz"))


def _moved(scene, rng, speed, acc, yaw):
    """The scene with its vehicles' speed, acceleration along the heading and yaw rate drawn anew.  A terminal that rode
    on a vehicle (same velocity) still does; one that drove by itself gets a speed within a fifth of its own."""
    bodies = scene.bodies.copy()
    term = {"tx": scene.tx.copy(), "rx": scene.rx.copy()}
    for b in range(1, len(bodies)):
        old = scene.bodies[b]
        head = old["v"] / np.linalg.norm(old["v"])
        bodies[b]["v"] = rng.uniform(*speed) * head
        bodies[b]["a"] = rng.uniform(*acc) * head
        bodies[b]["w0"] = rng.uniform(*yaw)
        for side, was in (("tx", scene.tx), ("rx", scene.rx)):
            near = np.linalg.norm((was["r"] - old["o"])[:2]) < 1e-9
            if near and np.array_equal(was["v"], old["v"]):
                term[side]["v"], term[side]["a"] = bodies[b]["v"], bodies[b]["a"]
    for side, was in (("tx", scene.tx), ("rx", scene.rx)):
        if np.array_equal(term[side]["v"], was["v"]):
            term[side]["v"] = was["v"] * rng.uniform(0.8, 1.2)
    return dataclasses.replace(scene, bodies=bodies, tx=term["tx"], rx=term["rx"])


KIN = {"tiny": ((12.0, 18.0), (0.0, 0.0), (0.0, 0.0)), "link": ((12.0, 18.0), (0.0, 0.0), (0.0, 0.0)),
       "canyon": ((5.0, 30.0), (-2.0, 2.0), (-0.3, 0.3)), "highway": ((20.0, 36.0), (-1.0, 1.0), (-0.02, 0.02))}


def _link_inputs(name, n_paths, rng, k=None):
    """One link of a workload: scene with new kinematics, and n_paths of its chains (the line of sight and others) in an
    order of their own."""
    k = int(rng.integers(4 if name == "link" else 2 if name == "tiny" else 1)) if k is None else k
    scene, paths = _base(name, k)
    idx = 1 + rng.permutation(paths.n_paths - 1)[:max(0, min(n_paths, paths.n_paths) - 1)]
    return _moved(scene, rng, *KIN[name]), paths.subset(rng.permutation(np.concatenate([[0], idx])))


def _inputs(case, seed):
    """(links, entries): the links' scenes and chains, and what is asked of them: (link, time grid, frequency grid)."""
    rng = np.random.default_rng([seed, 77])
    kind = case["kind"]
    if kind == "batch":
        links = [_link_inputs("link", 2048, rng, k) for k in range(I.LINK_SCENES)]
        B = I.BATCH
        entries = [(s, min(p, links[s][1].n_paths), I.TimeGrid(0.0, B["dt"], t), I.FreqGrid(B["fc"], B["bandwidth"], case["bins"]))
                   for s, p, t in I.batch_links(case["links"], case["mix"])]
        return links, entries
    if kind == "highway":
        scene = _moved(I.scene_highway(0, case["link"]), rng, *KIN["highway"])
        paths = I.highway_pathset(_highway_rd(), case["link"])
        tg = I.TimeGrid(0.0, I.HIGHWAY["dt"], case["steps"])
        return [(scene, paths)], [(0, paths.n_paths, tg, I.FreqGrid(f, I.HIGHWAY["bandwidth"], case["bins"]))
                                  for f in I.HIGHWAY["carriers"]]
    if kind == "serve":
        links = [_link_inputs("canyon", p, rng) for p in (512, 128, 32)]
        return links, [(s, links[s][1].n_paths, I.TimeGrid(float(rng.integers(1000)) * 1e-3, 1e-3, t),
                        I.FreqGrid(60e9, 1e9, case["bins"])) for s, t in _request_mix(case)]
    links = [_link_inputs(case["scene"], case["paths"], rng)]
    fc, bw = CARRIER[case["scene"]]
    return links, [(0, links[0][1].n_paths, I.TimeGrid(0.0, case["dt"], case["steps"]),
                    I.FreqGrid(fc, bw, case.get("bins", 1) if kind not in ("records", "profile") else 1))]


def _request_mix(case):
    rng = np.random.default_rng([case["mix"], 5])
    return [(int(s), int(t)) for s, t in zip(rng.choice(3, size=case["requests"], p=[0.6, 0.25, 0.15]),
                                             rng.integers(50, 501, case["requests"]))]


def _starts(case):
    """Window starts of a retraced span: equal windows."""
    return [case["steps"] * w // case["windows"] for w in range(case["windows"])]


_CTX = []


def _ctx():
    """The program's one context."""
    if not _CTX:
        _CTX.append(drt.Context(0))
    return _CTX[0]


class _State:
    """What a program keeps: loaded links, a batch plan, output buffers."""

    def __init__(self, case):
        self.case, self.links, self.plan = case, [], None

    def __del__(self):
        try:
            if self.plan is not None:
                self.plan.close()
            for lk in self.links:
                lk.unload()
        except Exception:
            pass


def _flat(entries):
    """One buffer for all entries' H, and the views the entries write."""
    n = [tg.n_steps * fg.n_bins for _, _, tg, fg in entries]
    flat = torch.empty(sum(n), dtype=torch.complex64, device="cuda")
    return flat, [v.view(tg.n_steps, fg.n_bins) for v, (_, _, tg, fg) in zip(flat.split(n), entries)]


def prepare(case, seed):
    links, entries = _inputs(case, seed)
    ctx, S, kind = _ctx(), _State(case), case["kind"]
    S.entries = entries
    S.prec = PREC[case.get("prec", "bulk")]
    if kind == "batch":   # entry i: the first p chains of its scene
        S.links = [ctx.load(links[s][0], links[s][1].subset(np.arange(p))) for s, p, _, _ in entries]
        S.flat, S.H = _flat(entries)
        S.plan = ctx.batch(S.links, [e[2] for e in entries], [e[3] for e in entries], S.H)
    else:
        S.links = [ctx.load(sc, ps) for sc, ps in links]
        if kind in ("highway", "serve"):
            S.flat, S.H = _flat(entries)
        if kind == "highway":
            S.plan = ctx.batch([S.links[0]] * 2, [e[2] for e in entries], [e[3] for e in entries], S.H)
        if kind in ("synth", "windows", "retraced"):
            S.flat, (S.H,) = _flat(entries)
    return S


def run(S):
    case, kind = S.case, S.case["kind"]
    _, _, tg, fg = S.entries[0]
    if kind == "synth":
        return S.links[0].synthesize_H(tg, fg, S.prec, H=S.H)
    if kind == "records":
        return S.links[0].extrapolate(tg, fg, S.prec)
    if kind == "profile":
        what = drt.PP_DOPPLER if case["what"] == "doppler" else drt.PP_DELAY
        return S.links[0].power_profile(tg, fg, case["per_bin"], case["x0"], case["dx"], case["bins"], what, S.prec)
    if kind == "windows":
        starts, major = S.links[0].lifetime_windows(tg, fg, case["share"], case["min_steps"], case["max_steps"], S.prec)
        H = S.links[0].synthesize_H_windows(tg, fg, starts, S.prec, H=S.H)
        return {"starts": np.array(starts + [-1] * (case["steps"] - len(starts))), "major": major, "H": H}
    if kind == "retraced":
        return S.links[0].synthesize_H_retraced(tg, fg, _starts(case), precision=S.prec, H=S.H)
    if kind in ("batch", "highway"):
        S.plan.run()
        return S.flat
    ctx = S.links[0].ctx
    tickets = [ctx.submit(S.links[s], g, f, H) for (s, _, g, f), H in zip(S.entries, S.H)]
    for t in tickets:
        if ctx.wait(t)["status"] != 0:
            raise RuntimeError("request failed")
    return S.flat


def work(case):
    """Scene and chains read once, outputs written once; about 1000 operations for the geometry and field of a path-step
    and 8 for a term of H."""
    kind = case["kind"]
    if kind in ("batch", "serve"):
        sizes = [(p, t) for _, p, t in I.batch_links(case["links"], case["mix"])] if kind == "batch" else \
            [((512, 128, 32)[s], t) for s, t in _request_mix(case)]
        ps = sum(p * t for p, t in sizes)
        out = 8 * case["bins"] * sum(t for _, t in sizes)
        chains = sum(p for p, _ in sizes) if kind == "batch" else 672
        return {"bytes": out + 200 * chains, "flops": ps * (1000 + 8 * case["bins"])}
    if kind == "highway":
        n, t, f = 20300, case["steps"], case["bins"]
        return {"bytes": 2 * 8 * t * f + 200 * n, "flops": n * t * (400 + 2 * (600 + 8 * f))}
    n, t, f = case["paths"], case["steps"], case.get("bins", 0)
    if kind == "retraced":   # some 5000 rays, each window's candidates solved once
        return {"bytes": 8 * t * f + 5e3 * 200, "flops": 5e3 * t * (1000 + 8 * f) + case["windows"] * 1e5 * 500}
    if kind == "records":
        size = 8 + (24 if case["prec"] == "fp64" else 12) + 16 + 1
        return {"bytes": n * t * size + 200 * n, "flops": 1500 * n * t}
    if kind == "profile":
        return {"bytes": 8 * f * -(-t // case["per_bin"]) + 200 * n, "flops": 1500 * n * t}
    return {"bytes": 8 * t * f + 200 * n, "flops": n * t * (1000 + 8 * f) * (1 if kind == "synth" else 2)}


# ------------------------------------------------------------------------------------------------
# the same outputs in 64 bits, from the method alone (plain torch)

def _dot(a, b):
    return (a * b).sum(-1)


def _unit(a):
    return a / _dot(a, a).sqrt()[..., None]


def _cross(a, b):
    return torch.linalg.cross(a, b, dim=-1)


class _World:
    """A scene's primitives at instants t [T]: poses of the bodies, primitives of chain vertices [T, G, 3]."""

    def __init__(self, scene, dev):
        self.s, self.dev = scene, dev

    def const(self, a):
        return torch.as_tensor(np.ascontiguousarray(a), device=self.dev)

    def terminal(self, m, t):
        t = t[:, None, None]
        return self.const(m["r"]) + self.const(m["v"]) * t + 0.5 * self.const(m["a"]) * t * t

    def body(self, b, t):
        """Rotation [T, G, 3, 3] and reference point [T, G, 3] of the bodies b [G]."""
        B = {k: self.const(self.s.bodies[k][b]) for k in ("o", "v", "a", "k", "w0", "wdot")}
        t1 = t[:, None]
        th = B["w0"] * t1 + 0.5 * B["wdot"] * t1 * t1
        k = B["k"]
        z = torch.zeros_like(k[:, 0])
        K = torch.stack([z, -k[:, 2], k[:, 1], k[:, 2], z, -k[:, 0], -k[:, 1], k[:, 0], z], -1).view(-1, 3, 3)
        R = torch.eye(3, dtype=t.dtype, device=t.device) + th.sin()[..., None, None] * K \
            + (1 - th.cos())[..., None, None] * (K @ K)
        t2 = t1[..., None]
        return R, B["o"] + B["v"] * t2 + 0.5 * B["a"] * t2 * t2

    def vertex(self, ty, idx, t):
        table = {I.T_R: self.s.faces, I.T_D: self.s.edges, I.T_S: self.s.tiles}[ty][idx]
        R, O = self.body(table["body"], t)
        o = self.s.bodies["o"][table["body"]]
        rot = lambda d: (R @ self.const(d)[..., None])[..., 0]   # noqa: E731
        q = {"ty": ty, "mat": table["material"], "row": table}
        if ty == I.T_D:
            e = table["b"] - table["a"]
            q["len"] = np.linalg.norm(e, axis=1)
            e = e / q["len"][:, None]
            q["len"] = self.const(q["len"])
            q.update(p=O + rot(table["a"] - o), a=rot(e), b=rot(np.cross(table["n0"], e)), c=rot(table["n0"]))
        else:
            q.update(p=O + rot(table["c"] - o), a=rot(table["n"]))
            if ty == I.T_R:
                q["b"] = rot(table["u"])
        return q


def _mirror(X, q):
    return X - 2 * _dot(X - q["p"], q["a"])[..., None] * q["a"]


def _mirror_dir(d, q):
    return d - 2 * _dot(d, q["a"])[..., None] * q["a"]


def _keller(S, R, q):
    wa, wb = S - q["p"], R - q["p"]
    sa, sb = _dot(wa, q["a"]), _dot(wb, q["a"])
    ra = _dot(wa - q["a"] * sa[..., None], wa - q["a"] * sa[..., None]).sqrt()
    rb = _dot(wb - q["a"] * sb[..., None], wb - q["a"] * sb[..., None]).sqrt()
    return sa + (sb - sa) * ra / (ra + rb)


def _newton(A, E, S, R, s0):
    """Edge parameters that make the length S -> edges (A_i + s_i E_i) -> R stationary (convex): damped Newton, the
    tridiagonal system solved by elimination."""
    m = len(A)
    s = [x for x in s0]

    def legs(s):
        X = [S] + [A[i] + E[i] * s[i][..., None] for i in range(m)] + [R]
        d = [X[i + 1] - X[i] for i in range(m + 1)]
        return d, [_dot(x, x).sqrt() for x in d]

    for _ in range(40):
        d, ln = legs(s)
        u = [x / y[..., None] for x, y in zip(d, ln)]
        g = [_dot(u[i] - u[i + 1], E[i]) for i in range(m)]
        h = [(1 - _dot(u[i], E[i]) ** 2) / ln[i] + (1 - _dot(u[i + 1], E[i]) ** 2) / ln[i + 1] for i in range(m)]
        o = [(_dot(u[i + 1], E[i]) * _dot(u[i + 1], E[i + 1]) - _dot(E[i], E[i + 1])) / ln[i + 1] for i in range(m - 1)]
        cp, dp = [], []
        for i in range(m):
            den = h[i] - (o[i - 1] * cp[-1] if i else 0.0)
            dp.append((-g[i] - (o[i - 1] * dp[-1] if i else 0.0)) / den)
            cp.append(o[i] / den if i < m - 1 else None)
        x = [None] * m
        for i in reversed(range(m)):
            x[i] = dp[i] - (cp[i] * x[i + 1] if i < m - 1 else 0.0)
        total = sum(ln)
        f = torch.ones_like(total)
        for _ in range(4):   # a step that lengthens the path is shortened
            longer = sum(legs([s[i] + f * x[i] for i in range(m)])[1]) > total + 1e-9
            f = torch.where(longer, f * 0.25, f)
        s = [s[i] + f * x[i] for i in range(m)]
    return s


def _points(W, chain, s0, t):
    """Vertices V_0 .. V_{n+1} [T, G, 3] of chains of one signature at t, and their posed primitives."""
    pr = [W.vertex(ty, idx, t) for ty, idx in chain]
    n = len(pr)
    G = len(chain[0][1]) if n else 1
    tx, rx = (W.terminal(m, t).expand(len(t), G, 3) for m in (W.s.tx, W.s.rx))
    V = [tx] + [q["p"] if q["ty"] == I.T_S else None for q in pr] + [rx]
    ends = [0] + [i + 1 for i, q in enumerate(pr) if q["ty"] == I.T_S] + [n + 1]
    for a, b in zip(ends, ends[1:]):
        D = [i for i in range(a + 1, b) if pr[i - 1]["ty"] == I.T_D]
        walls = {i: [pr[k - 1] for k in range(a + 1, i) if pr[k - 1]["ty"] == I.T_R] for i in D + [b]}

        def unfold(X, ws, f):
            for q in reversed(ws):
                X = f(X, q)
            return X

        if len(D) == 1:
            S = V[a]
            for q in walls[D[0]]:
                S = _mirror(S, q)
            back = [pr[k - 1] for k in range(D[0] + 1, b)]
            V[D[0]] = pr[D[0] - 1]["p"] + pr[D[0] - 1]["a"] * _keller(S, unfold(V[b], back, _mirror), pr[D[0] - 1])[..., None]
        elif D:
            A = [unfold(pr[i - 1]["p"], walls[i], _mirror) for i in D]
            E = [unfold(pr[i - 1]["a"], walls[i], _mirror_dir) for i in D]
            s = _newton(A, E, V[a], unfold(V[b], walls[b], _mirror), [s0[i - 1].expand(len(t), G) for i in D])
            for i, si in zip(D, s):
                V[i] = pr[i - 1]["p"] + pr[i - 1]["a"] * si[..., None]
        known = [a] + D + [b]
        for u, v in zip(known, known[1:]):   # reflection points, from the right
            img = [V[u]]
            for k in range(u + 1, v):
                img.append(_mirror(img[-1], pr[k - 1]))
            nxt = V[v]
            for k in reversed(range(u + 1, v)):
                q, src = pr[k - 1], img[k - u - 1]
                hs, hr = _dot(src - q["p"], q["a"]), _dot(nxt - q["p"], q["a"])
                Q = src + (nxt - src) * (hs / (hs + hr))[..., None]
                V[k] = nxt = Q - q["a"] * _dot(Q - q["p"], q["a"])[..., None]
    return V, pr


def _valid(W, V, pr):
    """Whether the chain is a ray: points on their faces and edges, neighbours on the lit sides."""
    ok = torch.ones(V[0].shape[:2], dtype=torch.bool, device=W.dev)
    for a, b in zip(V, V[1:]):
        ok = ok & (_dot(b - a, b - a) >= 1e-18)
    for i, q in enumerate(pr, 1):
        if q["ty"] == I.T_R:
            r = V[i] - q["p"]
            ok = ok & (_dot(r, q["b"]).abs() <= W.const(q["row"]["hu"])) & \
                (_dot(r, _cross(q["b"], q["a"])).abs() <= W.const(q["row"]["hw"]))
        if q["ty"] != I.T_D:
            ok = ok & (_dot(V[i - 1] - q["p"], q["a"]) > 0) & (_dot(V[i + 1] - q["p"], q["a"]) > 0)
        else:
            s = _dot(V[i] - q["p"], q["a"])
            ok = ok & (s >= 0) & (s <= q["len"])
            for X in (V[i - 1], V[i + 1]):
                ph = torch.atan2(_dot(X - V[i], q["c"]), _dot(X - V[i], q["b"]))
                ph = torch.where(ph < 0, ph + 2 * math.pi, ph)
                ok = ok & (ph > 0) & (ph < W.const(q["row"]["wedge_n"]) * math.pi)
    return ok


def _transition(X):
    """UTD transition function sqrt(pi X) e^{j pi/4} erfcx(e^{j pi/4} sqrt X): series, continued fraction, asymptotic."""
    F = torch.zeros(X.shape, dtype=torch.complex128, device=X.device)
    rot = complex(math.sqrt(0.5), math.sqrt(0.5))
    lo, hi = (X > 0) & (X < 4), X >= 40
    mid = (X >= 4) & ~hi
    x = X[lo]
    if len(x):
        z, jx = rot * x.sqrt().to(F.dtype), 1j * x
        term, acc = torch.ones_like(z), torch.ones_like(z)
        for k in range(1, 60):
            term = -term * jx / k
            acc = acc + term / (2 * k + 1)
        F[lo] = math.sqrt(math.pi) * z * torch.exp(jx) * (1 - z * acc * 2 / math.sqrt(math.pi))
    x = X[mid]
    if len(x):
        z = rot * x.sqrt().to(F.dtype)
        f = z
        for k in range(130, 0, -1):
            f = z + 0.5 * k / f
        F[mid] = z / f
    x = X[hi]
    if len(x):
        term = torch.ones(x.shape, dtype=F.dtype, device=X.device)
        acc = term
        for k in range(1, 30):
            new = term * (-(2 * k - 1)) / (2j * x)
            term = torch.where(new.abs() < term.abs(), new, torch.zeros_like(new))
            acc = acc + term
        F[hi] = acc
    return F


def _fresnel(W, q, fc, ct):
    m = W.s.materials[q["mat"]]
    ec = W.const(m["eps_r"] - 1j * m["sigma"] / (2 * math.pi * fc * EPS0))
    sq = (ec - 1 + ct * ct).sqrt()
    te, tm = (ct - sq) / (ct + sq), (ec * ct - sq) / (ec * ct + sq)
    pec = W.const(m["pec"] != 0)
    one = torch.ones_like(te)
    return torch.where(pec, -one, te), torch.where(pec, one, tm)


def _er_norm(alpha, ct):
    """Integral of ((1 + cos psi) / 2)^alpha over the hemisphere (a polynomial: the quadrature is exact for alpha <= 6)."""
    st = (1 - ct * ct).clamp(min=0).sqrt()
    acc = torch.zeros_like(ct)
    x, w = np.polynomial.legendre.leggauss(8)
    for z, wz in zip(0.5 * (x + 1), 0.5 * w):
        for j in range(8):
            c = z * ct + math.sqrt(1 - z * z) * math.cos(math.pi * j / 4) * st
            acc = acc + wz * (2 * math.pi / 8) * (0.5 * (1 + c)) ** alpha
    return acc


def _vertical(k):
    z = torch.zeros_like(k)
    z[..., 2] = 1
    p = z - k * k[..., 2:]
    return _unit(p)


def _amplitude(W, V, pr, fc):
    """lambda / 4 pi x spreading x polarimetric chain of Fresnel, UTD and effective-roughness factors."""
    n = len(pr)
    seg = [b - a for a, b in zip(V, V[1:])]
    ln = [_dot(x, x).sqrt() for x in seg]
    kd = [x / y[..., None] for x, y in zip(seg, ln)]   # kd[i]: vertex i to i + 1
    k = 2 * math.pi * fc / C0
    rays = torch.ones_like(ln[0])
    nxt, acc = {}, 0.0   # distance from each diffraction to the next one or the next point source
    for i in range(n, 0, -1):
        acc = acc + ln[i]
        if pr[i - 1]["ty"] != I.T_R:
            nxt[i], acc = acc, 0.0
    Lf, d, after, re, X1 = {}, 0.0, False, None, None
    for i in range(1, n + 2):
        d = d + ln[i - 1]
        ty = pr[i - 1]["ty"] if i <= n else I.T_S
        if ty == I.T_R:
            X1 = _mirror_dir(X1, pr[i - 1]) if after else X1
            continue
        rays = rays * ((re / (d * (re + d))).sqrt() if after else 1 / d)
        if ty == I.T_S:
            d, after = 0.0, False
            continue
        e, s = pr[i - 1]["a"], nxt[i]
        if after:
            u = e - kd[i - 1] * _dot(e, kd[i - 1])[..., None]
            cg2 = _dot(u, X1) ** 2 / _dot(u, u)
            r1, r2 = d, re + d
            rhe = 1 / (cg2 / r1 + (1 - cg2) / r2)
        else:
            r1 = r2 = rhe = d
        Lf[i] = s * (rhe + s) * r1 * r2 / (rhe * (r1 + s) * (r2 + s))
        X1, re, after, d = _unit(_cross(e, kd[i])), rhe, True, 0.0
    cdot = lambda E, v: (E * v).sum(-1)   # noqa: E731
    E = _vertical(kd[0]).to(torch.complex128)
    for i, q in enumerate(pr, 1):
        kin, kout = kd[i - 1], kd[i]
        if q["ty"] == I.T_R:
            nf = -q["a"] * _dot(q["a"], kin).sign()[..., None]
            ct = -_dot(nf, kin)
            ep = _unit(_cross(kin, nf))
            te, tm = _fresnel(W, q, fc, ct)
            rough = W.const(np.sqrt(1 - W.s.materials[q["mat"]]["rough_s"] ** 2))
            E = (rough * te * cdot(E, ep))[..., None] * ep + (rough * tm * cdot(E, _cross(ep, kin)))[..., None] * _cross(ep, kout)
        elif q["ty"] == I.T_D:
            e, wn = q["a"], W.const(q["row"]["wedge_n"])
            ang = lambda v: torch.remainder(torch.atan2(_dot(v, q["c"]), _dot(v, q["b"])), 2 * math.pi)   # noqa: E731
            phi, phip, sb = ang(kout), ang(-kin), _dot(_cross(kin, e), _cross(kin, e)).sqrt()
            kL = k * Lf[i] * sb * sb

            def term(sign, beta):
                N = torch.round((math.pi + sign * beta) / (2 * math.pi * wn))
                eps = math.pi + sign * beta - 2 * math.pi * wn * N
                return _transition(2 * kL * torch.sin(0.5 * eps) ** 2) / torch.tan(eps / (2 * wn))

            r0, rn = _fresnel(W, q, fc, phip.sin().abs()), _fresnel(W, q, fc, (wn * math.pi - phi).sin().abs())
            t1, t2, t3, t4 = term(1, phi - phip), term(-1, phi - phip), term(-1, phi + phip), term(1, phi + phip)
            Cc = -complex(math.sqrt(0.5), -math.sqrt(0.5)) / (2 * wn * math.sqrt(2 * math.pi * k) * sb)
            Ds, Dh = (Cc * (t1 + t2 + a * t3 + b * t4) for a, b in zip(r0, rn))
            php, ph = -_unit(_cross(e, kin)), _unit(_cross(e, kout))
            E = (-Ds * cdot(E, _cross(php, kin)))[..., None] * _cross(ph, kout) + (-Dh * cdot(E, php))[..., None] * ph
        else:
            nt = -q["a"] * _dot(q["a"], kin).sign()[..., None]
            ct = -_dot(nt, kin)
            cpsi = _dot(kin + 2 * ct[..., None] * nt, kout)
            alpha, S, area, phase = (W.const(q["row"][x]) for x in ("alpha_r", "s", "area", "phase"))
            amp = S * (area * ct / _er_norm(alpha, ct)).sqrt() * (0.5 * (1 + cpsi)) ** (0.5 * alpha)
            nE = (E.abs() ** 2).sum(-1).sqrt()
            E = E - cdot(E, kout)[..., None] * kout
            E = E * (nE / (E.abs() ** 2).sum(-1).sqrt() * amp * torch.exp(1j * phase))[..., None]
    return C0 / fc / (4 * math.pi) * rays * cdot(E, _vertical(kd[n]))


def _groups(paths):
    """Chains by signature: (indices, types)."""
    code = (paths.types.astype(np.int64) * (1 << np.array([0, 8, 16, 24]))).sum(1)
    for c in np.unique(code):
        idx = np.nonzero(code == c)[0]
        yield idx, [int(x) for x in paths.types[idx[0]] if x]


def _rays(scene, paths, t, fcs, dev, rates=False, fields=True):
    """tau [T, P], valid, amplitude per carrier and, asked for, Doppler shift and angles, in 64 bits."""
    W, T, P = _World(scene, dev), len(t), paths.n_paths
    tau = torch.empty((T, P), dtype=torch.float64, device=dev)
    ok = torch.empty((T, P), dtype=torch.bool, device=dev)
    amp = [torch.empty((T, P), dtype=torch.complex128, device=dev) for _ in fcs]
    fd, ang = torch.empty_like(tau), torch.empty((T, P, 4), dtype=torch.float64, device=dev) if rates else None
    for idx, types in _groups(paths):
        chain = [(ty, paths.prims[idx, j]) for j, ty in enumerate(types)]
        s0 = [W.const(paths.s0[idx, j]) for j in range(len(types))]
        at = torch.as_tensor(idx, device=dev)
        step = max(1, 400000 // len(idx))
        for a in range(0, T, step):
            tt, rows = t[a:a + step], slice(a, min(T, a + step))
            V, pr = _points(W, chain, s0, tt)
            seg = [y - x for x, y in zip(V, V[1:])]
            tau[rows, at] = sum(_dot(x, x).sqrt() for x in seg) / C0
            ok[rows, at] = _valid(W, V, pr)
            for A, fc in zip(amp, fcs if fields else ()):
                A[rows, at] = _amplitude(W, V, pr, fc)
            if rates:
                _, dV = torch.func.jvp(lambda x: tuple(_points(W, chain, s0, x)[0]), (tt,), (torch.ones_like(tt),))
                ks = [_unit(x) for x in seg]
                lg = sum(torch.log1p(-_dot(dV[i + 1], k) / C0) - torch.log1p(-_dot(dV[i], k) / C0) for i, k in enumerate(ks))
                fd[rows, at] = fcs[0] * torch.expm1(lg)
                for j, k in ((0, ks[0]), (2, -ks[-1])):
                    ang[rows, at, j] = torch.atan2(k[..., 1], k[..., 0])
                    ang[rows, at, j + 1] = torch.atan2(k[..., 2], torch.hypot(k[..., 0], k[..., 1]))
    return tau, ok, amp, fd, ang


def _sum_H(tau, a, fg):
    """sum_p a_p exp(-j 2 pi f_k tau_p): bins k = 32 u + v, a product of exponentials in u and in v."""
    T, P = tau.shape
    df, f0 = fg.bandwidth / fg.n_bins, fg.fc - 0.5 * fg.bandwidth
    nu = -(-fg.n_bins // 32)
    H = torch.empty((T, nu * 32), dtype=torch.complex128, device=tau.device)
    cis = lambda cyc: torch.polar(torch.ones_like(cyc), -2 * math.pi * (cyc - cyc.floor()))   # noqa: E731
    u, v = (torch.arange(m, dtype=tau.dtype, device=tau.device) for m in (nu, 32))
    step = max(1, 8000000 // (max(P, 1) * (nu + 32)))
    for r in range(0, T, step):
        x = tau[r:r + step, :, None]
        E1 = (a[r:r + step, :, None] * cis(f0 * x)) * cis(32 * df * u * x)
        H[r:r + step] = torch.einsum("tpu,tpv->tuv", E1, cis(df * v * x)).reshape(x.shape[0], -1)
    return H[:, :fg.n_bins]


def _times(tg, dev):
    return tg.t_start + tg.dt * torch.arange(tg.n_steps, dtype=torch.float64, device=dev)


def _traced(scene, t, dev):
    """The rays of a ray-tracing run at t: chains of at most two faces and edges and single tiles, solved, valid and not
    blocked by a face."""
    nf, ne, nt = len(scene.faces), len(scene.edges), len(scene.tiles)
    W, tt = _World(scene, dev), torch.full((1,), t, dtype=torch.float64, device=dev)
    F = W.vertex(I.T_R, np.arange(nf), tt)
    size = {I.T_R: nf, I.T_D: ne, I.T_S: nt}
    half = 0.5 * np.linalg.norm(scene.edges["b"] - scene.edges["a"], axis=1)
    found = []
    for types in [[], [I.T_R], [I.T_D], [I.T_S]] + [[x, y] for x in (I.T_R, I.T_D) for y in (I.T_R, I.T_D)]:
        ix = [g.reshape(-1) for g in np.meshgrid(*[np.arange(size[x]) for x in types], indexing="ij")]
        if len(types) == 2 and types[0] == types[1]:
            ix = [g[np.not_equal(*ix)] for g in ix]
        n = len(ix[0]) if types else 1
        s0 = [W.const(half[g]) if x == I.T_D else torch.zeros(n, dtype=torch.float64, device=dev) for x, g in zip(types, ix)]
        V, pr = _points(W, list(zip(types, ix)), s0, tt)
        ok = _valid(W, V, pr)[0]
        for A, B in zip(V, V[1:]):
            ha, hb = (_dot(X[0, :, None] - F["p"][0], F["a"][0]) for X in (A, B))
            r = A[0, :, None] + (B - A)[0, :, None] * (ha / (ha - hb))[..., None] - F["p"][0]
            inside = (_dot(r, F["b"][0]).abs() <= W.const(F["row"]["hu"])) & \
                (_dot(r, _cross(F["b"], F["a"])[0]).abs() <= W.const(F["row"]["hw"]))
            hit = inside & (ha.abs() >= 1e-9) & (hb.abs() >= 1e-9) & ((ha > 0) != (hb > 0))
            ok = ok & ~hit.any(1)
        keep = torch.nonzero(ok)[:, 0].cpu().numpy()
        ps = I.empty_paths(len(keep))
        ps.n_int[:] = len(types)
        for j, x in enumerate(types):
            ps.types[:, j], ps.prims[:, j] = x, ix[j][keep]
            if x == I.T_D:
                ps.s0[:, j] = _dot(V[j + 1] - pr[j]["p"], pr[j]["a"])[0].cpu().numpy()[keep]
        found.append(ps)
    return I.PathSet.concat(found)


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    links, entries = _inputs(case, seed)
    kind = case["kind"]
    _, _, tg, fg = entries[0]
    t = _times(tg, dev)
    if kind in ("batch", "serve"):   # all instants of a link at once; the entries are ranges of them
        H = [None] * len(entries)
        for s, (scene, paths) in enumerate(links):
            mine = [i for i, e in enumerate(entries) if e[0] == s]
            if not mine:
                continue
            if kind == "batch":
                P = max(entries[i][1] for i in mine)
                grid = _times(max((entries[i][2] for i in mine), key=lambda g: g.n_steps), dev)
                at = [0] * len(mine)
            else:
                P, ts = paths.n_paths, [_times(entries[i][2], dev) for i in mine]
                grid, at = torch.cat(ts), np.cumsum([0] + [len(x) for x in ts])
            tau, ok, (a,), _, _ = _rays(scene, paths.subset(np.arange(P)), grid, [entries[mine[0]][3].fc], dev)
            a = torch.where(ok, a, torch.zeros_like(a))
            for i, k in zip(mine, at):
                _, p, g, f = entries[i]
                H[i] = _sum_H(tau[k:k + g.n_steps, :p], a[k:k + g.n_steps, :p], f).reshape(-1)
        return torch.cat(H)
    scene, paths = links[0]
    if kind == "highway":
        H = []
        tau, ok, amps, _, _ = _rays(scene, paths, t, [e[3].fc for e in entries], dev)
        for a, e in zip(amps, entries):
            H.append(_sum_H(tau, torch.where(ok, a, torch.zeros_like(a)), e[3]).reshape(-1))
        return torch.cat(H)
    if kind == "retraced":
        H, starts = [], _starts(case) + [tg.n_steps]
        for a, b in zip(starts, starts[1:]):
            ps = _traced(scene, float(t[a]), dev)
            tau, ok, (A,), _, _ = _rays(scene, ps, t[a:b], [fg.fc], dev)
            H.append(_sum_H(tau, torch.where(ok, A, torch.zeros_like(A)), fg))
        return torch.cat(H)
    tau, ok, (a,), fd, ang = _rays(scene, paths, t, [fg.fc], dev, rates=kind in ("records", "profile"))
    power = torch.where(ok, a.abs() ** 2, torch.zeros_like(tau))
    if kind == "synth":
        return _sum_H(tau, torch.where(ok, a, torch.zeros_like(a)), fg)
    if kind == "records":
        # a road link's terminals lie in the plane y = 0, where an azimuth of -pi and one of pi are the same direction
        return {"tau": tau, "amp": torch.view_as_real(a), "doppler": fd, "flags": None,
                "angles": ang if case["scene"] == "canyon" else None}
    if kind == "profile":
        x = fd if case["what"] == "doppler" else tau
        j = torch.floor((x - case["x0"]) / case["dx"])
        j = torch.where((j >= 0) & (j < case["bins"]), j, torch.full_like(j, -1)).to(torch.int64)
        row = torch.arange(tg.n_steps, device=dev)[:, None] // case["per_bin"]
        n = -(-tg.n_steps // case["per_bin"])
        out = torch.zeros(n * case["bins"], dtype=torch.float64, device=dev)
        keep = ok & (j >= 0)
        out.index_add_(0, (row * case["bins"] + j)[keep], power[keep])
        return out.view(n, case["bins"])
    # windows: a major change is a chain of at least `share` of the power appearing or disappearing
    total = power.sum(1)
    big = power >= case["share"] * total[:, None]
    ch = ok[1:] != ok[:-1]
    major = torch.zeros(tg.n_steps, dtype=torch.bool, device=dev)
    major[1:] = (ch & torch.where(ok[1:], big[1:], big[:-1])).any(1)
    mj, starts = major.cpu().numpy(), [0]
    while True:
        s = starts[-1]
        nxt = next((k for k in range(s + case["min_steps"], min(s + case["max_steps"], tg.n_steps - 1) + 1) if mj[k]),
                   s + case["max_steps"])
        if nxt >= tg.n_steps:
            break
        starts.append(nxt)
    first = torch.as_tensor(np.array(starts)[np.searchsorted(starts, np.arange(tg.n_steps), side="right") - 1], device=dev)
    a = torch.where(ok & ok[first], a, torch.zeros_like(a))
    return {"starts": None, "major": None, "H": _sum_H(tau, a, fg)}
