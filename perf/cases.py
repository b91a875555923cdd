"""What users of this framework have it do, as measurable cases.

A program describes grains (``inputs.Workload``), binds a ``Simulation`` to the
GPU, advances it a window of time steps and reads the state back; beside that
it samples energies, restarts from stored states, steps aggregates on the
learned surrogate and trains or evaluates the surrogate's networks (``MLP``).
Each case is one such call with the state left on the GPU, where a program that
goes on working with it (a viewer, a data set of trajectories) wants it.

The FP64 path's results are kept in float64; the FP32 split evaluates forces in
single precision, and its results are kept in float32.  Grain outlines and
placements follow the case, displacements, velocities, network parameters and
samples follow the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2108_07212_gb300 import binding as B
from paper_2108_07212_gb300 import inputs as I
from paper_2108_07212_gb300 import surrogate as SU

DEV = "cuda:0"
STIFF = (2.0, 3.0, 2.0, 2.0)      # the second material's E, k, rho, Gc over the first's


def listed():
    return [
        # the smallest run: the two-disk impact of the tests, default path, no tuning
        dict(name="two_disks_f64_default", kind="two_disks", h_ratio=8, precision="fp64", path="default", steps=10),
        # a bed of two materials with the conic micromodulus, default path
        dict(name="materials_f32_default", kind="settling", grains=120, h_ratio=15, geometry=5, precision="fp32",
             path="default", steps=25, materials=True, conic=True),
        # the 50-grain settling run of the benchmark, tuned, both precisions
        dict(name="settling50_f32", kind="settling", grains=50, h_ratio=15, geometry=1, precision="fp32",
             path="tuned", steps=50),
        dict(name="settling50_f64", kind="settling", grains=50, h_ratio=15, geometry=1, precision="fp64",
             path="tuned", steps=50),
        # the 500-grain compaction of the benchmark, grains thrown at each other
        dict(name="compaction500_f32", kind="compaction", grains=500, h_ratio=23, geometry=3, precision="fp32",
             path="tuned", steps=32),
        dict(name="compaction500_f64", kind="compaction", grains=500, h_ratio=23, geometry=3, precision="fp64",
             path="tuned", steps=16),
        # a parameter study: independent aggregates batched in one context
        dict(name="ensemble24_f32", kind="ensemble", aggregates=24, h_ratio=21, geometry=11, precision="fp32",
             path="tuned", steps=16),
        # many short windows from stored states (training data, rollouts)
        dict(name="restart_f32", kind="restart", grains=230, h_ratio=19, geometry=9, precision="fp32", path="tuned",
             steps=8),
        # grains advanced on the learned modal surrogate, one judge step per window
        dict(name="surrogate300_f32", kind="surrogate", grains=300, h_ratio=23, geometry=5, steps=50),
        # energy and observable output of a compaction run
        dict(name="energy100_f64", kind="energy", grains=100, h_ratio=23, geometry=3, precision="fp64", path="tuned",
             steps=10),
        # the surrogate's networks: Adam steps on minibatches of the training recipe, evaluation of a sample set
        dict(name="mlp_train_1024", kind="mlp_train", batch=1024, steps=4),
        dict(name="mlp_forward_20001", kind="mlp_forward", batch=20001),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["two_disks", "settling", "settling", "compaction", "compaction", "ensemble", "restart",
                       "surrogate", "energy", "mlp_train", "mlp_grad", "mlp_forward"])
    if kind == "mlp_forward":
        return dict(kind=kind, batch=_log(rng, 1, 200000))
    if kind in ("mlp_train", "mlp_grad"):
        return dict(kind=kind, batch=_log(rng, 33, 16000), steps=rng.randint(1, 6))
    geometry = rng.randint(1, 10 ** 6)
    if kind == "surrogate":
        return dict(kind=kind, grains=_log(rng, 30, 400), h_ratio=rng.randint(13, 20), geometry=geometry,
                    steps=rng.choice([20, 50, 70]))
    c = dict(kind=kind, h_ratio=rng.randint(8, 23), precision=rng.choice(["fp32", "fp64"]),
             path=rng.choice(["tuned", "tuned", "default"]), steps=_log(rng, 5, 50))
    if kind == "two_disks":
        c["h_ratio"] = _log(rng, 6, 60)
    elif kind == "ensemble":
        c.update(geometry=geometry, aggregates=_log(rng, 2, 9))
    else:
        c.update(geometry=geometry, grains=_log(rng, 12, 400))
        if kind == "settling":
            c.update(materials=rng.random() < 0.5, conic=rng.random() < 0.5)
    return c


# ---------------------------------------------------------------------------
# inputs


def _dt(h):
    """The workloads' time steps (5e-8 s at h = 67 um, 2e-8 s at 35 um) for any lattice spacing."""
    return 5e-8 * (h / 6.7e-5) ** 1.5


def _workload(case):
    kind, hr = case["kind"], case.get("h_ratio")
    if kind == "two_disks":
        w = I.two_disks(h_ratio=hr, dt=min(1e-7, _dt(1e-3 / hr)), k_bulk=5e5)
        h = 1e-3 / hr
        rc = w.params["rc_ratio"] * h
        # lattice rows in touch with the floor and with each other
        w.grain_geom[0, 1] = (hr - 1) * h + 0.7 * rc
        w.grain_geom[1, 0] = 2 * h
        w.grain_geom[1, 1] = w.grain_geom[0, 1] + 2 * (hr - 1) * h + 0.9 * rc
        return w
    if kind == "settling":
        s = math.sqrt(case["grains"] / 50)
        w = I.settling(case["grains"], box=(20e-3 * s + 3e-3, 30e-3 * s + 3e-3), h_ratio=hr, seed=case["geometry"],
                       dt=_dt(1e-3 / hr), micromodulus=1 if case.get("conic") else 0)
        if case.get("materials"):
            p = w.params
            soft = np.array([p["E"], p["k_bulk"], p["rho"], p["Gc"]])
            which = np.random.default_rng(case["geometry"]).integers(0, 2, w.n_grains).astype(np.int32)
            w.materials = (np.stack([soft, soft * np.array(STIFF)]), which)
        return w
    if kind == "ensemble":
        w = I.ensemble(case["aggregates"], h_ratio=hr, seed=case["geometry"] % 10 ** 6, dt=_dt(0.8e-3 / hr))
        return w
    if kind == "surrogate":
        rng_box = case["grains"] * math.pi * (1.35e-3) ** 2 / 0.33
        return I.settling(case["grains"], box=(math.sqrt(rng_box / 2) + 3e-3, 2 * math.sqrt(rng_box / 2) + 3e-3),
                          h_ratio=hr, seed=case["geometry"], mix=("hexagon", "drop"), dt=_dt(1e-3 / hr))
    # compaction, restart, energy: mixed grains between walls, the top one moving down
    n = case["grains"]
    return I.compaction(n, width=40e-3 * math.sqrt(n / 500) + 3e-3, h_ratio=hr, seed=case["geometry"],
                        dt=_dt(0.8e-3 / hr))


def _loaded(case, w, seed, X, grain):
    """Displacements and velocities of grains in motion: per grain a rigid
    velocity (5 m/s at most), a spin, and a smooth strain of about 1e-3."""
    rng = np.random.default_rng([int(seed), w.n_grains])
    G = w.n_grains
    c = w.grain_geom[grain, :2]
    R = w.grain_geom[grain, 2]
    r = X - c
    A = rng.normal(scale=7e-4, size=(G, 2, 2))[grain]
    k = (rng.normal(scale=2.0, size=(G, 2, 2)) / w.grain_geom[:, 2][:, None, None])[grain]
    ph = rng.uniform(0, 2 * math.pi, size=(G, 2))[grain]
    u = np.einsum("nij,nj->ni", A, r) + 3e-4 * R[:, None] * np.sin(np.einsum("nij,nj->ni", k, r) + ph)
    ang = rng.uniform(0, 2 * math.pi, G)
    speed = rng.uniform(0.5, 5.0, G)
    v = np.stack([speed * np.cos(ang), speed * np.sin(ang)], 1)
    if case["kind"] == "two_disks":
        v = np.array([[0.0, 0.0], [0.0, -1.0 - speed[1] / 5]])
    spin = rng.normal(scale=200.0, size=G)[grain]
    v = v[grain] + spin[:, None] * np.stack([-r[:, 1], r[:, 0]], 1) + np.einsum("nij,nj->ni", A[:, ::-1], r) * 3e4
    return u, v


_BASES: dict = {}     # modal bases by outline set and resolution: a program computes or loads them once


def _basis(case, w):
    key = (case["h_ratio"], tuple(np.round(s[0], 12).tobytes() for s in w.shapes))
    if key not in _BASES:
        one = I.Workload(shapes=w.shapes, grain_shape=np.arange(len(w.shapes), dtype=np.int32),
                         grain_geom=np.array([[3e-3 * (q + 1), 3e-3, 1e-3, 0, 0, 0, 1e-3 / case["h_ratio"]]
                                              for q in range(len(w.shapes))]), params=w.params, n_steps=1)
        S = B.Simulation(one, precision="fp32")
        cfg = SU.build_basis(S)
        offs = np.concatenate([[0], np.cumsum([2 * d["nodes"] * 32 for d in cfg["templates"]])])
        lam = cfg["lambda_"].reshape(-1, 32)
        _BASES[key] = [(cfg["basis"][offs[t]:offs[t + 1]], lam[t], cfg["templates"][t])
                       for t in cfg["template_of_grain"]]
        S.close()
    return _BASES[key]


def _params(seed):
    """He-initialised parameters with a small last layer (a network in training)."""
    p = SU.init_params(int(seed) % (1 << 31))
    rng = np.random.default_rng([int(seed), 3])
    o = 128 * 32 + 128 + 128 * 128 + 128
    p[o:o + 32 * 128] = rng.normal(scale=0.05, size=32 * 128)
    return p.astype(np.float32)


def _samples(seed, n, k):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    x = torch.randn((k, n, 32), generator=g, device=DEV)
    A = 0.3 * torch.randn((32, 32), generator=g, device=DEV)
    return x, (torch.tanh(x @ A) + 0.1 * x.flip(2)).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind.startswith("mlp"):
        steps = case.get("steps", 1)
        x, t = _samples(seed, case["batch"], steps)
        return dict(kind=kind, net=B.MLP(max_batch=case["batch"], params=_params(seed)), x=x, t=t)
    w = _workload(case)
    if kind == "surrogate":
        cfg = {}

        def setup(sim):
            pieces = _basis(case, w)
            tmpl = sim.get("GRAIN_TEMPLATE")
            first = [int(w.grain_shape[int(np.argmax(tmpl == q))]) for q in range(int(tmpl.max()) + 1)]
            cfg.update(basis=np.concatenate([pieces[s][0] for s in first]),
                       lambda_=np.concatenate([pieces[s][1] for s in first]), n_modes=32, judge_every=50, gate=0.5,
                       err_tol=1e-3, templates=[pieces[s][2] for s in first], template_of_grain=tmpl)
            return cfg

        sim = B.Simulation(w, precision="fp32", device=DEV, surrogate=setup)
        for q, n in enumerate(np.bincount(cfg["template_of_grain"])):
            sim.surrogate_set_mlp(q, B.MLP(max_batch=int(n), params=SU.init_params(int(seed) % (1 << 31))))
        rng = np.random.default_rng([int(seed), 7])
        sim.set("DISP", SU.modal_field(sim, cfg, rng.normal(scale=2e-5, size=(w.n_grains, 32))))
        grain = sim.get("GRAIN")
        sim.set("VEL", rng.normal(scale=1.0, size=(w.n_grains, 2))[grain])
        sim.surrogate_enable(True)
    else:
        sim = B.Simulation(w, precision=case["precision"], device=DEV)
        u, v = _loaded(case, w, seed, sim.get("X"), sim.get("GRAIN"))
        sim.set("DISP", u)
        sim.set("VEL", v)
    sim.eval_forces()
    if case.get("path", "tuned") == "tuned":
        sim.autotune()
    out = {f: torch.empty((sim.N, 2), dtype=torch.float64, device=DEV) for f in ("DISP", "VEL", "ACC")}
    st = dict(kind=kind, sim=sim, steps=case["steps"], out=out, single=sim.precision == B.PD_FP32_SPLIT)
    if kind == "restart":
        st["stored"] = {f: sim.get_device(f, torch.empty_like(out[f])) for f in out}
    return st


def run(state):
    kind = state["kind"]
    if kind == "mlp_forward":
        return state["net"].forward(state["x"][0])
    if kind == "mlp_grad":
        loss, grad = state["net"].loss_grad(state["x"][0], state["t"][0])
        return dict(loss=loss, grad=grad)
    if kind == "mlp_train":
        losses = [state["net"].train_step(x, t, 2e-3) for x, t in zip(state["x"], state["t"])]
        return dict(loss=losses, params=state["net"].get_params())
    sim, out = state["sim"], state["out"]
    if kind == "restart":
        for f, stored in state["stored"].items():
            sim.set(f, stored)
    sim.step(state["steps"])
    res = {}
    if kind == "energy":
        res["energy"] = sim.diagnostics()
        res["observables"] = sim.observables()
    for f, buf in out.items():
        sim.get_device(f, buf)
        res[f] = buf.float() if state["single"] else buf
    return res


def _nodes(case):
    """Nodes per grain of the shape mixes: about 0.6 of the security disk's area over h^2."""
    per = 0.62 * math.pi * case["h_ratio"] ** 2
    kind = case["kind"]
    if kind == "two_disks":
        return 2 * math.pi * case["h_ratio"] ** 2
    if kind == "ensemble":
        return case["aggregates"] * 110 * per
    return case["grains"] * per


def work(case):
    kind = case["kind"]
    if kind == "mlp_forward":
        return dict(bytes=case["batch"] * 256 + 2 * 24864, flops=case["batch"] * 2.0 * 24576)
    if kind in ("mlp_train", "mlp_grad"):
        k = case["steps"] if kind == "mlp_train" else 1
        return dict(bytes=k * (case["batch"] * 256 + 6 * 4 * 24864), flops=k * case["batch"] * 6.0 * 24576)
    # a step reads and writes u, v and a and reads the reference position, the
    # bonds a node has (one bit each), the broken ones, and the grain; about
    # eleven bonds per node at some thirty operations each
    n = _nodes(case)
    state = 16 + 16 + (16 if case.get("precision", "fp32") == "fp64" else 8)
    return dict(bytes=case["steps"] * n * (2 * state + 16 + 12), flops=case["steps"] * n * 400.0)


# ---------------------------------------------------------------------------
# the same in 64 bits: lattices, bonds, contact and walls from the equations


def _inside(loops, p, clear):
    """Points of p strictly inside the outline (loops: outer, then holes) and `clear` away from it."""
    wn = np.zeros(len(p), dtype=bool)
    near = np.zeros(len(p), dtype=bool)
    for lp in loops:
        for a, b in zip(lp, np.roll(lp, -1, axis=0)):
            e, q = b - a, p - a
            up = (a[1] <= p[:, 1]) != (b[1] <= p[:, 1])
            with np.errstate(divide="ignore", invalid="ignore"):
                x = a[0] + (p[:, 1] - a[1]) * e[0] / e[1] if e[1] != 0 else np.zeros(len(p))
            wn ^= up & (p[:, 0] < x)
            t = np.clip(q @ e / (e @ e), 0, 1)
            near |= np.hypot(q[:, 0] - t * e[0], q[:, 1] - t * e[1]) < clear
    return wn & ~near


def _crosses(loops, p, q):
    """Segments p-q that cross the outline (a touch at a corner is none)."""
    hit = np.zeros(len(p), dtype=bool)

    def cr(a, b):
        return a[..., 0] * b[..., 1] - a[..., 1] * b[..., 0]

    d = q - p
    for lp in loops:
        for a, b in zip(lp, np.roll(lp, -1, axis=0)):
            s1, s2 = cr(d, a - p), cr(d, b - p)
            s3, s4 = cr(b - a, p - a), cr(b - a, q - a)
            hit |= (s1 * s2 < -1e-12) & (s3 * s4 < -1e-12)
    return hit


def _mesh(w):
    """Positions, grains, spacings and undirected bonds (i, j, offset length / h) of a workload."""
    cache, X, gr, bi, bj, bn, base = {}, [], [], [], [], [], 0
    for g in range(w.n_grains):
        cx, cy, R, th, _, _, h = w.grain_geom[g]
        key = (int(w.grain_shape[g]), round(R / h, 9))
        if key not in cache:
            loops = [np.asarray(lp) * (R / h) for lp in w.shapes[key[0]]]
            m = int(math.ceil(R / h)) + 1
            jj, ii = np.mgrid[-m:m + 1, -m:m + 1]
            lat = np.stack([ii.ravel(), jj.ravel()], 1)
            lat = lat[_inside(loops, lat.astype(float), 1e-6)]
            idx = np.full((2 * m + 7, 2 * m + 7), -1)
            idx[lat[:, 0] + m + 3, lat[:, 1] + m + 3] = np.arange(len(lat))
            ei, ej, en = [], [], []
            for dj in range(0, 3):
                for di in range(-2, 3):
                    if (dj, di) <= (0, 0) or di * di + dj * dj >= 9:
                        continue
                    o = idx[lat[:, 0] + di + m + 3, lat[:, 1] + dj + m + 3]
                    a = np.nonzero(o >= 0)[0]
                    keep = ~_crosses(loops, lat[a].astype(float), lat[o[a]].astype(float))
                    ei.append(a[keep]), ej.append(o[a][keep])
                    en.append(np.full(keep.sum(), math.sqrt(di * di + dj * dj)))
            cache[key] = lat, np.concatenate(ei), np.concatenate(ej), np.concatenate(en)
        lat, ei, ej, en = cache[key]
        l = lat * h
        X.append(np.stack([cx + (math.cos(th) * l[:, 0] - math.sin(th) * l[:, 1]),
                           cy + (math.sin(th) * l[:, 0] + math.cos(th) * l[:, 1])], 1))
        gr.append(np.full(len(lat), g))
        bi.append(ei + base), bj.append(ej + base), bn.append(en)
        base += len(lat)
    return (np.concatenate(X), np.concatenate(gr), np.concatenate(bi), np.concatenate(bj), np.concatenate(bn))


def _pairs(p, grp, agg, radius):
    """Directed pairs of nodes of different grains of one aggregate closer than radius."""
    c = torch.floor(p / radius).long()
    c = c - c.min(0).values + 1
    W, H = int(c[:, 0].max()) + 2, int(c[:, 1].max()) + 2
    key = (agg * W + c[:, 0]) * H + c[:, 1]
    sk, order = torch.sort(key)
    out = []
    for dx in (-1, 0, 1):
        for dy in (-1, 0, 1):
            q = key + dx * H + dy
            lo, hi = torch.searchsorted(sk, q), torch.searchsorted(sk, q, right=True)
            n = hi - lo
            i = torch.repeat_interleave(torch.arange(len(q), device=p.device), n)
            k = torch.arange(len(i), device=p.device) - torch.repeat_interleave(torch.cumsum(n, 0) - n, n)
            j = order[lo[i] + k]
            ok = (grp[i] != grp[j]) & ((p[i] - p[j]).norm(dim=1) < radius)
            out.append(torch.stack([i[ok], j[ok]]))
    return torch.cat(out, 1)


def _exact_steps(case, seed):
    w = _workload(case)
    if w.n_grains * 0.62 * math.pi * case["h_ratio"] ** 2 > 8e5:
        return None
    P = w.params
    X, grain, bi, bj, bn = _mesh(w)
    u, v = _loaded(case, w, seed, X, grain)
    dev = DEV if torch.cuda.is_available() else "cpu"

    def T(a):
        return torch.as_tensor(np.ascontiguousarray(a), device=dev)

    G = w.n_grains
    props = np.array([[P["E"], P["k_bulk"], P["rho"], P["Gc"]]]) if w.materials is None else w.materials[0]
    gm = np.zeros(G, int) if w.materials is None else w.materials[1]
    E, kb, rho, Gc = (props[gm, q] for q in range(4))
    agg = np.zeros(G, int) if w.grain_agg is None else np.asarray(w.grain_agg)
    walls = np.array([[P["wall_lo"][0], P["wall_hi"][0], P["wall_lo"][1], P["wall_hi"][1], P["wall_vel_lo"][0],
                       P["wall_vel_hi"][0], P["wall_vel_lo"][1], P["wall_vel_hi"][1]]]) \
        if w.agg_walls is None else w.agg_walls
    h = w.grain_geom[:, 6]
    eps = P["horizon_ratio"] * h
    hmin = np.array([h[agg == a].min() for a in range(agg.max() + 1)])[agg]
    Rc = P["rc_ratio"] * hmin
    Kn = 18 * kb / (math.pi * (P["horizon_ratio"] * hmin) ** 5)
    conic = P["micromodulus"] == 1
    cw = (24 if conic else 6) * E / (math.pi * eps ** 3 * (1 - P["nu"]))
    s0 = np.sqrt((5 if conic else 4) * math.pi * Gc / (9 * E * eps))
    gr = T(grain)
    V, rn, Rcn, Knn = (T((q)[grain]) for q in (h ** 2, rho, Rc, Kn))
    gb = grain[bi]
    xi = T(bn * h[gb])
    cb = T(cw[gb] * h[gb] ** 4) * (1 - xi / T(eps[gb]) if conic else 1)
    s0b = T(s0[gb])
    bi, bj = T(bi), T(bj)
    alive = torch.ones_like(xi)
    Xt, u, v = T(X), T(u), T(v)
    W = T(walls[agg[grain]])
    dt, mu, rd = P["dt"], P["friction"], P["damping_ratio"]
    grav = torch.tensor([P["gx"], P["gy"]], dtype=torch.float64, device=dev)
    reach = float(Rc.max()) * 1.02 + 2 * (case["steps"] + 2) * dt * float(v.norm(dim=1).max())
    near = _pairs(Xt + u, gr, T(agg)[gr], reach)
    pi, pj = near[0], near[1]

    def rub(e, vr, Fr, Vx, Vy, K, rd_, rx):
        vn = (vr * e).sum(1)
        vt = vr - vn[:, None] * e
        s = vt.norm(dim=1)
        c = torch.where(s > mu * Fr * dt / (rx * Vx), mu * Fr / s.clamp_min(1e-300), rx * Vx / dt)
        return -(2 * rd * torch.sqrt(K * rd_ / Vy) * Vx * Vy * vn)[:, None] * e - c[:, None] * vt

    def forces(t):
        p = Xt + u
        F = torch.zeros_like(p)
        d = p[bj] - p[bi]
        L = d.norm(dim=1)
        s = (L - xi) / xi
        alive.mul_((s.abs() <= s0b).double())
        f = (alive * cb * s / L)[:, None] * d
        F.index_add_(0, bi, f)
        F.index_add_(0, bj, -f)
        d = p[pj] - p[pi]
        L = d.norm(dim=1)
        k = torch.nonzero(L < Rcn[pi])[:, 0]
        if len(k):
            i, j, d, L = pi[k], pj[k], d[k], L[k]
            e = d / L[:, None]
            K = 2 * Knn[i] * Knn[j] / (Knn[i] + Knn[j])
            Fr = K * (Rcn[i] - L) * V[i] * V[j]
            F.index_add_(0, i, -Fr[:, None] * e + rub(e, v[i] - v[j], Fr, V[i], V[j], K,
                                                      2 * rn[i] * rn[j] / (rn[i] + rn[j]), rn[i]))
        for l in range(4):
            ax, sg = l // 2, (-1.0, 1.0)[l % 2]
            dd = (sg * ((W[:, l] + W[:, 4 + l] * t) - p[:, ax])).clamp_min(0)
            k = torch.nonzero(dd < Rcn)[:, 0]
            if len(k) == 0:
                continue
            R, d1 = Rcn[k], dd[k]
            th = torch.atan2(torch.sqrt((R - d1) * (R + d1)), d1)
            sn = torch.sin(th)
            h1 = th - sn * torch.cos(th)
            gap = R * (h1 - 2 / 3 * sn ** 3) / h1
            area = R * R * h1
            Fr = Knn[k] * gap * V[k] * area
            e = torch.zeros((len(k), 2), dtype=torch.float64, device=dev)
            e[:, ax] = sg
            vw = torch.zeros_like(e)
            vw[:, ax] = W[k, 4 + l]
            F.index_add_(0, k, -Fr[:, None] * e + rub(e, v[k] - vw, Fr, V[k], area, Knn[k], rn[k], rn[k]))
        return F

    def acc(t):
        return forces(t) / (rn * V)[:, None] + grav

    a = acc(0.0)
    for n in range(case["steps"]):
        u = u + dt * v + 0.5 * dt * dt * a
        an = acc((n + 1) * dt)
        v = v + 0.5 * dt * (a + an)
        a = an
    res = {}
    if case["kind"] == "energy":
        p, m = Xt + u, rn * V
        s = ((p[bj] - p[bi]).norm(dim=1) - xi) / xi
        res["energy"] = dict(KE=float((0.5 * m * (v * v).sum(1)).sum()), E_bond=float((0.5 * alive * cb * s * s * xi).sum()),
                             Px=float((m * v[:, 0]).sum()), Py=float((m * v[:, 1]).sum()),
                             Lz=float((m * (p[:, 0] * v[:, 1] - p[:, 1] * v[:, 0])).sum()), n_broken=None,
                             E_contact=None, E_wall=None)
        res["observables"] = None
    res.update(DISP=u, VEL=v, ACC=a)
    return res


def _exact_mlp(case, seed):
    x, t = _samples(seed, case["batch"], case.get("steps", 1))
    flat = torch.tensor(_params(seed), dtype=torch.float64, device=DEV, requires_grad=True)

    def net(z):
        o, v = 0, []
        for shape in ((128, 32), (128,), (128, 128), (128,), (32, 128), (32,)):
            n = math.prod(shape)
            v.append(flat[o:o + n].reshape(shape))
            o += n
        F = torch.nn.functional
        z = F.gelu(z.double() @ v[0].T + v[1])
        return F.gelu(z @ v[2].T + v[3]) @ v[4].T + v[5]

    if case["kind"] == "mlp_forward":
        return net(x[0]).detach()
    opt = torch.optim.Adam([flat], lr=2e-3, betas=(0.9, 0.999), eps=1e-8)
    losses = []
    for xb, tb in zip(x, t):
        opt.zero_grad()
        loss = ((net(xb) - tb) ** 2).mean()
        loss.backward()
        losses.append(float(loss))
        if case["kind"] == "mlp_grad":
            return dict(loss=losses[0], grad=flat.grad.clone())
        opt.step()
    return dict(loss=losses, params=flat.detach())


def exact(case, seed):
    if case["kind"].startswith("mlp"):
        return _exact_mlp(case, seed)
    if case["kind"] == "surrogate":      # its forces are a modal model of the bonds', not the equations'
        return None
    return _exact_steps(case, seed)
