"""Measured cases of the granular time step.

A pass is what a coupled host program does once per time step with device
memory: it hands the body state to the scene (nbgs_set_bodies, or
nbgs_update_bodies where the previous step's impulses start the solve), takes
one time step (or a few replayed graph steps) and reads the body state back
(nbgs_get_bodies), some with the contacts and their impulses too
(nbgs_get_contacts).  The velocities handed in alternate between two sets, as
under changing external forces, so that a warm-started solve never starts
from its own answer and every pass is the same amount of work.  One kind of
case trains or evaluates the warm-start network instead.

Inputs are synthetic and drawn from the seed.  Piles are hexagonal close
packings whose spheres either touch their neighbours (radius 1/2 up to a few
1e-5) or are smaller by 2-20 % and touch nothing: with 68 % touching, a pile
has 2.8 contacts per sphere in 13 to 14 colours, like the settled
polydisperse 1M-sphere pour; with all touching it is the dense packing.

`exact` computes the same steps in FP64 with plain torch: neighbour search on
a cell grid, the first-fit colouring in decreasing hashed priority, the
sweeps colour by colour, integration.
"""
from __future__ import annotations

import ctypes as C
import math

import numpy as np
import torch

from paper_1501_05810_gb300 import nbgs

DEV = "cuda"
SEED = 0x5EED        # colour_seed of every scene
N_PARAMS = 9347      # warm-start network: 12 -> 64 -> 64 -> 64 -> 3
SIZES = (12, 64, 64, 64, 3)


def _pile(n, **kw):
    c = dict(kind="spheres", n=n, touch=0.68, periodic=False, order="lattice", precision="fp32", sweeps=100, tol=0.0,
             warm=False, contacts=False, sub="none", omega=1.0, dt=5e-4)
    c.update(kw)
    return c


def listed():
    return [
        # the 1,000-sphere FP64 parity workload: 50 sweeps a step; latency of the smallest scenes
        _pile(1000, name="box_1k_fp64", precision="fp64", sweeps=50, dt=1e-3),
        # a small FP32 scene solved to 1e-4 every step, as in a many-step simulation of a few thousand grains
        _pile(2003, name="box_2k_tol", sweeps=500, tol=1e-4),
        # a medium pile coupled to a host code that also reads the contact forces back; odd size
        _pile(30011, name="pile_30k_contacts", warm=True, contacts=True),
        # a pile whose spheres come in no spatial order (random insertion, a long-mixed bed)
        _pile(250000, name="pile_250k_mixed", order="mixed", sweeps=50, warm=True),
        # FP64 sweeps, for tight tolerances and parity runs of production-like piles
        _pile(120007, name="pile_120k_fp64", precision="fp64", sweeps=30, warm=True, contacts=True),
        # the main workload: 1M-sphere pile, 100 sweeps or 1e-6, previous-step warm start
        _pile(1000000, name="pile_1m", tol=1e-6, warm=True),
        # the densest: hexagonal close packing 100 x 100 x 100, periodic in x and y
        _pile(1000000, name="dense_1m", touch=1.0, periodic=True, warm=True),
        # Alg. 1 with a grid of subdomains
        _pile(262144, name="ramp_262k_subdomains", touch=1.0, periodic=True, sweeps=50, sub="8,8,1", omega=0.5),
        # dilute granular gas, triply periodic: detection and integration, few sweeps
        dict(name="gas_4m", kind="gas", n=4000000, precision="fp32", sweeps=10, dt=2e-3),
        # many small independent scenes under one captured graph, each solved to 1e-6
        dict(name="batch_256", kind="batch", scenes=256, n_lo=200, n_hi=20000, touch=0.3, sweeps=200, tol=1e-6, steps=2),
        # composite particles (2-4 spheres each) falling into a pile
        dict(name="composite_100k", kind="composite", n=100000, precision="fp32", sweeps=50, dt=1e-2),
        # one epoch-sized batch of training the warm-start network: forward, backward, Adam
        dict(name="mlp_train_1m", kind="mlp", rows=1000000, train=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["spheres"] * 6 + ["gas", "batch", "composite", "mlp"])
    if kind == "gas":
        return dict(kind="gas", n=_log(rng, 50000, 4000000), precision=rng.choice(["fp32", "fp32", "fp64"]),
                    sweeps=rng.choice([10, 20]), dt=rng.choice([1e-3, 2e-3]))
    if kind == "batch":
        return dict(kind="batch", scenes=_log(rng, 8, 256), n_lo=200, n_hi=rng.choice([2000, 20000]),
                    touch=rng.choice([0.2, 0.3]), sweeps=200, tol=1e-6, steps=rng.choice([1, 2]))
    if kind == "composite":
        return dict(kind="composite", n=_log(rng, 1000, 100000), precision="fp32", sweeps=rng.choice([10, 30, 50]),
                    dt=rng.choice([5e-3, 1e-2]))
    if kind == "mlp":
        return dict(kind="mlp", rows=_log(rng, 5000, 1000000), train=rng.random() < 0.5)
    fp64 = rng.random() < 0.25
    c = _pile(_log(rng, 500, 100000 if fp64 else 1000000), touch=rng.choice([0.5, 0.68, 0.68, 1.0]),
              precision="fp64" if fp64 else "fp32", sweeps=rng.choice([10, 30, 50, 100]) if not fp64 else 30,
              order="mixed" if rng.random() < 0.2 else "lattice", warm=rng.random() < 0.5,
              contacts=rng.random() < 0.3, periodic=rng.random() < 0.4, dt=rng.choice([2e-4, 5e-4]))
    if c["n"] > 300000:
        c["sweeps"] = min(c["sweeps"], 50)
    r = rng.random()
    if r < 0.1:
        g = rng.choice([2, 4, 8])
        c.update(sub="%d,%d,1" % (g, g), omega=0.5)
    elif r < 0.2:
        c.update(sub="jacobi", omega=0.3)
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _walls(lo, hi, axes=(0, 1, 2)):
    out = []
    for a in axes:
        e = [0.0, 0.0, 0.0]
        e[a] = 1.0
        out.append((tuple(e), float(lo[a])))
        out.append((tuple(-x for x in e), -float(hi[a])))
    return out


def _packing(n, touch, periodic, rng):
    """n spheres of a hexagonal close packing, x fastest and z slowest, in a
    walled box (periodic in x and y with walls in z, layers then complete)."""
    nx = max(3, round(n ** (1.0 / 3.0)))
    ny = max(4, 2 * round(nx / 2.0))
    nz = max(2, round(n / (nx * ny))) if periodic else -(-n // (nx * ny))
    if periodic:
        n = nx * ny * nz
    idx = np.arange(n)
    i, j, k = idx % nx, (idx // nx) % ny, idx // (nx * ny)
    pos = np.empty((n, 3))
    pos[:, 0] = 0.5 * (2.0 * i + ((j + k) % 2))
    pos[:, 1] = 0.5 * math.sqrt(3.0) * (j + (k % 2) / 3.0)
    pos[:, 2] = 0.5 + math.sqrt(6.0) / 3.0 * k
    # a periodic packing has nowhere to give: gaps only; a walled one has 1e-3 of slack at its side walls and no lid
    near = rng.normal(0.0, 2e-5, n)
    e = np.where(rng.random(n) < touch, np.abs(near) if periodic else near, rng.uniform(0.02, 0.2, n))
    radius = 0.5 * (1.0 - e)
    lo = np.zeros(3)
    if periodic:
        pos[:, :2] += 0.25   # no sphere on the periodic faces, where a rounding would decide its image
        hi = np.array([float(nx), math.sqrt(3.0) / 2.0 * ny, 1.0 + math.sqrt(6.0) / 3.0 * (nz - 1)])
        return pos, radius, lo, hi, (1, 1, 0), _walls(lo, hi, (2,))
    pos[:, :2] += 0.501
    hi = np.array([nx + 0.502, math.sqrt(3.0) / 2.0 * (ny - 1 + 2.0 / 3.0) + 1.002, 2.0 + math.sqrt(6.0) / 3.0 * (nz - 1)])
    return pos, radius, lo, hi, (0, 0, 0), _walls(lo, hi)


def _inputs(case, seed):
    """The scenes of a case (one, or the batch's), and the two velocity sets
    the passes alternate between."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    base = dict(gravity=(0.0, 0.0, -9.81), mu=0.5, omega=case.get("omega", 1.0), tau=0.004, beta=1.0, colour_seed=SEED,
                precision=case.get("precision", "fp32"), warm_start="prev" if case.get("warm") else "none")
    if kind == "spheres":
        pos, radius, lo, hi, per, planes = _packing(case["n"], case["touch"], case["periodic"], rng)
        if case["order"] == "mixed":
            q = rng.permutation(len(radius))
            pos, radius = pos[q], radius[q]
        sub = {"none": None, "jacobi": "jacobi"}.get(case["sub"], case["sub"])
        if sub not in (None, "jacobi"):
            sub = tuple(int(g) for g in sub.split(","))
        prm = dict(base, dt=case["dt"], box_lo=tuple(lo), box_hi=tuple(hi), periodic=per, subdomains=sub)
        scenes = [dict(params=prm, pos=pos, radius=radius, planes=planes)]
        sigma = 0.01
    elif kind == "gas":
        cells = max(4, round((case["n"] / 4.0) ** (1.0 / 3.0)))
        n = 4 * cells ** 3
        radius = rng.uniform(0.45, 0.55, n)
        side = (4.0 / 3.0 * math.pi * float(np.sum(radius ** 3)) / 0.5) ** (1.0 / 3.0)
        g = np.stack(np.meshgrid(*[np.arange(cells)] * 3, indexing="ij"), -1).reshape(-1, 1, 3)
        corners = np.array([[0.25, 0.25, 0.25], [0.75, 0.75, 0.25], [0.75, 0.25, 0.75], [0.25, 0.75, 0.75]])
        pos = ((g + corners) * (side / cells)).reshape(-1, 3) + rng.uniform(-0.025, 0.025, (n, 3))
        prm = dict(base, gravity=(0.0, 0.0, 0.0), mu=0.3, dt=case["dt"], box_lo=(0.0,) * 3, box_hi=(side,) * 3,
                   periodic=(1, 1, 1), contacts_per_body=4)
        scenes = [dict(params=prm, pos=pos, radius=radius, planes=[])]
        sigma = 1.0
    elif kind == "batch":
        # log-uniform sizes in a shuffled order, the same for every seed
        sizes = np.rint(np.geomspace(case["n_lo"], case["n_hi"], case["scenes"])).astype(int)
        sizes = np.random.default_rng(case["scenes"]).permutation(sizes)
        mus = rng.uniform(0.2, 0.8, len(sizes))
        cols = math.ceil(math.sqrt(len(sizes)))
        scenes = []
        for k, (m, mu) in enumerate(zip(sizes, mus)):
            pos, radius, lo, hi, per, _ = _packing(int(m), case["touch"], False, rng)
            off = np.array([(k % cols) * 32.0, (k // cols) * 32.0, 0.0])
            prm = dict(base, warm_start="prev", mu=float(mu), dt=5e-4, box_lo=tuple(lo + off), box_hi=tuple(hi + off),
                       contacts_per_body=4)
            scenes.append(dict(params=prm, pos=pos + off, radius=radius, planes=_walls(lo + off, hi + off)))
        sigma = 0.01
    elif kind == "composite":
        nx = max(2, round(case["n"] ** (1.0 / 3.0)))
        n = nx * nx * max(1, round(case["n"] / (nx * nx)))
        idx = np.arange(n)
        pos = (np.stack([idx % nx, (idx // nx) % nx, idx // (nx * nx)], -1) + 0.5) * 0.95
        hi = pos.max(0) + 0.475
        counts = rng.integers(2, 5, n)
        body = np.repeat(np.arange(n), counts)
        r = rng.uniform(0.3, 0.4, len(body))
        d = rng.normal(size=(len(body), 3))
        d /= np.linalg.norm(d, axis=1, keepdims=True)
        prm = dict(base, mu=0.4, tau=0.005, dt=case["dt"], box_lo=(0.0,) * 3, box_hi=tuple(hi), warm_start="prev")
        scenes = [dict(params=prm, pos=pos, planes=_walls(np.zeros(3), hi),
                       members=dict(body=body.astype(np.int32), offset=d * (0.5 - r)[:, None], radius=r))]
        sigma = 0.2
    n_all = sum(len(s["pos"]) for s in scenes)
    vels = []
    for _ in range(2):
        v = rng.normal(0.0, sigma, (n_all, 3)).astype(np.float32).astype(np.float64)
        if kind == "composite":
            v[:, 2] -= 3.0
        vels.append(v)
    ang = rng.normal(0.0, sigma, (n_all, 3)).astype(np.float32).astype(np.float64)
    at = 0
    for s in scenes:
        m = len(s["pos"])
        s.update(vel=vels[0][at:at + m], angvel=ang[at:at + m], density=np.ones(m), cones=[])
        at += m
    return scenes, vels, ang


def _mlp_inputs(case, seed):
    g = torch.Generator(DEV).manual_seed(seed)
    theta = []
    for i, o in zip(SIZES[:-1], SIZES[1:]):
        lim = math.sqrt(6.0 / (i + o))
        theta += [(torch.rand(o * i, generator=g, device=DEV) * 2 - 1) * lim,
                  (torch.rand(o, generator=g, device=DEV) * 2 - 1) * 0.1]
    X = torch.randn(case["rows"], 12, generator=g, device=DEV)
    T = torch.randn(case["rows"], 3, generator=g, device=DEV)
    return torch.cat(theta), X, T


def _contact_cap(n):
    """At most six contacts per sphere of a pile, walls included."""
    return 7 * n


def prepare(case, seed):
    if case["kind"] == "mlp":
        theta, X, T = _mlp_inputs(case, seed)
        z = torch.zeros(N_PARAMS, device=DEV)
        return dict(case=case, theta=theta, X=X, T=T, m=z.clone(), v=z.clone(), grad=z.clone(), step=0,
                    loss=torch.zeros(1, dtype=torch.float64, device=DEV), Y=torch.empty(case["rows"], 3, device=DEV))
    scenes, vels, ang = _inputs(case, seed)
    if case["kind"] == "batch":
        scene = nbgs.BatchScene(scenes)
        pos = np.concatenate([s["pos"] for s in scenes])
    else:
        scene = nbgs.Scene(scenes[0])
        pos = scene.get_bodies()["pos"] if case["kind"] == "composite" else scenes[0]["pos"]
    n = len(pos)
    quat = torch.zeros(n, 4, dtype=torch.float64, device=DEV)
    quat[:, 0] = 1.0
    f64 = lambda a: torch.as_tensor(a, dtype=torch.float64).to(DEV)  # noqa: E731
    out = {k: torch.empty(n, w, dtype=torch.float64, device=DEV)
           for k, w in (("pos", 3), ("quat", 4), ("vel", 3), ("angvel", 3))}
    if case.get("contacts"):   # contact buffers of a fixed capacity; rows past the count keep what they hold
        cap = _contact_cap(n)
        out.update(ends=torch.zeros(3, cap, dtype=torch.int32, device=DEV),
                   **{k: torch.zeros(cap, w, dtype=torch.float64, device=DEV)
                      for k, w in (("normal", 3), ("xi", 1), ("impulse", 3))})
    state = dict(case=case, scene=scene, pos=f64(pos), quat=quat, vels=[f64(v) for v in vels], ang=f64(ang), out=out,
                 turn=0, warm=scenes[0]["params"]["warm_start"] == "prev",
                 cast=torch.float32 if scenes[0]["params"]["precision"] == "fp32" else torch.float64)
    if case["kind"] == "batch":
        scene.step(case["sweeps"], case["tol"], stats=False)   # sizes the buffers before the first graph step
    return state


def _check(status, what):
    if status != nbgs.NBGS_OK:
        raise RuntimeError("%s: status %d" % (what, status))


def run(state):
    case = state["case"]
    lib = nbgs.library()
    if case["kind"] == "mlp":
        stream = torch.cuda.current_stream().cuda_stream
        th, X = state["theta"], state["X"]
        if not case["train"]:
            _check(lib.nbgs_mlp_infer(th.data_ptr(), X.data_ptr(), state["Y"].data_ptr(), len(X), stream), "infer")
            return state["Y"]
        _check(lib.nbgs_mlp_grad(th.data_ptr(), X.data_ptr(), state["T"].data_ptr(), len(X), state["grad"].data_ptr(),
                                 state["loss"].data_ptr(), stream), "grad")
        state["step"] += 1
        _check(lib.nbgs_mlp_adam(th.data_ptr(), state["grad"].data_ptr(), state["m"].data_ptr(), state["v"].data_ptr(),
                                 N_PARAMS, 2e-3, 0.9, 0.999, 1e-8, state["step"], stream), "adam")
        return {"theta": th, "grad": state["grad"], "m": state["m"], "v": state["v"], "loss": state["loss"].float()}
    sc, out = state["scene"], state["out"]
    vel = state["vels"][state["turn"] % 2]
    state["turn"] += 1
    (sc.update_bodies if state["warm"] else sc.set_bodies)(state["pos"], state["quat"], vel, state["ang"])
    if case["kind"] == "batch":
        sc.graph_step(case["sweeps"], case["tol"], case["steps"])
        got = {}
    else:
        st = sc.step(case["sweeps"], case.get("tol", 0.0))
        got = {"n_contacts": st["n_contacts"], "n_colours": st["n_colours"]}
    _check(lib.nbgs_get_bodies(sc.h, *[out[k].data_ptr() for k in ("pos", "quat", "vel", "angvel")]), "get_bodies")
    # FP32 sweeps hold velocities, orientations and impulses in FP32
    got.update({k: out[k].to(state["cast"]) for k in ("quat", "vel", "angvel")}, pos=out["pos"])
    if case.get("contacts"):
        j, count = out["ends"], C.c_int64()
        _check(lib.nbgs_get_contacts(sc.h, j.shape[1], j[0].data_ptr(), j[1].data_ptr(), j[2].data_ptr(),
                                     *[out[k].data_ptr() for k in ("normal", "xi", "impulse")], C.byref(count)),
               "get_contacts")
        got.update(j1=j[0], j2=j[1], colour=j[2], normal=out["normal"], xi=out["xi"],
                   impulse=out["impulse"].to(state["cast"]))
    return got


def _expected(case):
    """(bodies, contacts) of a case by its recipe."""
    if case["kind"] == "batch":
        mean = (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])
        n = case["scenes"] * mean
        return n, 6.0 * case["touch"] ** 2 * n * 0.9
    if case["kind"] == "gas":
        return case["n"], 0.05 * case["n"]
    if case["kind"] == "composite":
        return case["n"], 1.5 * case["n"]
    return case["n"], 6.0 * case["touch"] ** 2 * case["n"]


def work(case):
    if case["kind"] == "mlp":
        k = sum(i * o for i, o in zip(SIZES[:-1], SIZES[1:]))
        if case["train"]:
            return {"bytes": case["rows"] * 60.0 + 32.0 * N_PARAMS, "flops": 6.0 * k * case["rows"]}
        return {"bytes": case["rows"] * 60.0 + 4.0 * N_PARAMS, "flops": 2.0 * k * case["rows"]}
    n, c = _expected(case)
    # state in and out (pos, quat, vel, angvel in FP64); contacts out; a neighbour test per body and
    # candidate, and about 150 operations per contact and sweep (400 for a composite contact)
    steps = case.get("steps", 1)
    by = n * 2 * 104.0 + (c * 68.0 if case.get("contacts") else 0.0)
    per = 400.0 if case["kind"] == "composite" else 150.0
    return {"bytes": by, "flops": steps * (n * 300.0 + c * case["sweeps"] * per)}


# ---------------------------------------------------------------------------
# the same steps in FP64 with plain torch
# ---------------------------------------------------------------------------
def _basis(n):
    """Tangents t, o of unit normals (Duff et al., JCGT 2017)."""
    x, y, z = n.unbind(1)
    s = torch.copysign(torch.ones_like(z), z)
    a = -1.0 / (s + z)
    b = x * y * a
    return torch.stack([1.0 + s * x * x * a, s * b, -s * x], 1), torch.stack([b, s + y * y * a, -y], 1)


def _dot(a, b):
    return (a * b).sum(1)


def _pairs(pos, r, h, lo, hi, periodic, scene):
    """Pairs i < j whose hulls meet, by a cell grid."""
    L = torch.tensor(hi, device=DEV) - torch.tensor(lo, device=DEV)
    width = 2.0 * float((r + h).max()) * (1.0 + 1e-9)
    dims = torch.clamp((L / width).floor(), min=1.0).to(torch.int64)
    d = [int(x) for x in dims]
    c = ((pos - torch.tensor(lo, device=DEV)) / L * dims).floor().to(torch.int64)
    c = torch.minimum(torch.clamp(c, min=0), dims - 1)
    key = (c[:, 2] * d[1] + c[:, 1]) * d[0] + c[:, 0]
    order = torch.argsort(key, stable=True)
    count = torch.bincount(key, minlength=d[0] * d[1] * d[2])
    start = torch.cumsum(count, 0) - count
    P, Q = [], []
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                q = c + torch.tensor([dx, dy, dz], device=DEV)
                ok = torch.ones(len(pos), dtype=torch.bool, device=DEV)
                for a in range(3):
                    if periodic[a]:
                        q[:, a] %= d[a]
                    else:
                        ok &= (q[:, a] >= 0) & (q[:, a] < d[a])
                qk = torch.where(ok, (q[:, 2] * d[1] + q[:, 1]) * d[0] + q[:, 0], 0)
                m = torch.where(ok, count[qk], 0)
                for k in range(int(m.max())):
                    i = torch.nonzero(m > k)[:, 0]
                    j = order[start[qk[i]] + k]
                    keep = i < j
                    if scene is not None:
                        keep &= scene[i] == scene[j]
                    i, j = i[keep], j[keep]
                    x = pos[i] - pos[j]
                    for a in range(3):
                        if periodic[a]:
                            x[:, a] -= L[a] * torch.round(x[:, a] / L[a])
                    dist = x.square().sum(1).sqrt()
                    keep = dist - r[i] - r[j] <= h[i] + h[j]
                    P.append(torch.stack([i[keep], j[keep]], 1))
                    Q.append(torch.cat([x[keep] / dist[keep, None], dist[keep, None]], 1))
    return torch.cat(P), torch.cat(Q)


def _mix(x):
    """splitmix64 on int64 bit patterns, as an order-preserving signed value."""
    def shr(v, k):
        return (v >> k) & ((1 << (64 - k)) - 1)
    s64 = lambda u: u - (1 << 64) if u >= 1 << 63 else u  # noqa: E731
    z = x + s64(0x9E3779B97F4A7C15)
    z = (z ^ shr(z, 30)) * s64(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * s64(0x94D049BB133111EB)
    return (z ^ shr(z, 31)) ^ s64(1 << 63)


def _colours(prio, a, b, n):
    """First-fit colours in decreasing priority, in Jones-Plassmann rounds; b >= n is a wall."""
    C_ = len(prio)
    colour = torch.full((C_,), -1, dtype=torch.int64, device=DEV)
    masks = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    bb = torch.clamp(b, max=n)
    left = torch.arange(C_, device=DEV)
    low = torch.iinfo(torch.int64).min
    while len(left):
        top = torch.full((n + 1,), low, dtype=torch.int64, device=DEV)
        top.scatter_reduce_(0, a[left], prio[left], "amax")
        top.scatter_reduce_(0, bb[left], prio[left], "amax")
        win = (top[a[left]] == prio[left]) & ((bb[left] == n) | (top[bb[left]] == prio[left]))
        w = left[win]
        used = masks[a[w]] | torch.where(bb[w] == n, 0, masks[bb[w]])
        free = ~used
        bit = free & -free
        colour[w] = torch.round(torch.log2(bit.to(torch.float64))).to(torch.int64)
        masks[a[w]] |= bit
        dyn = bb[w] < n
        masks[bb[w][dyn]] |= bit[dyn]
        left = left[~win]
    return colour


class _Reference:
    """Sphere scenes stepped in FP64."""

    def __init__(self, scenes, batch):
        p = scenes[0]["params"]
        cat = lambda k: torch.as_tensor(np.concatenate([s[k] for s in scenes]), device=DEV)  # noqa: E731
        self.p, self.r = p, cat("radius")
        self.n = len(self.r)
        sizes = torch.tensor([len(s["pos"]) for s in scenes], device=DEV)
        self.scene = torch.repeat_interleave(torch.arange(len(scenes), device=DEV), sizes)
        self.offset = torch.cumsum(sizes, 0) - sizes
        self.sizes, self.batch, self.S = sizes, batch, len(scenes)
        self.mu = torch.tensor([s["params"]["mu"] for s in scenes], dtype=torch.float64, device=DEV)
        self.planes = [s["planes"] for s in scenes]
        los, his = np.array([s["params"]["box_lo"] for s in scenes]), np.array([s["params"]["box_hi"] for s in scenes])
        self.lo, self.hi = los.min(0), his.max(0)
        self.periodic = p.get("periodic", (0, 0, 0))
        mass = 4.0 / 3.0 * math.pi * self.r ** 3
        self.im, self.iI = 1.0 / mass, 1.0 / (0.4 * mass * self.r ** 2)
        self.prev = None

    def step(self, pos, quat, vel, ang, sweeps, tol):
        p, n, dt = self.p, self.n, self.p["dt"]
        h = dt * (vel.norm(dim=1) + ang.norm(dim=1) * self.r) + p["tau"]
        pairs, geo = _pairs(pos, self.r, h, self.lo, self.hi, self.periodic, self.scene if self.batch else None)
        i, j = pairs.unbind(1)
        la, lb = geo[:, 3] - self.r[j], self.r[j]
        rows = [(i, j, geo[:, :3], geo[:, 3] - self.r[i] - self.r[j], la, lb)]
        for w in range(len(self.planes[0])):   # wall w of every scene
            nrm = torch.tensor([P[w][0] for P in self.planes], dtype=torch.float64, device=DEV)[self.scene]
            off = torch.tensor([P[w][1] for P in self.planes], dtype=torch.float64, device=DEV)[self.scene]
            sd = _dot(nrm, pos) - off
            k = torch.nonzero(sd - self.r <= h + p["tau"])[:, 0]
            wall = n + (6 * self.scene[k] + w if self.batch else torch.full_like(k, w))
            rows.append((k, wall, nrm[k], sd[k] - self.r[k], sd[k], torch.zeros_like(sd[k])))
        a, b, nrm, xi, la, lb = (torch.cat([row[q] for row in rows]) for q in range(6))
        key = (a << 32) | b
        order = torch.argsort(key)
        a, b, nrm, xi, la, lb, key = (x[order] for x in (a, b, nrm, xi, la, lb, key))
        sc = self.scene[a]
        # priorities from keys in the scene's own numbering
        bl = torch.where(b < n, b - self.offset[sc], self.sizes[sc] + (b - n) - (6 * sc if self.batch else 0))
        prio = _mix((((a - self.offset[sc]) << 32) | bl) ^ SEED)
        sub = p.get("subdomains")
        if sub == "jacobi":
            colour = torch.zeros_like(a)
        else:
            colour = _colours(prio, a, b, n)
        g = torch.tensor(p["gravity"], dtype=torch.float64, device=DEV)
        speed = torch.zeros(self.S, dtype=torch.float64, device=DEV).scatter_reduce_(0, self.scene, vel.norm(dim=1), "amax")
        vref = torch.clamp(speed, min=max(float(g.norm()) * dt, 1e-12))
        v, w = vel + dt * g, ang.clone()
        t, o = _basis(nrm)
        dyn = b < n
        bz = torch.where(dyn, b, 0)
        zero = torch.zeros_like(xi)
        ima, iIa = self.im[a], self.iI[a]
        imb, iIb = torch.where(dyn, self.im[bz], zero), torch.where(dyn, self.iI[bz], zero)
        wn = ima + imb
        wt = wn + iIa * la ** 2 + iIb * lb ** 2
        bias = torch.where(xi >= 0, xi, p["beta"] * xi) / dt
        mu = self.mu[sc]
        imp = torch.zeros(len(a), 3, dtype=torch.float64, device=DEV)
        if self.prev is not None and p["warm_start"] == "prev" and len(self.prev[0]):
            at = torch.clamp(torch.searchsorted(self.prev[0], key), max=len(self.prev[0]) - 1)
            P = torch.where((self.prev[0][at] == key)[:, None], self.prev[1][at], 0.0)
            pn = torch.clamp(_dot(nrm, P), min=0.0)
            pt = torch.stack([_dot(t, P), _dot(o, P)], 1)
            ln = pt.norm(dim=1)
            pt = pt * torch.where(ln > mu * pn, mu * pn / torch.clamp(ln, min=1e-300), 1.0)[:, None]
            imp = torch.cat([pn[:, None], pt], 1)
        # velocity records of the contact ends: the bodies, or one per (body, subdomain)
        ra, rb, base = a, torch.where(dyn, b, n), None
        if sub is not None:
            if sub == "jacobi":
                s = torch.arange(len(a), device=DEV)
            else:
                c = torch.stack([torch.clamp(((pos[:, e] - self.lo[e]) * sub[e] / (self.hi[e] - self.lo[e])).floor(),
                                             0, sub[e] - 1) for e in range(3)], 1).to(torch.int64)
                s = ((c[:, 2] * sub[1] + c[:, 1]) * sub[0] + c[:, 0])[a]
            span = int(s.max()) + 1 if len(s) else 1
            ends, inv = torch.unique(torch.cat([a * span + s, bz[dyn] * span + s[dyn]]), return_inverse=True)
            base = ends // span
            ra = inv[:len(a)]
            rb = torch.full_like(a, len(base))
            rb[dyn] = inv[len(a):]

        def scatter(V, W, k, d):
            """Add the impulse change d (contact frame) of contacts k to the velocity records."""
            P = d[:, :1] * nrm[k] + d[:, 1:2] * t[k] + d[:, 2:] * o[k]
            q = torch.linalg.cross(nrm[k], P)
            V.index_add_(0, ra[k], ima[k, None] * P)
            W.index_add_(0, ra[k], -(la * iIa)[k, None] * q)
            V.index_add_(0, rb[k], -imb[k, None] * P)
            W.index_add_(0, rb[k], -(lb * iIb)[k, None] * q)

        every = torch.arange(len(a), device=DEV)
        pad = torch.zeros(1, 3, dtype=torch.float64, device=DEV)
        if base is None:
            V, W = torch.cat([v, pad]), torch.cat([w, pad])
            scatter(V, W, every, imp)
        else:
            V = torch.zeros(len(base) + 1, 3, dtype=torch.float64, device=DEV)
            W = torch.zeros_like(V)
            scatter(V, W, every, imp)
            v.index_add_(0, base, V[:-1])
            w.index_add_(0, base, W[:-1])
        lists = [torch.nonzero(colour == c)[:, 0] for c in range(int(colour.max()) + 1 if len(a) else 0)]
        done = torch.zeros(self.S, dtype=torch.bool, device=DEV)
        om = p["omega"]
        for _ in range(sweeps):
            if base is not None:
                V, W = torch.cat([v[base], pad]), torch.cat([w[base], pad])
            res = torch.zeros(self.S, dtype=torch.float64, device=DEV)
            for k in lists:
                if self.batch:
                    k = k[~done[sc[k]]]
                m = nrm[k]
                u = (V[ra[k]] - la[k, None] * torch.linalg.cross(W[ra[k]], m)) \
                    - (V[rb[k]] + lb[k, None] * torch.linalg.cross(W[rb[k]], m))
                old = imp[k]
                bn = _dot(m, u) - wn[k] * old[:, 0] + bias[k]
                bt = torch.stack([_dot(t[k], u), _dot(o[k], u)], 1) - wt[k, None] * old[:, 1:]
                yn = torch.clamp(-bn / wn[k], min=0.0)
                yt = -bt / wt[k, None]
                ln, lim = yt.norm(dim=1), mu[k] * yn
                yt = yt * torch.where(ln > lim, lim / torch.clamp(ln, min=1e-300), 1.0)[:, None]
                new = om * torch.cat([yn[:, None], yt], 1) + (1.0 - om) * old
                d = new - old
                imp[k] = new
                scatter(V, W, k, d)
                r = torch.sqrt((wn[k] * d[:, 0]) ** 2 + ((wt[k, None] * d[:, 1:]) ** 2).sum(1))
                res.scatter_reduce_(0, sc[k], r, "amax")
            if base is not None:
                v = v.index_add(0, base, V[:-1] - v[base])
                w = w.index_add(0, base, W[:-1] - w[base])
            if tol > 0.0:
                done |= res / vref <= tol
                if bool(done.all()):
                    break
        if base is None:
            v, w = V[:-1], W[:-1]
        self.prev = (key, imp[:, :1] * nrm + imp[:, 1:2] * t + imp[:, 2:] * o)
        pos = pos + dt * v
        for e in range(3):
            if self.periodic[e]:
                pos[:, e] = self.lo[e] + torch.remainder(pos[:, e] - self.lo[e], float(self.hi[e] - self.lo[e]))
        q0, q1, q2, q3 = quat.unbind(1)
        x, y, z = w.unbind(1)
        dq = torch.stack([-q1 * x - q2 * y - q3 * z, q0 * x + q3 * y - q2 * z, -q3 * x + q0 * y + q1 * z,
                          q2 * x - q1 * y + q0 * z], 1)
        quat = quat + 0.5 * dt * dq
        quat = quat / quat.norm(dim=1, keepdim=True)
        return pos, quat, v, w, dict(normal=nrm, xi=xi, impulse=imp)


def _mlp_reference(case, seed):
    theta, X, T = (x.double() for x in _mlp_inputs(case, seed))
    th = theta.clone().requires_grad_(True)
    grad, loss, out = torch.zeros_like(th), 0.0, []
    for x, y in zip(X.split(1 << 18), T.split(1 << 18)):
        at, hdn = 0, x
        for k, (i, o) in enumerate(zip(SIZES[:-1], SIZES[1:])):
            hdn = hdn @ th[at:at + o * i].view(o, i).T + th[at + o * i:at + o * i + o]
            at += o * i + o
            if k < 3:
                hdn = hdn * torch.sigmoid(hdn)
        Y = hdn + x[:, 3:6]
        if case["train"]:
            part = (Y - y).square().sum() / (2.0 * len(X))
            grad += torch.autograd.grad(part, th)[0]
            loss += float(part.detach())
        else:
            out.append(Y.detach())
    if not case["train"]:
        return torch.cat(out)
    m, v = 0.1 * grad, 0.001 * grad * grad
    new = theta - 2e-3 * (m / 0.1) / (torch.sqrt(v / 0.001) + 1e-8)
    return {"theta": new, "grad": grad, "m": m, "v": v, "loss": torch.tensor([loss], dtype=torch.float64, device=DEV)}


def exact(case, seed):
    if case["kind"] == "mlp":
        return _mlp_reference(case, seed)
    # a composite contact's sliding search is hundreds of operations per contact and colour, and a
    # body has up to dozens of contacts: minutes here
    if case["kind"] == "composite":
        return None
    scenes, vels, ang = _inputs(case, seed)
    batch = case["kind"] == "batch"
    ref = _Reference(scenes, batch)
    pos = torch.as_tensor(np.concatenate([s["pos"] for s in scenes]), device=DEV)
    quat = torch.zeros(len(pos), 4, dtype=torch.float64, device=DEV)
    quat[:, 0] = 1.0
    vel, ang = torch.as_tensor(vels[0], device=DEV), torch.as_tensor(ang, device=DEV)
    tol = case.get("tol", 0.0)
    if batch:
        ref.step(pos, quat, vel, ang, case["sweeps"], tol)   # the step that starts the history
    for _ in range(case.get("steps", 1)):
        pos, quat, vel, ang, con = ref.step(pos, quat, vel, ang, case["sweeps"], tol)
    got = {"pos": pos, "quat": quat, "vel": vel, "angvel": ang, "n_contacts": None, "n_colours": None}
    if case.get("contacts"):
        cap, m = _contact_cap(len(pos)), len(con["xi"])
        con["xi"] = con["xi"][:, None]
        for k, x in con.items():
            got[k] = torch.zeros(cap, x.shape[1], dtype=torch.float64, device=DEV)
            got[k][:m] = x
        got.update(j1=None, j2=None, colour=None)
    return got
