"""The dataflow sweeps against the other schedules of the same sweeps: the
kernels chosen by size (lanes per contact, warps), tiles that are not full,
bodies that take no impulses, the tolerance test, warm starts and omega."""
import numpy as np
import pytest

from paper_1501_05810_gb300 import scenes

pytestmark = pytest.mark.gpu

GLOBAL_SYNC = 1


def _scene(shape, precision, **kw):
    sc = scenes.hcp_packing(*shape, dt=5e-4, mu=0.5, precision=precision, warm_start="prev", **kw)
    rng = np.random.default_rng(sum(shape))
    n = len(sc["radius"])
    sc["radius"] = sc["radius"] * (1.0 - 1e-3 * rng.random(n))
    sc["pos"][:, :2] += 0.25
    sc["vel"] = rng.normal(0.0, 0.01, (n, 3))
    sc["angvel"] = rng.normal(0.0, 0.01, (n, 3))
    return sc


def _run(sc, flags, tol, sweeps, fixed):
    from paper_1501_05810_gb300 import nbgs
    s = dict(sc)
    s["params"] = dict(sc["params"], sweep_flags=flags)
    g = nbgs.Scene(s)
    if fixed:   # every fifth body has no linear, every seventh no angular mobility; some have neither
        n = g.n
        m = 4.0 / 3.0 * np.pi * sc["radius"] ** 3
        im, iI = 1.0 / m, 2.5 / (m * sc["radius"] ** 2)
        i = np.arange(n)
        im[i % 5 == 0] = 0.0
        iI[(i % 7 == 0) | (i % 10 == 0)] = 0.0
        g.set_mass_properties(im, iI)
    out = []
    for _ in range(2):   # a cold and a warm-started step
        st = g.step(sweeps, tol)
        b = g.get_bodies()
        out.append((st, g.residual_history(), b, g.get_contacts()))
    g.close()
    return out


@pytest.mark.parametrize("shape,precision,tol,omega,fixed", [
    ((5, 6, 2), "fp32", 0.0, 1.0, False), ((5, 6, 4), "fp32", 1e-3, 1.0, True),
    ((5, 6, 2), "fp32", 1e30, 1.0, False), ((30, 30, 30), "fp32", 2e-2, 1.0, False), ((5, 6, 4), "fp32", 1e-30, 1.0, True),
    ((12, 12, 12), "fp64", 1e-2, 1.0, False), ((44, 46, 44), "fp32", 2e-2, 1.0, False), ((9, 10, 9), "fp32", 0.0, 0.8, True),
    ((44, 46, 44), "fp32", 0.0, 1.0, False), ((45, 46, 46), "fp32", 0.0, 1.0, False),
    ((70, 72, 70), "fp32", 0.0, 1.0, True), ((5, 6, 2), "fp64", 0.0, 1.0, True), ((7, 8, 6), "fp64", 1e-6, 0.9, True),
    ((40, 40, 39), "fp64", 0.0, 1.0, False), ((40, 42, 40), "fp64", 0.0, 1.0, True)])
def test_flow_equals_grid_synchronised_sweeps(shape, precision, tol, omega, fixed):
    sc = _scene(shape, precision, omega=omega)
    sweeps = 12
    flow, ref = _run(sc, 0, tol, sweeps, fixed), _run(sc, GLOBAL_SYNC, tol, sweeps, fixed)
    for (sa, ha, ba, ca), (sb, hb, bb, cb) in zip(flow, ref):
        assert sa["n_contacts"] == sb["n_contacts"] and sa["n_colours"] == sb["n_colours"]
        assert sa["sweeps_done"] == sb["sweeps_done"]
        for k in ("j1", "j2", "colour"):
            assert np.array_equal(ca[k], cb[k])
        if precision == "fp32":   # the same roundings in every kernel
            for k in ("pos", "quat", "vel", "angvel"):
                assert np.array_equal(ba[k], bb[k]), k
            assert np.array_equal(ca["impulse"], cb["impulse"])
            assert np.array_equal(ha, hb) and sa["residual"] == sb["residual"]
        else:
            # a few roundings of 1.1e-16 per relaxation, some 12 x 12 relaxations per body and step, two
            # steps, passed on with a gain of at most 10
            bound = 1.1e-16 * 4 * 144 * 2 * 10
            for k in ("vel", "angvel"):
                assert np.abs(ba[k] - bb[k]).max() <= bound * np.abs(bb[k]).max()
            assert np.abs(ca["impulse"] - cb["impulse"]).max() <= bound * np.abs(cb["impulse"]).max()


@pytest.mark.parametrize("shape,sub,precision,tol,fixed", [
    ((5, 6, 2), (2, 2, 2), "fp32", 0.0, False), ((5, 6, 4), "jacobi", "fp32", 0.0, True),
    ((9, 10, 9), (3, 1, 2), "fp32", 1e-3, True), ((20, 20, 20), (20, 20, 20), "fp32", 0.0, False),
    ((44, 46, 44), (4, 4, 1), "fp32", 0.0, True), ((55, 56, 54), (8, 8, 1), "fp32", 0.0, False),
    ((55, 56, 54), "jacobi", "fp32", 0.0, False), ((7, 8, 6), (2, 2, 2), "fp64", 1e-6, True),
    ((9, 10, 9), "jacobi", "fp64", 0.0, False), ((40, 42, 40), (5, 5, 5), "fp64", 0.0, True)])
def test_subdomain_flow_equals_grid_synchronised_sweeps(shape, sub, precision, tol, fixed):
    """Bodies with one instance, a few, one per contact; sums that fill no
    tile or more than the grid has warps."""
    sc = _scene(shape, precision, omega=0.5, subdomains=sub)
    sweeps = 12
    flow, ref = _run(sc, 0, tol, sweeps, fixed), _run(sc, GLOBAL_SYNC, tol, sweeps, fixed)
    for (sa, ha, ba, ca), (sb, hb, bb, cb) in zip(flow, ref):
        assert sa["n_contacts"] == sb["n_contacts"] and sa["n_colours"] == sb["n_colours"]
        assert sa["sweeps_done"] == sb["sweeps_done"]
        if precision == "fp32":   # the same roundings in every kernel
            for k in ("pos", "quat", "vel", "angvel"):
                assert np.array_equal(ba[k], bb[k]), k
            assert np.array_equal(ca["impulse"], cb["impulse"])
            assert np.array_equal(ha, hb) and sa["residual"] == sb["residual"]
        else:   # as above
            bound = 1.1e-16 * 4 * 144 * 2 * 10
            for k in ("vel", "angvel"):
                assert np.abs(ba[k] - bb[k]).max() <= bound * np.abs(bb[k]).max()
            assert np.abs(ca["impulse"] - cb["impulse"]).max() <= bound * np.abs(cb["impulse"]).max()


@pytest.mark.parametrize("sizes,precision,tol", [
    ((1, 1, 2), "fp32", 1e-6), ((60, 151, 300, 97, 420, 33), "fp32", 1e-6), ((60, 151, 300), "fp32", 1e300),
    ((37,) * 700, "fp32", 1e-4), ((2000, 20, 9000, 400, 20000), "fp32", 0.0), ((300, 20, 900), "fp64", 0.0)])
def test_batch_flow_equals_grid_synchronised_sweeps(sizes, precision, tol):
    """Scenes that share tiles or fill many, that meet their tolerance at
    different sweeps, at once or never, with more scenes than a block has
    threads."""
    from paper_1501_05810_gb300 import nbgs
    rng = np.random.default_rng(len(sizes))
    scs = []
    for k, n in enumerate(sizes):
        sc = scenes.batch_scene(k, n, mu=float(rng.uniform(0.2, 0.8)), precision=precision, warm_start="prev")
        sc["vel"], sc["angvel"] = rng.normal(0.0, 2.0, (2, n, 3))
        sc["params"]["dt"] = 0.03
        scs.append(sc)
    out = []
    for flags in (0, GLOBAL_SYNC):
        batch = scenes.layout_batch(scs)
        for sc in batch:
            sc["params"] = dict(sc["params"], sweep_flags=flags)
        g = nbgs.BatchScene(batch)
        got = [g.step_scenes(30, tol) for _ in range(2)]
        out.append((got, g.residual_history(), g.get_bodies(), g.get_contacts()))
        g.close()
    (ga, ha, ba, ca), (gb, hb, bb, cb) = out
    for (ka, ra), (kb, rb) in zip(ga, gb):
        assert np.array_equal(ka, kb)
        if precision == "fp32":
            assert np.array_equal(ra, rb)
    if precision == "fp32":   # the same roundings in every kernel
        assert np.array_equal(ha, hb) and np.array_equal(ca["impulse"], cb["impulse"])
        for k in ("pos", "quat", "vel", "angvel"):
            assert np.array_equal(ba[k], bb[k]), k
    else:   # as above, with 30 sweeps a step
        bound = 1.1e-16 * 4 * 360 * 2 * 10
        for k in ("vel", "angvel"):
            assert np.abs(ba[k] - bb[k]).max() <= bound * np.abs(bb[k]).max()


@pytest.mark.parametrize("shape,precision,tol", [((2, 2, 2), "fp32", 0.0), ((6, 5, 4), "fp64", 1e-4), ((7, 7, 7), "fp32", 1e-3),
                                                 ((40, 40, 38), "fp32", 0.0), ((85, 85, 84), "fp32", 0.0),
                                                 ((25, 25, 24), "fp64", 0.0)])
def test_composite_flow_equals_grid_synchronised_sweeps(shape, precision, tol):
    """Lanes per contact by size (8, 4, 1); the slides found by several lanes
    against the serial search."""
    from paper_1501_05810_gb300 import nbgs
    sc = scenes.composite_gas(*shape, seed=1, spacing=0.97, v_max=0.5, dt=5e-3, mu=0.4, omega=0.9,
                              gravity=(0.0, 0.0, -9.81), precision=precision, warm_start="prev")
    sc["vel"][:, 2] -= 3.0
    out = []
    for flags in (0, GLOBAL_SYNC):
        s = dict(sc)
        s["params"] = dict(sc["params"], sweep_flags=flags)
        g = nbgs.Scene(s)
        steps = [g.step(10, tol) for _ in range(2)]
        out.append((steps, g.get_bodies(), g.get_contacts()))
        g.close()
    (sa, ba, ca), (sb, bb, cb) = out
    for x, y in zip(sa, sb):
        assert x["n_contacts"] == y["n_contacts"] and x["n_colours"] == y["n_colours"]
    assert np.array_equal(ca["j1"], cb["j1"]) and np.array_equal(ca["j2"], cb["j2"])
    # a few roundings per relaxation, some 8 x 10 relaxations per body and step, two steps, a gain of at most 10;
    # where the tolerance may end one sweep earlier, what such a sweep still changes
    eps = 6e-8 if precision == "fp32" else 1.1e-16
    bound = eps * 4 * 80 * 2 * 10 + 10 * tol
    for k in ("vel", "angvel"):
        assert np.abs(ba[k] - bb[k]).max() <= bound * np.abs(bb[k]).max()
    assert np.abs(ca["impulse"] - cb["impulse"]).max() <= bound * np.abs(cb["impulse"]).max()
