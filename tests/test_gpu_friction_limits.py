"""Friction coefficients at the ends of what a scene may have: 0, a tiny one
and an infinite one, on contacts that press, separate and slide."""
import numpy as np
import pytest

from paper_1501_05810_gb300 import scenes

pytestmark = pytest.mark.gpu


def _floor(n_side, mu, precision):
    """Separate spheres on a floor: pressed, resting, and just leaving it (no
    normal impulse), all sliding and spinning."""
    k = np.arange(n_side)
    xy = np.stack(np.meshgrid(k, k, indexing="ij"), -1).reshape(-1, 2) * 1.5
    n = len(xy)
    rng = np.random.default_rng(3)
    pos = np.concatenate([xy, np.full((n, 1), 0.5)], 1)
    vel = rng.normal(0.0, 1.0, (n, 3))
    vel[:, 2] = np.array([-1.0, 0.0, 0.2])[np.arange(n) % 3]
    prm = scenes.default_params(dt=1e-3, tau=5e-3, mu=mu, box_lo=(-5.0, -5.0, -5.0),
                                box_hi=(1.5 * n_side + 5.0,) * 2 + (5.0,), precision=precision)
    return scenes._scene("floor", prm, pos, vel, rng.normal(0.0, 1.0, (n, 3)), np.full(n, 0.5), np.ones(n),
                         [((0.0, 0.0, 1.0), 0.0)])


@pytest.mark.parametrize("mu", [0.0, 1e-300, 1e-30, 0.3, float("inf")])
@pytest.mark.parametrize("precision,rel", [("fp64", 1e-12), ("fp32", 1e-5)])   # one contact a body, 5 sweeps, ~30 roundings each
def test_friction_coefficients(oracle_mod, mu, precision, rel):
    from paper_1501_05810_gb300 import nbgs
    sc = _floor(9, mu, precision)
    g, o = nbgs.Scene(sc), oracle_mod.OracleScene(dict(sc, params=dict(sc["params"], precision="fp64")))
    a, b = g.step(5, 0.0), o.step(5, 0.0)
    assert a["n_contacts"] == b["n_contacts"] == 81
    x, y, p, q = g.get_bodies(), o.get_bodies(), g.get_contacts(), o.get_contacts()
    for u, v in ((x["vel"], y["vel"]), (x["angvel"], y["angvel"]), (p["impulse"], q["impulse"])):
        assert np.isfinite(v).all() and np.abs(u - v).max() <= rel * np.abs(v).max()
    g.close()


@pytest.mark.parametrize("precision,n_side", [("fp64", 260), ("fp32", 260), ("fp32", 600), ("fp32", 1000)])
def test_infinite_friction_in_every_kernel(precision, n_side):
    """The kernels of larger scenes (one lane a contact) against the sweeps
    with a barrier after every colour."""
    from paper_1501_05810_gb300 import nbgs
    sc, out = _floor(n_side, float("inf"), precision), []
    for flags in (0, nbgs.NBGS_SWEEP_GLOBAL_SYNC):
        g = nbgs.Scene(dict(sc, params=dict(sc["params"], sweep_flags=flags)))
        assert g.step(5, 0.0)["n_contacts"] == n_side ** 2
        out.append((g.get_bodies(), g.get_contacts()["impulse"]))
        g.close()
    (x, p), (y, q) = out
    for u, v in ((x["vel"], y["vel"]), (x["angvel"], y["angvel"]), (p, q)):
        assert np.isfinite(v).all()
        assert np.abs(u - v).max() <= (1e-12 * np.abs(v).max() if precision == "fp64" else 0.0)


@pytest.mark.parametrize("density", [1e-152, 1e-118, 1e-112, 1e-77, 1.0, 1e77, 1e112, 1e118, 1e140])
def test_sliding_over_the_exponents(oracle_mod, density):
    """Sliding impulses whose squares reach from the first subnormals to 1e280:
    FP64 sweeps against the oracle's square root and division."""
    from paper_1501_05810_gb300 import nbgs
    sc = _floor(9, 0.3, "fp64")
    sc["density"] = np.full(81, density)
    g, o = nbgs.Scene(sc), oracle_mod.OracleScene(sc)
    a, b = g.step(5, 0.0), o.step(5, 0.0)
    assert a["n_contacts"] == b["n_contacts"] == 81
    x, y, p, q = g.get_bodies(), o.get_bodies(), g.get_contacts(), o.get_contacts()
    for u, v in ((x["vel"], y["vel"]), (x["angvel"], y["angvel"]), (p["impulse"], q["impulse"])):
        assert np.isfinite(v).all() and np.abs(u - v).max() <= 1e-12 * np.abs(v).max()
    slides = np.hypot(q["impulse"][:, 1], q["impulse"][:, 2]) > 0.299 * q["impulse"][:, 0]
    assert slides.sum() > 10
    g.close()
