"""Contact detection against the oracle's test of every pair: grids of one,
three and more cells per axis, images across faces, edges and corners, hulls
that just touch, hulls far apart in size."""
import numpy as np
import pytest

from paper_1501_05810_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,side,periodic,r,speed,precision", [
    (1, 4.0, (0, 0, 0), (0.5, 0.5), 0.0, "fp32"), (129, 3.7, (1, 1, 1), (0.3, 0.5), 0.0, "fp32"),
    (60, 2.0, (0, 0, 0), (0.2, 0.4), 3.0, "fp32"), (300, 6.0, (1, 0, 1), (0.2, 0.4), 0.5, "fp64"),
    (400, 6.0, (0, 1, 0), (0.2, 0.4), 0.5, "fp32"), (700, 9.0, (1, 1, 1), (0.05, 0.5), 2.0, "fp32"),
    (1000, 12.5, (1, 1, 0), (0.5, 0.5), 0.01, "fp64"), (343, 7.0, (1, 1, 1), (0.49, 0.49), 0.0, "fp32")])
def test_contacts_equal_every_pair_tested(oracle_mod, n, side, periodic, r, speed, precision):
    from paper_1501_05810_gb300 import nbgs as nb
    rng = np.random.default_rng(n)
    if n == 343:   # a lattice whose hulls meet but for rounding: 1 - 0.49 - 0.49 > 0.01 + 0.01 in FP64
        pos = np.stack(np.meshgrid(*[np.arange(7) + 0.5] * 3, indexing="ij"), -1).reshape(-1, 3)
        tau = 0.01
    else:
        pos, tau = rng.uniform(0.0, side, (n, 3)), 1e-3
    prm = scenes.default_params(dt=1e-2, tau=tau, gravity=(0, 0, 0), box_lo=(0.0,) * 3, box_hi=(side,) * 3,
                                periodic=periodic, precision=precision)
    walls = scenes.box_walls((0.0,) * 3, (side,) * 3, axes=[a for a in range(3) if not periodic[a]])
    vel, ang = rng.normal(0.0, 1.0, (2, n, 3)) * speed
    if precision == "fp32":   # the state that the scene holds
        vel, ang = vel.astype(np.float32).astype(float), ang.astype(np.float32).astype(float)
    sc = scenes._scene("cloud", prm, pos, vel, ang, rng.uniform(*r, n), np.ones(n), walls)
    g, o = nb.Scene(sc), oracle_mod.OracleScene(sc)
    assert g.detect_contacts() == o.detect_contacts()
    cg, co = g.get_contacts(), o.get_contacts()
    for k in ("j1", "j2", "xi", "normal"):
        assert np.array_equal(cg[k], co[k]), k
    assert (len(cg["j1"]) > 0) == (n != 343)
    g.close()
    o.close()
