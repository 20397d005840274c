"""Every schedule of the FP32 sweeps gives the same bits, for relaxation
parameters whose blend of old and new impulse rounds."""
import numpy as np
import pytest

from paper_1501_05810_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("omega", [0.3, 0.4, 0.75, 0.8, 1.1])
@pytest.mark.parametrize("sub", [None, (2, 3, 2), "jacobi"])
@pytest.mark.parametrize("side", [10, 18, 40])
def test_schedules_agree_to_the_bit(omega, sub, side):
    from paper_1501_05810_gb300 import nbgs
    if sub == "jacobi" and omega > 0.5:
        omega *= 0.4   # Jacobi diverges above
    sc = scenes.hcp_packing(side, side, side, dt=5e-4, mu=0.5, precision="fp32", warm_start="prev", omega=omega,
                            subdomains=sub)
    sc["vel"] = np.random.default_rng(2).normal(0.0, 0.01, sc["vel"].shape)
    sc["pos"][:, :2] += 0.25
    out = []
    for flags in (0, nbgs.NBGS_SWEEP_GLOBAL_SYNC, nbgs.NBGS_SWEEP_TMA_STAGE, nbgs.NBGS_SWEEP_WARP_SYNC,
                  nbgs.NBGS_SWEEP_GATHER2):
        g = nbgs.Scene(dict(sc, params=dict(sc["params"], sweep_flags=flags)))
        for _ in range(2):
            g.step(10, 0.0)
        out.append((g.residual_history(), g.get_contacts()["impulse"], g.get_bodies()))
        g.close()
    assert len(out[0][1]) > 4 * side ** 3
    for h, p, b in out[1:]:
        assert np.array_equal(h, out[0][0]) and np.array_equal(p, out[0][1])
        assert all(np.array_equal(b[k], out[0][2][k]) for k in ("vel", "angvel"))


@pytest.mark.parametrize("sweeps,tol", [(15, 0.0), (16, 0.0), (40, 1e-3), (40, 1e30)])
@pytest.mark.parametrize("shape", [(18, 18, 16), (18, 18, 17), (27, 26, 23), (27, 26, 24)])
def test_jacobi_schedules_by_size_give_the_same(shape, sweeps, tol):
    """Around 32k and 100k contacts and 16 sweeps, where the schedule of a solve
    without flags changes, against the sweeps with grid barriers; a second
    solve of the same contacts may take the other schedule."""
    from paper_1501_05810_gb300 import nbgs
    sc = scenes.hcp_packing(*shape, dt=5e-4, mu=0.5, precision="fp32", warm_start="prev", omega=0.4, subdomains="jacobi")
    rng = np.random.default_rng(2)
    sc["vel"] = rng.normal(0.0, 0.01, sc["vel"].shape)
    sc["pos"][:, :2] += 0.25
    out = []
    for flags in (0, nbgs.NBGS_SWEEP_GLOBAL_SYNC):
        g = nbgs.Scene(dict(sc, params=dict(sc["params"], sweep_flags=flags)))
        steps = [g.step(sweeps, tol) for _ in range(2)]
        g.detect_contacts()
        g.colour_contacts()
        solves = [g.solve_nbgs(20, 0.0), g.solve_nbgs(5, 0.0), g.solve_nbgs(20, 0.0)]
        out.append((steps, solves, g.residual_history(), g.get_bodies(), g.get_contacts()["impulse"]))
        g.close()
    (sa, ra, ha, ba, pa), (sb, rb, hb, bb, pb) = out
    assert sa == sb and ra == rb and np.array_equal(ha, hb) and np.array_equal(pa, pb)
    assert all(np.array_equal(ba[k], bb[k]) for k in ("pos", "quat", "vel", "angvel"))


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("kind", ["single", "graph", "batch"])
def test_bodies_without_contacts(precision, kind):
    """Few contacts among many bodies, some without linear or any mobility: the
    bodies that nothing touches move as under the other schedule."""
    from paper_1501_05810_gb300 import nbgs
    out = []
    for flags in (0, nbgs.NBGS_SWEEP_GLOBAL_SYNC):
        if kind == "batch":
            g = nbgs.BatchScene(scenes.batch_scenes(9, seed=3, n_lo=50, n_hi=900, precision=precision, sweep_flags=flags,
                                                    warm_start="prev"))
        else:
            g = nbgs.Scene(scenes.periodic_cloud(seed=4, per_side=16, spacing=1.1, dt=1e-2, gravity=(0.1, 0.2, -9.81),
                                                 precision=precision, sweep_flags=flags, warm_start="prev"))
        i, m = np.arange(g.n), 0.5
        im, iI = np.full(g.n, 1.0 / m), np.full(g.n, 10.0 / m)
        im[i % 5 == 0] = 0.0
        iI[(i % 7 == 0) | (i % 10 == 0)] = 0.0
        g.set_mass_properties(im, iI)
        g.step(12, 1e-6)
        if kind == "graph":
            g.graph_step(12, 1e-6, 3)
        else:
            for _ in range(3):
                g.step(12, 1e-6)
        b, c = g.get_bodies(), g.get_contacts()
        out.append((b, c["impulse"]))
        hit = np.zeros(g.n, bool)
        hit[c["j1"]] = hit[c["j2"][c["j2"] < g.n]] = True
        assert hit.any() and (~hit).sum() > g.n // 4
        g.close()
    (x, p), (y, q) = out
    rel = 0.0 if precision == "fp32" else 1e-11   # some 50 relaxations of a body, a few roundings each
    for k in ("pos", "quat", "vel", "angvel"):
        assert np.abs(x[k] - y[k]).max() <= rel * np.abs(y[k]).max()
    assert np.abs(p - q).max() <= rel * np.abs(q).max()
