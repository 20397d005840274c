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
