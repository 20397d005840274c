"""Steps that find no contact: bodies in free flight before, between and after
steps with contacts, in every mode whose arrays follow the contacts."""
import numpy as np
import pytest

from paper_1501_05810_gb300 import scenes

pytestmark = pytest.mark.gpu


def _cube(spacing, m=4):
    """m^3 unit spheres on a lattice: spacing 3 touches nothing, 0.999 everything."""
    k = np.arange(m) - 0.5 * (m - 1)
    return np.stack(np.meshgrid(k, k, k, indexing="ij"), -1).reshape(-1, 3) * spacing


def _scene(**params):
    pos = _cube(3.0)
    rng = np.random.default_rng(5)
    prm = scenes.default_params(dt=1e-3, tau=1e-3, mu=0.5, box_lo=(-20.0,) * 3, box_hi=(20.0,) * 3, **params)
    vel = rng.normal(0.0, 0.05, pos.shape)
    return scenes._scene("cube", prm, pos, vel, 0.1 * vel[:, ::-1], np.full(len(pos), 0.5), np.ones(len(pos)), [])


@pytest.mark.parametrize("sub", [(2, 2, 2), "jacobi"])
@pytest.mark.parametrize("precision,rel", [("fp64", 1e-10), ("fp32", 2e-5)])   # fp32: 10 sweeps of some 30 roundings
def test_subdomain_steps_without_contacts(oracle_mod, sub, precision, rel):
    from paper_1501_05810_gb300 import nbgs
    sc = _scene(subdomains=sub, omega=0.6)
    g = nbgs.Scene(dict(sc, params=dict(sc["params"], precision=precision)))
    for spacing, touch in ((3.0, False), (0.999, True), (3.0, False), (0.999, True)):
        o = oracle_mod.OracleScene(sc)
        for s in (g, o):
            s.set_bodies(_cube(spacing), np.tile([1.0, 0.0, 0.0, 0.0], (64, 1)), sc["vel"], sc["angvel"])
        a, b = g.step(10, 0.0), o.step(10, 0.0)
        assert a["n_contacts"] == b["n_contacts"] and (a["n_contacts"] > 0) == touch
        assert len(g.get_subdomains()) == a["n_contacts"]
        x, y = g.get_bodies(), o.get_bodies()
        for k in ("vel", "angvel"):
            assert np.abs(x[k] - y[k]).max() <= rel * np.abs(y[k]).max()
    g.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("tol", [0.0, 1e-6])
def test_graph_step_without_contacts_has_its_own_outcome(precision, tol):
    """A replayed step that loses every contact reports what an ordinary step
    does: all sweeps, residual 0, not the outcome of the step before."""
    import ctypes
    from paper_1501_05810_gb300 import nbgs

    def outcome(g):
        k, r = ctypes.c_int32(), ctypes.c_double()
        nbgs._call(g.h, "nbgs_get_scene_stats", ctypes.byref(k), ctypes.byref(r))
        return k.value, r.value, g.residual_history().tolist()
    sc = _scene(precision=precision)
    a, b = nbgs.Scene(sc), nbgs.Scene(sc)
    for spacing, sweeps in ((0.999, 30), (0.999, 30), (3.0, 30), (0.999, 30), (3.0, 7)):
        for g in (a, b):
            g.update_bodies(_cube(spacing), None, sc["vel"], sc["angvel"])
        sa = a.step(sweeps, tol)
        if b.get_contacts()["j1"].size == 0 and sa["n_contacts"] > 0:
            b.step(sweeps, tol)      # sizes the buffers, or finds the contacts again
        else:
            b.graph_step(sweeps, tol, 1)
        assert (sa["n_contacts"] > 0) == (spacing < 1.0)
        assert outcome(a) == outcome(b)
    a.close()
    b.close()
