"""Replayed steps among other calls: a scene that replays does exactly what its
twin does with ordinary steps, whatever was called in between."""
import numpy as np
import pytest

from paper_1501_05810_gb300 import scenes

pytestmark = pytest.mark.gpu


def _pour(precision, warm):
    sc = scenes.loose_pour(seed=4, n=1500, precision=precision, warm_start=warm)
    sc["vel"] = np.random.default_rng(3).normal(0.0, 2.0, sc["vel"].shape)
    sc["params"]["dt"] = 0.02
    return sc


def _same(a, b, what):
    x, y, p, q = a.get_bodies(), b.get_bodies(), a.get_contacts(), b.get_contacts()
    for k in ("pos", "quat", "vel", "angvel"):
        assert np.array_equal(x[k], y[k]), (what, k)
    for k in ("j1", "j2", "colour", "normal", "xi", "impulse"):
        assert np.array_equal(p[k], q[k]), (what, k)


@pytest.mark.parametrize("precision,warm", [("fp32", "prev"), ("fp64", "prev"), ("fp32", "none"), ("fp64", "none")])
def test_replays_among_other_calls(precision, warm, tmp_path):
    from paper_1501_05810_gb300 import nbgs
    sc = _pour(precision, warm)
    a, b = nbgs.Scene(sc), nbgs.Scene(sc)
    start = a.get_bodies()
    ops = ["graph1", "graph2", "step", "graph1", "step", "step", "graph3", "update", "graph1", "set", "graph2", "step",
           "set", "graph1", "detect", "graph1", "graph1", "save", "step", "load", "step", "graph1", "step", "load", "graph2",
           "zero", "graph1"]
    for g in (a, b):
        g.step(20, 0.0)
    for k, op in enumerate(ops):
        if op.startswith("graph"):
            b.graph_step(20, 0.0, int(op[5:]))
            for _ in range(int(op[5:])):
                a.step(20, 0.0)
        for i, g in enumerate((a, b)):
            if op == "step":
                g.step(20, 0.0)
            elif op == "zero":
                g.step(0, 0.0)
            elif op == "update":
                s = g.get_bodies()
                g.update_bodies(s["pos"], s["quat"], 0.5 * s["vel"], s["angvel"])
            elif op == "set":
                g.set_bodies(start["pos"], start["quat"], start["vel"], start["angvel"])
            elif op == "detect":
                g.detect_contacts()
            elif op == "save":
                g.save_state(str(tmp_path / f"{i}.ckpt"))
            elif op == "load":
                g.load_state(str(tmp_path / f"{i}.ckpt"))
        if op not in ("set", "update", "detect", "load"):
            assert len(a.get_contacts()["j1"]) > 300
            _same(a, b, (k, op))
            assert np.array_equal(a.residual_history(), b.residual_history())
    a.close()
    b.close()


def test_calls_straight_after_replays(tmp_path):
    """Calls that read the contact count, with nothing in between that has
    brought it from the device."""
    from paper_1501_05810_gb300 import nbgs
    sc = _pour("fp32", "prev")
    a, b, c = nbgs.Scene(sc), nbgs.Scene(sc), nbgs.Scene(sc)
    for g in (a, b, c):
        g.step(20, 0.0)
    path = str(tmp_path / "replayed.ckpt")
    a.step(20, 0.0)
    b.graph_step(20, 0.0, 1)
    b.save_state(path)                    # the contacts there are, not the capacity
    c.graph_step(20, 0.0, 2)
    c.load_state(path)                    # its own replays end here
    for _ in range(2):
        for g in (a, b, c):
            g.step(20, 0.0)
        _same(a, b, "saved")
        _same(a, c, "loaded")
    b.graph_step(20, 0.0, 1)
    a.step(20, 0.0)
    assert len(b.get_subdomains()) == len(a.get_contacts()["j1"])
    b.graph_step(20, 0.0, 1)
    for g in (a, b):                      # after a step there are no coloured contacts to compute features of
        with pytest.raises(nbgs.NBGSError, match="detect and colour"):
            g.mlp_features()
        g.close()
    c.close()


def test_replays_after_changes_of_the_scene(tmp_path):
    """Walls, masses, warm start and parameters that change between replays."""
    from paper_1501_05810_gb300 import nbgs
    sc = _pour("fp32", "prev")
    a, b = nbgs.Scene(sc), nbgs.Scene(sc)
    other = nbgs.Scene(dict(sc, params=dict(sc["params"], mu=0.1, dt=5e-3, gravity=(3.0, 0.0, -4.0))))
    other.step(20, 0.0)
    other.save_state(str(tmp_path / "other.ckpt"))
    other.close()
    mass = 4.0 / 3.0 * np.pi * sc["radius"] ** 3
    hi = sc["params"]["box_hi"]
    changes = [lambda g: nbgs._call(g.h, "nbgs_add_plane", (nbgs.C.c_double * 3)(-1.0, 0.0, 0.0), 0.05 - float(hi[0])),
               lambda g: nbgs._call(g.h, "nbgs_set_warm_start", nbgs.NBGS_WARM_NONE),
               lambda g: g.set_mass_properties(0.5 / mass, 2.5 / (mass * sc["radius"] ** 2)),
               lambda g: nbgs._call(g.h, "nbgs_add_plane", (nbgs.C.c_double * 3)(0.0, -1.0, 0.0), 0.05 - float(hi[1])),
               lambda g: nbgs._call(g.h, "nbgs_set_warm_start", nbgs.NBGS_WARM_PREV),
               lambda g: g.load_state(str(tmp_path / "other.ckpt"))]
    for g in (a, b):
        g.step(20, 0.0)
    for k, change in enumerate(changes):
        b.graph_step(20, 0.0, 2)
        for _ in range(2):
            a.step(20, 0.0)
        for g in (a, b):
            change(g)
        if k == len(changes) - 1:   # other parameters and no solve since: an ordinary step first
            with pytest.raises(nbgs.NBGSError):
                b.graph_step(20, 0.0, 1)
            break
        a.step(20, 0.0)
        b.graph_step(20, 0.0, 1)
        assert len(a.get_contacts()["j1"]) > 100
        _same(a, b, k)
    a.close()
    b.close()
