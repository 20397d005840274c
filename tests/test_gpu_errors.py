"""States that a step must refuse: what the solve does when the colouring or
the detection has reached a limit, and what the caller is told."""
import numpy as np
import pytest

from paper_1501_05810_gb300 import scenes

pytestmark = pytest.mark.gpu


def _hub(n, r_shell=2.05, **params):
    """A sphere of radius 2 (the last body) in a shell of n small ones at r_shell."""
    d = np.random.default_rng(n).normal(size=(n, 3))
    pos = np.concatenate([d / np.linalg.norm(d, axis=1, keepdims=True) * r_shell, np.zeros((1, 3))]) + 5.0
    prm = scenes.default_params(dt=1e-4, tau=5e-3, gravity=(0, 0, 0), box_lo=(0.0,) * 3, box_hi=(10.0,) * 3, **params)
    return scenes._scene("hub", prm, pos, np.zeros_like(pos), np.zeros_like(pos), np.r_[np.full(n, 0.05), 2.0],
                         np.ones(n + 1), [])


@pytest.mark.parametrize("kind,precision,tol", [
    ("spheres", "fp32", 0.0), ("spheres", "fp32", 1e-3), ("spheres", "fp64", 0.0), ("spheres", "fp64", 1e-3),
    ("grid", "fp32", 0.0), ("grid", "fp64", 1e-3), ("composite", "fp32", 0.0), ("composite", "fp64", 1e-3)])
def test_more_colours_than_there_are(kind, precision, tol):
    """300 contacts of one body need 300 colours: a capacity error, at once
    (the wait for a version that never comes takes a second)."""
    import time
    from paper_1501_05810_gb300 import nbgs
    for n in (40, 300):   # the first loads the kernels
        sc = _hub(n, precision=precision, omega=0.5 if kind == "grid" else 1.0,
                  subdomains=(2, 2, 2) if kind == "grid" else None)
        g = nbgs.Scene(scenes.as_composites(sc) if kind == "composite" else sc)
        if n == 40:
            g.step(20, tol)
            g.close()
    g.sync()
    t = time.perf_counter()
    with pytest.raises(nbgs.NBGSError, match="256 colours") as e:
        g.step(20, tol)
    assert time.perf_counter() - t < 0.8
    assert e.value.status == nbgs.NBGS_ECAPACITY
    g.close()


def test_as_many_colours_as_there_are():
    """256 contacts of one body, all colours in use, are solved."""
    from paper_1501_05810_gb300 import nbgs
    ks = []
    for n in (230, 256):
        g = nbgs.Scene(_hub(n, precision="fp64"))
        st = g.step(20, 0.0)
        ks.append((st["n_colours"], st["sweeps_done"]))
        g.close()
    assert ks[0][0] >= 230 and ks[0][1] == ks[1][1] == 20 and ks[1][0] == 256


@pytest.mark.parametrize("limit", ["neighbours", "cells"])
def test_graph_steps_report_the_limits_of_the_detection(limit):
    """Replayed steps that drive a body past 32 neighbours of higher index, or
    the hulls past a third of a periodic box: reported like an ordinary step's."""
    from paper_1501_05810_gb300 import nbgs
    if limit == "neighbours":
        sc = _hub(40, r_shell=2.2)
        sc["params"]["dt"] = 1e-2
        sc["vel"][:-1] = (5.0 - sc["pos"][:-1]) / 2.2   # inwards at 1
        for k in ("pos", "vel", "angvel", "radius", "density"):
            sc[k] = np.ascontiguousarray(sc[k][::-1])   # the big sphere first: every pair is in its list
        status, text = nbgs.NBGS_ECAPACITY, "hull neighbours"
    else:
        sc = scenes.periodic_cloud(seed=1, per_side=6, gravity=(0.0, 0.0, -981.0))
        status, text = nbgs.NBGS_EINVAL, "fewer than 3 grid cells"
    a, b = nbgs.Scene(sc), nbgs.Scene(sc)
    with pytest.raises(nbgs.NBGSError, match=text):
        for _ in range(21):
            a.step(5, 0.0)
    b.step(5, 0.0)
    b.graph_step(5, 0.0, 20)
    with pytest.raises(nbgs.NBGSError, match=text) as e:
        b.sync()
    assert e.value.status == status
    a.close()
    b.close()


@pytest.mark.parametrize("refuse", [0, 1, 7, 15, 20, 21])
def test_no_memory_for_more_contacts(refuse):
    """The allocation that fails while the contact buffers grow: an error, and
    every buffer is given back once."""
    import torch
    from paper_1501_05810_gb300 import nbgs
    sc = scenes.hcp_packing(16, 16, 16, dt=5e-4, precision="fp32", contacts_per_body=1)
    sc["pos"][:, :2] += 0.25
    live, twice, left = set(), [], [None]
    proto_a, proto_f = nbgs.nbgs_allocator._fields_[1][1], nbgs.nbgs_allocator._fields_[2][1]

    def alloc(ctx, nbytes, stream):
        if left[0] is not None:
            left[0] -= 1
            if left[0] < 0:
                return None
        p = torch.cuda.caching_allocator_alloc(int(nbytes), 0, int(stream or 0))
        live.add(p)
        return p

    def free(ctx, p, stream):
        if p in live:
            live.remove(p)
            torch.cuda.caching_allocator_delete(int(p))
        else:
            twice.append(p)

    a = nbgs.nbgs_allocator(None, proto_a(alloc), proto_f(free))
    arrs = [np.ascontiguousarray(sc[k], dtype=np.float64) for k in ("pos", "vel", "angvel", "radius", "density")]
    params = nbgs.make_params(sc["params"])
    st, h = nbgs.nbgs_create_scene(params, len(sc["radius"]), *[nbgs._ptr(x) for x in arrs], a,
                                   torch.cuda.current_stream().cuda_stream)
    assert st == nbgs.NBGS_OK
    left[0] = refuse
    with pytest.raises(nbgs.NBGSError) as e:
        nbgs._call(h, "nbgs_detect_contacts", None)
    assert e.value.status == nbgs.NBGS_ENOMEM
    nbgs.library().nbgs_destroy_scene(h)
    assert not twice and not live
