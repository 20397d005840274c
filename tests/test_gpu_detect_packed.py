"""Detection in packed piles of composites, where warps work their queues of
pairs off together, against the kernel of a scene's first detection."""
import numpy as np
import pytest

from paper_1501_05810_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,precision", [((3, 3, 3), "fp32"), ((9, 8, 9), "fp32"), ((20, 21, 20), "fp32"), ((9, 8, 9), "fp64")])
def test_packed_composites_find_the_same_contacts(shape, precision):
    from paper_1501_05810_gb300 import nbgs
    sc = scenes.composite_gas(*shape, seed=2, spacing=1.02, v_max=0.5, dt=2e-2, mu=0.4, gravity=(0.0, 0.0, -9.81),
                              precision=precision, warm_start="prev")
    sc["vel"][:, 2] -= 3.0
    g = nbgs.Scene(sc)
    members, dense = len(sc["members"]["body"]), 0
    for _ in range(40):
        m = g.step(30, 0.0)["n_contacts"]
        b = g.get_bodies()
        f = nbgs.Scene(sc)
        f.set_bodies(b["pos"], b["quat"], b["vel"], b["angvel"])
        g.detect_contacts()
        f.detect_contacts()
        x, y = g.get_contacts(), f.get_contacts()
        f.close()
        for k in ("j1", "j2", "xi", "normal"):
            assert np.array_equal(x[k], y[k]), k
        dense += 2 * m >= 3 * members
    assert dense > 3
    g.close()
