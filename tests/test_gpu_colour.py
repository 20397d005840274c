"""The colouring against the sequential first-fit greedy colouring in
decreasing priority: queues that run empty, that overflow, several turns,
lists of one contact up to several hundred."""
import numpy as np
import pytest

from paper_1501_05810_gb300 import scenes

pytestmark = pytest.mark.gpu


def _greedy(j1, j2, n, seed, fixed):
    z = (((j1.astype(np.uint64) << np.uint64(32)) | j2.astype(np.uint64)) ^ np.uint64(seed)) + np.uint64(0x9E3779B97F4A7C15)
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    prio = z ^ (z >> np.uint64(31))
    order = np.argsort(~prio, kind="stable")   # ties to the lower key: canonical order
    used = [0] * n
    out = [0] * len(j1)
    a, b = j1.tolist(), j2.tolist()
    fin = [not f for f in fixed] + [False]
    for c in order.tolist():
        x, y = a[c], min(b[c], n)
        m = (used[x] if fin[x] else 0) | (used[y] if fin[y] else 0)
        bit = ~m & (m + 1)
        out[c] = bit.bit_length() - 1
        if fin[x]:
            used[x] |= bit
        if fin[y]:
            used[y] |= bit
    return np.array(out)


@pytest.mark.parametrize("kind,n", [("hcp", 72), ("hcp", 4000), ("hcp", 118000), ("hcp", 150000), ("hub", 40),
                                    ("hub", 200), ("hub", 300), ("pairs", 300000), ("fixed", 4000)])
def test_colours_equal_sequential_greedy(kind, n):
    from paper_1501_05810_gb300 import nbgs
    rng = np.random.default_rng(n)
    if kind in ("hcp", "fixed"):
        side = max(4, round(n ** (1 / 3) / 2) * 2)
        sc = scenes.hcp_packing(side, side, max(2, round(n / side ** 2 / 2) * 2), dt=5e-4)
        sc["pos"][:, :2] += 0.25
    else:
        if kind == "hub":   # a sphere in the middle of a shell of n small ones; the last body, so that all pairs are theirs
            d = rng.normal(size=(n, 3))
            pos = np.concatenate([d / np.linalg.norm(d, axis=1, keepdims=True) * 2.05, np.zeros((1, 3))]) + 5.0
            r = np.concatenate([np.full(n, 0.05), [2.0]])
            hi = 10.0
        else:               # n / 2 pairs: a contact each, no list longer than one
            m = round((n / 2) ** (1 / 3)) + 1
            g = np.stack(np.unravel_index(np.arange(n // 2), (m, m, m)), -1) * 3.0 + 1.0
            pos, r, hi = np.concatenate([g, g + [1.0, 0.0, 0.0]]), np.full(2 * (n // 2), 0.5), 3.0 * m + 1.0
        prm = scenes.default_params(dt=1e-4, tau=5e-3, gravity=(0, 0, 0), box_lo=(0.0,) * 3, box_hi=(hi,) * 3)
        sc = scenes._scene(kind, prm, pos, np.zeros_like(pos), np.zeros_like(pos), r, np.ones(len(r)), [])
    g = nbgs.Scene(sc)
    fixed = np.zeros(g.n, bool)
    if kind == "fixed":     # every third body takes no impulses and has no list
        fixed[::3] = True
        mass = 4.0 / 3.0 * np.pi * np.asarray(sc["radius"]) ** 3
        im, iI = 1.0 / mass, 2.5 / (mass * np.asarray(sc["radius"]) ** 2)
        im[fixed] = iI[fixed] = 0.0
        g.set_mass_properties(im, iI)
    g.detect_contacts()
    if kind == "hub" and n > 256:   # a colour each: refused
        with pytest.raises(nbgs.NBGSError, match="colours"):
            g.colour_contacts()
        return
    k = g.colour_contacts()
    c = g.get_contacts()
    want = _greedy(c["j1"], c["j2"], g.n, sc["params"]["colour_seed"], fixed)
    assert len(want) > 0 and k == want.max() + 1
    assert np.array_equal(c["colour"], want)
    g.close()
