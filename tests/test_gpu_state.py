"""State transfer from and to arrays on the GPU, on the host, off the
alignment of doubles, overlapping, and with some left out."""
import numpy as np
import pytest

from paper_1501_05810_gb300 import scenes

pytestmark = pytest.mark.gpu
WIDTH = {"pos": 3, "quat": 4, "vel": 3, "angvel": 3}


def _shifted(torch, a, off):
    """a's doubles on the GPU at a byte offset in a larger block."""
    raw = torch.zeros(a.nbytes + 64, dtype=torch.uint8, device="cuda")
    raw[off:off + a.nbytes] = torch.as_tensor(np.frombuffer(a.tobytes(), np.uint8).copy(), device="cuda")
    return raw, raw.data_ptr() + off


@pytest.mark.parametrize("n,precision,off", [(1, "fp64", 0), (33, "fp64", 4), (257, "fp32", 8), (1000, "fp64", 24)])
def test_state_round_trip(n, precision, off):
    import torch
    from paper_1501_05810_gb300 import nbgs
    lib, rng = nbgs.library(), np.random.default_rng(n)
    pos = rng.uniform(1.0, 49.0, (n, 3))
    prm = scenes.default_params(box_lo=(0.0,) * 3, box_hi=(50.0,) * 3, precision=precision)
    g = nbgs.Scene(scenes._scene("state", prm, pos, np.zeros((n, 3)), np.zeros((n, 3)), np.full(n, 0.1), np.ones(n), []))
    want = {"pos": pos[::-1].copy(), "quat": rng.normal(size=(n, 4)), "vel": rng.normal(size=(n, 3)),
            "angvel": rng.normal(size=(n, 3))}
    if precision == "fp32":
        want.update({k: want[k].astype(np.float32).astype(float) for k in ("vel", "angvel")})
    held = {k: _shifted(torch, a, off) for k, a in want.items()}
    torch.cuda.synchronize()
    assert lib.nbgs_set_bodies(g.h, *[held[k][1] for k in WIDTH]) == nbgs.NBGS_OK
    g.sync()
    got = g.get_bodies()   # to the host
    for k in WIDTH:
        assert np.array_equal(got[k], want[k]), k
    new = rng.normal(size=(n, 3)).astype(np.float32).astype(float)
    raw, p = _shifted(torch, new, off)
    torch.cuda.synchronize()
    assert lib.nbgs_update_bodies(g.h, None, None, p, None) == nbgs.NBGS_OK   # one array only
    g.sync()
    want["vel"] = new
    out = {k: _shifted(torch, np.zeros_like(a), off) for k, a in want.items()}
    torch.cuda.synchronize()
    assert lib.nbgs_get_bodies(g.h, out["pos"][1], None, out["vel"][1], out["angvel"][1]) == nbgs.NBGS_OK
    for k in ("pos", "vel", "angvel", "quat"):
        a = out[k][0][off:off + want[k].nbytes].cpu().numpy().tobytes()
        assert a == (want[k] if k != "quat" else np.zeros_like(want[k])).tobytes(), k
    # overlapping arrays: pos, then vel from its second body on
    both, p = _shifted(torch, np.zeros((n + 1, 3)), off)
    torch.cuda.synchronize()
    assert lib.nbgs_get_bodies(g.h, p, None, p + 24, None) == nbgs.NBGS_OK
    a = np.frombuffer(both[off:off + 24 * (n + 1)].cpu().numpy().tobytes()).reshape(n + 1, 3)
    assert np.array_equal(a[0], want["pos"][0]) and np.array_equal(a[1:], want["vel"])
    g.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("lo", [0.0, -3.0])
def test_integrate_at_the_edges_of_formats_and_boxes(precision, lo):
    """Conversions of numbers that FP32 holds exactly, rounded or not at all,
    and the wrap of positions on, next to and beyond the faces."""
    from paper_1501_05810_gb300 import nbgs
    R = np.float32 if precision == "fp32" else np.float64
    hi = lo + 10.0
    a = np.array([1.0, -2.5, 0.1, 1.0 / 3.0, -1e-18, 1.17549435e-38 * 2.0 ** 70, 2.0 ** 60, 1.0 + 2.0 ** -23, 1.0 + 2.0 ** -24])
    x = np.array([lo, hi, np.nextafter(hi, lo), np.nextafter(lo, -10.0), lo + 5.0, hi + 12.3, lo - 1e-300, -0.0, 1e-310])
    n = len(a)
    pos = np.stack([x, np.roll(x, 3), np.roll(x, 5)], -1)
    prm = scenes.default_params(box_lo=(lo,) * 3, box_hi=(hi,) * 3, periodic=(1, 1, 1), precision=precision)
    g = nbgs.Scene(scenes._scene("edges", prm, pos, np.zeros((n, 3)), np.zeros((n, 3)), np.full(n, 0.1), np.ones(n), []))
    quat = np.zeros((n, 4))
    quat[np.arange(n), np.arange(n) % 4] = a
    g.set_bodies(pos, quat, np.zeros((n, 3)), np.zeros((n, 3)))
    g.integrate()
    b = g.get_bodies()
    f = a.astype(R)
    want = np.zeros((n, 4))
    want[np.arange(n), np.arange(n) % 4] = (f * (R(1) / np.sqrt(f * f))).astype(np.float64)
    assert np.array_equal(b["quat"], want)
    s = np.fmod(pos - lo, 10.0)
    wrapped = np.where((pos >= lo) & (pos < lo + 10.0), pos, lo + np.where(s < 0.0, s + 10.0, s))
    assert np.array_equal(b["pos"], wrapped)
    g.close()
