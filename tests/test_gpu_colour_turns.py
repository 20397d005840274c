"""The colouring in turns (scenes of some 10^6 contacts on): every contact has
the smallest colour that none of its predecessors (incident contacts of higher
priority) has, which is the sequential greedy colouring; lists of up to 16
contacts and longer ones, 7 turns and 12."""
import numpy as np
import pytest

from paper_1501_05810_gb300 import scenes

pytestmark = pytest.mark.gpu


def _mixed_radii(m):
    """A cubic packing with every 64th sphere large: lists of more than 16 contacts among short ones."""
    k = np.arange(m)
    idx = np.stack(np.meshgrid(k, k, k, indexing="ij"), -1).reshape(-1, 3)
    r = np.where(np.all(idx % 4 == 2, axis=1), 1.2, 0.5)
    hi = (m + 0.5,) * 3
    prm = scenes.default_params(dt=5e-4, tau=0.004, box_lo=(0.0,) * 3, box_hi=hi, precision="fp32")
    z = np.zeros(idx.shape)
    return scenes._scene("radii", prm, idx + 0.75, z, z, r, np.ones(len(r)), scenes.box_walls((0,) * 3, hi))


@pytest.mark.parametrize("kind,size,least", [("radii", 68, 900_000), ("hcp", 54, 900_000), ("hcp", 128, 12_000_000)])
def test_colours_of_large_scenes_are_first_fit(kind, size, least):
    import torch
    from paper_1501_05810_gb300 import nbgs
    if kind == "radii":
        sc = _mixed_radii(size)
    else:
        sc = scenes.hcp_packing(size, size, size, dt=5e-4, precision="fp32")
        sc["pos"][:, :2] += 0.25
    g = nbgs.Scene(sc)
    for _ in range(2):   # the second step knows the number of contacts
        g.detect_contacts()
        assert g.colour_contacts() < 31
    c, n = g.get_contacts(), g.n
    g.close()
    z = ((c["j1"].astype(np.uint64) << np.uint64(32)) | c["j2"]) ^ np.uint64(sc["params"]["colour_seed"])
    z += np.uint64(0x9E3779B97F4A7C15)
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    prio = torch.as_tensor((z ^ (z >> np.uint64(31))).view(np.int64) ^ np.int64(-2 ** 63), device="cuda")
    j1, j2, col = (torch.as_tensor(c[k].astype(np.int64), device="cuda") for k in ("j1", "j2", "colour"))
    m = len(j1)
    assert m >= least and int(col.min()) == 0
    order = torch.sort(prio, descending=True, stable=True).indices   # ties to the lower index
    pair = j2 < n                                                    # walls have no list
    ends = torch.cat([torch.stack([j1[order], order]), torch.stack([j2[order], order])[:, pair[order]]], 1)
    rank = torch.empty(m, dtype=torch.int64, device="cuda")
    rank[order] = torch.arange(m, device="cuda")
    ends = ends[:, torch.sort(rank[ends[1]], stable=True).indices]
    ends = ends[:, torch.sort(ends[0], stable=True).indices]         # by body, its contacts by priority
    body, who = ends
    bit = 1 << col[who]
    taken = torch.zeros_like(bit)                                    # colours before an entry in its list
    longest = int(torch.bincount(body).max())
    assert (longest > 16) == (kind == "radii")
    for o in range(1, longest):
        taken[o:] |= torch.where(body[o:] == body[:-o], bit[:-o], 0)
    before = torch.zeros(m, dtype=torch.int64, device="cuda")
    first = torch.zeros(m, dtype=torch.bool, device="cuda")
    first[who] = True
    assert bool(first.all())
    is_a = j1[who] == body
    before[who[is_a]] |= taken[is_a]
    before[who[~is_a]] |= taken[~is_a]
    want = torch.zeros_like(col)
    for k in range(31):
        want = torch.where((want == k) & ((before >> k) & 1 == 1), k + 1, want)
    assert torch.equal(want, col)
