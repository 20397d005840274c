"""The training kernel at the edges of its tiles: a group without a tile,
ragged tiles, one tile more than the grid takes at once, inputs that are not
16-byte aligned, non-finite inputs."""
import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,shift", [(1, 0), (127, 0), (128, 1), (129, 0), (256, 3), (257, 0), (3001, 2), (38913, 0)])
def test_gradient_at_tile_edges(n, shift):
    import torch
    from paper_1501_05810_gb300 import nbgs, warmstart as ws
    rng = np.random.default_rng(n)
    theta = ws.init_params(4) + rng.normal(0, 0.02, ws.N_PARAMS).astype(np.float32)
    X, T = rng.normal(size=(n, 12)).astype(np.float32), rng.normal(size=(n, 3)).astype(np.float32)
    th, Td = torch.as_tensor(theta, device="cuda"), torch.as_tensor(T, device="cuda")
    Xd = torch.zeros(n * 12 + shift, device="cuda")[shift:]
    Xd.copy_(torch.as_tensor(X.reshape(-1)))
    g, loss = torch.zeros(ws.N_PARAMS, device="cuda"), torch.zeros(1, dtype=torch.float64, device="cuda")

    def run():
        assert nbgs.library().nbgs_mlp_grad(th.data_ptr(), Xd.data_ptr(), Td.data_ptr(), n, g.data_ptr(), loss.data_ptr(),
                                            torch.cuda.current_stream().cuda_stream) == nbgs.NBGS_OK
        torch.cuda.synchronize()
        return g.cpu().numpy().astype(np.float64), loss.item()

    got, L = run()
    Lr, G = omlp.loss_and_grad_rounded(theta.astype(np.float64), X.astype(np.float64), T.astype(np.float64))
    # FP32 sums; an operand that FP32 rounds to the other BF16 neighbour moves by 2^-8, which in a few
    # samples may be a largest entry's own
    bound = 5e-4 + (2.0 ** -8 if n < 1000 else 0.0)
    assert abs(L - Lr) <= (1e-5 + (2.0 ** -8 if n < 1000 else 0.0)) * Lr
    assert np.abs(got - G).max() <= bound * np.abs(G).max()
    Xd[12 * (n // 2)] = float("nan")   # reaches the loss and every layer's gradient
    bad, L = run()
    assert np.isnan(L) and np.isnan(bad).any()
