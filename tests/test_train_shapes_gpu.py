"""The training products at the edges of their tiles: rows in fours, k in
chunks of 128 cut into four slices, up to 64 hidden units, 256 outputs a
block.  Loss and gradient against the fp64 oracle."""
import numpy as np
import pytest

import paper_2506_20994_gb300 as ax
from oracle import mlp as omlp
from paper_2506_20994_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sym", [False, True])
@pytest.mark.parametrize("n_in,n_hid,B", [(1, 1, 1), (3, 2, 5), (27, 63, 127), (129, 64, 128),
                                          (343, 33, 129), (257, 48, 513), (4096, 64, 3)])
def test_loss_and_gradient_at_tile_edges(n_in, n_hid, B, sym):
    g = synth.rng(7 * n_in + B)
    nw = n_in * n_hid
    W1 = g.normal(size=(n_in, n_hid)) / np.sqrt(n_in)
    theta = np.concatenate([W1.ravel(), 0.1 * g.normal(size=n_hid),
                            g.normal(size=nw) / np.sqrt(n_hid), 0.1 * g.normal(size=n_in)])
    if sym:
        theta = np.concatenate([W1.ravel(), np.zeros(n_hid), W1.T.ravel(), np.zeros(n_in)])
    theta = theta.astype(np.float32)
    X, T = (g.normal(size=(B, n_in)).astype(np.float32) for _ in range(2))
    M = ax.Mlp(n_in, n_hid, params=theta, arch=ax.AX_MLP_SYM if sym else ax.AX_MLP_TANH)
    t = lambda a: torch.as_tensor(a, device="cuda")
    for _ in range(2):  # the second call reuses the workspace
        L, grad = M.loss_grad(t(X), t(T))
    f = omlp.mse_loss_grad_sym if sym else omlp.loss_and_grad
    L_ref, g_ref = f(theta.astype(np.float64), X, T, n_hid)
    # fp32 sums of up to 4096 terms in chains of at most 1024: their rounding
    # errors add like a random walk, 32 eps = 2e-6; two such sums in a row
    assert abs(L - L_ref) <= 1e-5 * max(L_ref, 1e-30)
    assert np.linalg.norm(grad - g_ref) <= 1e-5 * np.linalg.norm(g_ref)
    if sym:
        assert not grad[nw:].any()
