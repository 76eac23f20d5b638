"""Convolutions of the guess network against the FP64 reference at the edges of
their 96-pixel row segments, for grids smaller than the largest dilation and larger.

Tolerances: BF16 weights and activations (2^-9) through four layers, 2e-2 of the
largest output and 3e-2 of the gradient's norm, as for the 9 x 37 grid.
"""
import numpy as np
import pytest

from oracle import cno_ref as R
from test_cno import _params

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,B", [(3, 3, 1), (5, 95, 2), (4, 96, 1), (7, 97, 1), (29, 193, 1)])
def test_forward_and_gradient_at_segment_edges(H, W, B):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_08803_gb300 import build
    build.build()
    from paper_1709_08803_gb300 import surrogate as S
    rng = np.random.default_rng(W)
    p = _params(3).astype(np.float32)
    x = rng.standard_normal((B, H, W, 4)).astype(np.float32)
    t = rng.standard_normal((B, H, W, 3)).astype(np.float32)
    net = S.CNO(H, W, B)
    net.set_params(p)
    X, T = torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda")
    y = net.forward(X).cpu().numpy()
    yr, _, _ = R.forward(p.astype(np.float64), x.astype(np.float64))
    assert np.abs(y - yr).max() <= 2e-2 * np.abs(yr).max()
    g, loss = net.gradient(X, T)
    lr, gr = R.loss_grad(p.astype(np.float64), x.astype(np.float64), t.astype(np.float64))
    assert abs(loss - lr) <= 1e-3 * lr
    assert np.linalg.norm(g - gr) <= 3e-2 * np.linalg.norm(gr)
    net.close()
