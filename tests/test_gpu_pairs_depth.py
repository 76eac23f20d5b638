"""Double-float residuals whose depths are many mesh cells, against the FP64 oracle: a
depth difference of two nodes is then a small difference of large numbers.

Bar of test_gpu_pairs.py: 1e-10 of the row's sum of absolute terms plus 1e-13."""
import numpy as np
import pytest

import oracle as O
from paper_1709_08803_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(mesh, zeta, F=3.0, slope=0.0):
    from paper_1709_08803_gb300 import bfs, build
    build.build()
    topo = W.gaussian_bumps(mesh, [(0.05, 0.5, 0.0, 0.0)])
    v = W.smooth_guess(mesh, 4).reshape(3, mesh.M, mesh.N + 1)
    v[0, :, 0] += zeta
    v[0, :, 1:] += slope * np.cos(0.7 * np.arange(mesh.N))
    u = v.ravel()
    ref, scale = O.residual(O.problem(mesh, F), topo, u, with_scale=True)
    ctx = bfs.Context(mesh, topo, F)
    got = ctx.residual(torch.tensor(u, device="cuda"), precision=bfs.BFS_DF64).cpu().numpy()
    assert (np.abs(got - ref) <= 1e-10 * scale + 1e-13).all()
    ctx.close()


def _fine(cells, zeta, half=0, dy=1.0):
    dx = 1.0 / cells
    return W.Mesh(N=9, M=5, x1=-4 * dx, y1=0.0 if half else -2 * dx * dy, dx=dx, dy=dx * dy, half=half), zeta


# a surface 512 | 1024 cells above the undisturbed one; dx != dy; about 16 cells, where the
# kernel changes to renormalised differences
@pytest.mark.parametrize("mesh,zeta", [_fine(256, 2.0), _fine(256, 2.0, half=1), _fine(2048, 0.5), _fine(512, 1.0, dy=1.25),
                                       _fine(16, 0.99), _fine(16, 1.01), _fine(16, 1.01, dy=1.25)])
def test_differences_of_deep_nodes(mesh, zeta):
    _check(mesh, zeta)
