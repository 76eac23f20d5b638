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


# vertical distances around 1447 cells, up to which s^2 + t^2 + d^2 is formed from an exact
# square: surfaces up to 4 above the undisturbed one; slopes of 0.9 | 1.5 | 3 over 999 columns
# and of 3 over 30 (the half domain: 60) rows
@pytest.mark.parametrize("mesh,zeta,slope", [
    (*_fine(1024, 0.2), 0.0), (*_fine(1024, 0.22), 0.0), (*_fine(1024, 2.0), 0.0), (*_fine(1024, 3.0, half=1), 0.0),
    (*_fine(512, 3.5), 0.0), (*_fine(512, 4.0, dy=1.25), 0.0),
    (W.Mesh(N=1000, M=3, x1=-100.0, y1=-0.2, dx=0.2, dy=0.2), 0.0, 0.9),
    (W.Mesh(N=1000, M=3, x1=-100.0, y1=-0.2, dx=0.2, dy=0.2), 0.0, 1.5),
    (W.Mesh(N=1000, M=3, x1=-100.0, y1=-0.2, dx=0.2, dy=0.2), 0.0, 3.0),
    (W.Mesh(N=31, M=31, x1=-3.0, y1=0.0, dx=0.2, dy=0.2, half=1), 0.0, 3.0)])
def test_exact_squares(mesh, zeta, slope):
    _check(mesh, zeta, slope=slope)


@pytest.mark.parametrize("N,M,half", [(9, 5, 0), (9, 5, 1), (34, 18, 0)])
def test_depth_terms_alone(N, M, half):
    """A flat surface 2304 cells above a flat bottom, phi - x = 1 and psi = x (exact on this
    mesh): a kinematic row at the bottom is the sum of w K1 over the surface and nothing
    else, so it shows the accuracy of a single pair (1e-10 of the row, no absolute part)."""
    from paper_1709_08803_gb300 import bfs, build
    build.build()
    dx = 1.0 / 512
    mesh = W.Mesh(N=N, M=M, x1=-4 * dx, y1=0.0 if half else -2 * dx, dx=dx, dy=dx, half=half)
    topo = W.flat_topography(mesh)
    v = np.zeros((3, M, N + 1))
    v[0, :, 0], v[1, :, 0], v[2, :, 0] = 3.5, mesh.x1 + 1.0, mesh.x1
    v[1:, :, 1:] = 1.0
    ref, scale = O.residual(O.problem(mesh, 3.0), topo, v.ravel(), with_scale=True)
    ctx = bfs.Context(mesh, topo, 3.0)
    got = ctx.residual(torch.tensor(v.ravel(), device="cuda"), precision=bfs.BFS_DF64).cpu().numpy()
    assert (np.abs(got - ref) <= 1e-10 * scale).all()
    ctx.close()
