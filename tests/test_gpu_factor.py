"""Preconditioner factors and sweeps at the sizes where the path changes.

Against the dense banded operator of the oracle: the residual of P z = r.
Tolerances: FP64 factors, 1e-9 |r| |P| (entrywise maxima), as for an FP64 solve
of these ill-conditioned blocks.  FP32 sweeps: the rounding bound
4 sqrt(n) u32 (|P| |z|)_max + u32 |r|_max of sums of n = (2 h + 1) nb entries
(u32 = 2^-24) on small meshes; on wide ones, whose condition leaves an FP32 solve
few digits, P z within 5 % of r, which keeps the spectrum clustered at 1.
"""
import math

import numpy as np
import pytest

import oracle as O
from paper_1709_08803_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_08803_gb300 import build
    build.build()


def _solve(mesh, h, prec):
    from paper_1709_08803_gb300 import bfs
    ctx = bfs.Context(mesh, W.flat_topography(mesh), 0.7, bfs.default_options(precond_precision=prec))
    ctx.precond_factor(h)
    P = O.jtilde(O.problem(mesh, 0.7), half_band=h)
    r = np.random.default_rng(mesh.N).standard_normal(mesh.n_unknowns)
    z = ctx.precond_apply(torch.tensor(r, dtype=torch.float64, device="cuda")).cpu().numpy()
    assert ctx.check_finite()
    return P, r, z


# slice rows 126 | 129: elimination in FP64 | double-float inverse, one correction and
# sliced products; 192 | 195: whole tiles | one row over; 99 | 100 columns: full |
# condensed blocks; 449 rows: sums of products in two segments; a first node at
# x = 0, where phi_x is not eliminated
@pytest.mark.parametrize("N,M,h,x1", [(41, 9, 1, None), (42, 9, 1, None), (63, 9, 2, None), (64, 9, 2, None),
                                      (99, 7, 2, None), (100, 7, 2, None), (100, 9, 4, None), (222, 5, 1, None),
                                      (223, 5, 1, None), (110, 5, 1, 0.0075)])
def test_fp64_factor_edges(N, M, h, x1):
    from paper_1709_08803_gb300 import bfs
    mesh = W.mesh_box(N, M, 0.3, 0.35, x1=x1)
    P, r, z = _solve(mesh, h, bfs.BFS_FP64)
    assert np.abs(P @ z - r).max() <= 1e-9 * np.abs(r).max() * np.abs(P).max()


# half bands 4 to 6 in the two-chain sweeps, odd sizes, a half domain
@pytest.mark.parametrize("N,M,h,half", [(41, 9, 1, 0), (42, 9, 1, 0), (47, 13, 4, 0), (51, 15, 5, 1), (45, 16, 6, 0)])
def test_fp32_sweeps_small(N, M, h, half):
    from paper_1709_08803_gb300 import bfs
    mesh = W.mesh_box(N, M, 0.3, 0.35, half=half)
    P, r, z = _solve(mesh, h, bfs.BFS_FP32C)
    u32, n = 2.0 ** -24, (2 * h + 1) * 3 * (N + 1)
    bound = 4.0 * math.sqrt(n) * u32 * (np.abs(P) @ np.abs(z)).max() + u32 * np.abs(r).max()
    assert np.abs(P @ z - r).max() <= bound


# 139 | 140 and 256 | 257 columns: full | condensed | full blocks; 515 rows: two segments
@pytest.mark.parametrize("N,M,h,half", [(139, 9, 2, 0), (140, 9, 2, 0), (141, 7, 1, 1), (256, 5, 1, 0), (257, 5, 1, 0)])
def test_fp32_sweeps_wide(N, M, h, half):
    from paper_1709_08803_gb300 import bfs
    mesh = W.mesh_box(N, M, 0.4, 0.4, half=half)
    P, r, z = _solve(mesh, h, bfs.BFS_FP32C)
    assert np.abs(P @ z - r).max() <= 0.05 * np.abs(r).max()
