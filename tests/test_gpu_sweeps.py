"""FP32 preconditioner sweeps (the task-table kernel): tasks that may overlap,
and slices narrower than the GPU.

Against the dense banded operator of the oracle, with the rounding bound
4 sqrt(n) u32 (|P| |z|)_max + u32 |r|_max of sums of n = (2 h + 1) nb entries
(u32 = 2^-24, Higham and Mary, SIAM J. Sci. Comput. 41, 2019).
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


def _check(N, M, h, half=0, repeats=0):
    from paper_1709_08803_gb300 import bfs
    mesh = W.mesh_box(N, M, 0.3, 0.35, half=half)
    ctx = bfs.Context(mesh, W.flat_topography(mesh), 0.7, bfs.default_options(precond_precision=bfs.BFS_FP32C))
    ctx.precond_factor(h)
    P = O.jtilde(O.problem(mesh, 0.7), half_band=h)
    r = np.random.default_rng(N).standard_normal(mesh.n_unknowns)
    rd = torch.tensor(r, dtype=torch.float64, device="cuda")
    first = ctx.precond_apply(rd)
    differ = torch.zeros((), dtype=torch.int64, device="cuda")
    for _ in range(repeats):
        differ += (ctx.precond_apply(rd) != first).any()
    assert ctx.check_finite()  # raises BfsError(BFS_ETIMEOUT) if a wait gave up
    assert int(differ) == 0
    z = first.cpu().numpy()
    u32, n = 2.0 ** -24, (2 * h + 1) * 3 * (N + 1)
    bound = 4.0 * math.sqrt(n) * u32 * (np.abs(P) @ np.abs(z)).max() + u32 * np.abs(r).max()
    assert np.abs(P @ z - r).max() <= bound
    ctx.close()


# Tasks without a critical block, in which the rows of a CTA may be a task apart: all
# forward ones at half band 0 (one or two, two rows a CTA), some middle ones from half
# band 3 up (three rows a CTA).  Every launch stores every row of every task once, so
# repeated applies give the same bits.
@pytest.mark.parametrize("N,M,h,half", [(50, 9, 0, 0), (63, 9, 0, 0), (63, 13, 3, 0), (47, 13, 4, 0), (51, 15, 5, 1),
                                        (45, 16, 6, 0)])
def test_overlapping_tasks(N, M, h, half):
    _check(N, M, h, half, repeats=2000)


# Slices of fewer rows than a group has CTAs (15 to 141 rows, groups of 76 or 152): as many
# CTAs as rows; 72 | 75 | 78 rows around a group of 76, 150 | 153 around one of 152.
@pytest.mark.parametrize("N,M,h,half", [(4, 3, 0, 0), (4, 3, 1, 0), (10, 7, 0, 0), (10, 7, 2, 1), (23, 7, 1, 0), (24, 7, 1, 0),
                                        (25, 7, 1, 0), (46, 5, 0, 0), (49, 5, 0, 0), (50, 5, 0, 0)])
def test_fewer_rows_than_ctas(N, M, h, half):
    _check(N, M, h, half, repeats=20)
