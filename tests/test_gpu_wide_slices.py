"""FP64 preconditioner sweeps on slices of about 4096 rows, which the 32 warps of a thread
block cover in one pass, against the banded operator of the oracle (the bar of
test_gpu_factor.py, 1e-9 |r| |P|)."""
import numpy as np
import pytest

import oracle as O
from paper_1709_08803_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# 4095 | 4098 | 4203 rows
@pytest.mark.parametrize("N,M,h", [(1364, 3, 0), (1365, 3, 1), (1400, 3, 0)])
def test_fp64_sweeps_wide(N, M, h):
    from paper_1709_08803_gb300 import bfs, build
    build.build()
    mesh = W.mesh_box(N, M, 0.3, 0.35)
    ctx = bfs.Context(mesh, W.flat_topography(mesh), 0.7)
    ctx.precond_factor(h)
    r = np.random.default_rng(N).standard_normal(mesh.n_unknowns)
    z = ctx.precond_apply(torch.tensor(r, device="cuda")).cpu().numpy()
    assert ctx.check_finite()
    ctx.close()
    B = O.jtilde_band(O.problem(mesh, 0.7), h)
    R, Z = (v.reshape(3, M, N + 1).transpose(1, 0, 2).reshape(M, -1) for v in (r, z))
    for l in range(M):
        Pz = sum(B[l, m - l + h] @ Z[m] for m in range(max(0, l - h), min(M, l + h + 1)))
        assert np.abs(Pz - R[l]).max() <= 1e-9 * np.abs(B).max() * np.abs(r).max()
