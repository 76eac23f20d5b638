"""Condensed slice blocks of the preconditioner (phi_x eliminated) through the
public apply, against the banded operator of the oracle."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle as O
from paper_1709_08803_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_08803_gb300 import build
    build.build()


FRESH = """
import sys
import numpy as np
import torch
import oracle as O
from paper_1709_08803_gb300 import bfs, workloads as W

N, M, h, prec = (int(a) for a in sys.argv[1:])
mesh = W.mesh_box(N, M, 0.3, 0.35)
ctx = bfs.Context(mesh, W.flat_topography(mesh), 0.7, bfs.default_options(precond_precision=prec))
ctx.precond_factor(h)
r = np.random.default_rng(N).standard_normal(mesh.n_unknowns)
z = ctx.precond_apply(torch.tensor(r, dtype=torch.float64, device="cuda")).cpu().numpy()
assert ctx.check_finite()
B = O.jtilde_band(O.problem(mesh, 0.7), h)
by_slice = lambda v: v.reshape(3, M, N + 1).transpose(1, 0, 2).reshape(M, -1)
R, Z = by_slice(r), by_slice(z)
err = max(np.abs(sum(B[l, m - l + h] @ Z[m] for m in range(max(0, l - h), min(M, l + h + 1))) - R[l]).max() for l in range(M))
bar = 1e-9 * np.abs(B).max() if prec == bfs.BFS_FP64 else 0.05
assert err <= bar * np.abs(r).max(), (err, bar)
"""


# Dynamic shared memory within 48 KB that the kernels' static arrays take past it: 47 400
# bytes of k_cond_conv (2 KB static), 49 152 of k_cond_form (32 bytes).  In a process of its
# own: the limit that a launch asks for stays raised for the ones after it.
# Tolerances as in test_gpu_factor.py.
@pytest.mark.parametrize("N,M,h,prec", [(182, 16, 7, 0), (182, 16, 7, 1), (1534, 3, 0, 0)])
def test_first_launch_near_48_KB(N, M, h, prec):
    r = subprocess.run([sys.executable, "-c", FRESH, *map(str, (N, M, h, prec))], cwd=ROOT, capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]


def _apply(mesh, h, prec, F):
    from paper_1709_08803_gb300 import bfs
    ctx = bfs.Context(mesh, W.flat_topography(mesh), F, bfs.default_options(precond_precision=prec))
    ctx.precond_factor(h)
    r = np.random.default_rng(mesh.N).standard_normal(mesh.n_unknowns)
    z = ctx.precond_apply(torch.tensor(r, dtype=torch.float64, device="cuda")).cpu().numpy()
    assert ctx.check_finite()
    ctx.close()
    return O.jtilde(O.problem(mesh, F), half_band=h), r, z


# Coarse meshes and small Froude numbers, N dx^2 / F^2 from 40 over 74 (condensed) and 75.1 to 2e6:
# the tolerances of test_gpu_factor.py, 1e-9 |r| |P| for FP64 and P z within 5 % of r for FP32.
@pytest.mark.parametrize("N,M,h,dx,F,prec", [
    (110, 7, 2, 3.0, 0.1, 0), (110, 7, 2, 3.0, 0.02, 0), (110, 7, 2, 0.3, 0.02, 0), (150, 5, 1, 0.3, 0.02, 0),
    (101, 7, 2, 1.0, 1.16, 0), (101, 7, 2, 1.0, 1.17, 0), (101, 7, 2, 1.0, 1.6, 0),
    (150, 5, 1, 0.3, 0.1, 1), (150, 5, 1, 0.3, 0.3, 1), (150, 5, 1, 0.3, 0.58, 1)])
def test_small_froude_and_coarse_mesh(N, M, h, dx, F, prec):
    P, r, z = _apply(W.mesh_box(N, M, dx, dx * 7 / 6), h, prec, F)
    assert np.abs(P @ z - r).max() <= (1e-9 * np.abs(P).max() if prec == 0 else 0.05) * np.abs(r).max()
