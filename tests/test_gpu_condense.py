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
    wide = mesh.N >= 100 if prec == 0 else 140 <= mesh.N <= 256
    condensed = wide and mesh.N * mesh.dx ** 2 <= 75 * F ** 2
    assert ctx.precond_info()["rows"] == (2 * mesh.N + 3 if condensed else 3 * mesh.N + 3)
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


# half domains (the images' terms), FP64: N dx^2 / F^2 = 18 to 21, so condensed
@pytest.mark.parametrize("N,M,h", [(101, 7, 2), (102, 9, 3), (115, 6, 1)])
def test_half_domain_fp64(N, M, h):
    P, r, z = _apply(W.mesh_box(N, M, 0.3, 0.35, half=1), h, 0, 0.7)
    assert np.abs(P @ z - r).max() <= 1e-9 * np.abs(r).max() * np.abs(P).max()


# The FP32 sweeps against the FP64 ones: the relative errors stated with the kernels
# (8.9e-8 at 151 x 53, 1.2e-7 at 181 x 61) times 5/3, which plain FP32 sums of the
# eliminated unknowns exceed (2.8e-7 at 181 x 61).
@pytest.mark.parametrize("N,M,bar", [(151, 53, 1.5e-7), (181, 61, 2.0e-7)])
def test_fp32_sweeps_against_fp64(N, M, bar):
    from paper_1709_08803_gb300 import bfs
    mesh = W.mesh_box(N, M, 0.3, 0.3)
    r = torch.tensor(np.random.default_rng(N).standard_normal(mesh.n_unknowns), device="cuda")
    z = {}
    for prec in (bfs.BFS_FP64, bfs.BFS_FP32C):
        ctx = bfs.Context(mesh, W.flat_topography(mesh), 0.7, bfs.default_options(precond_precision=prec))
        ctx.precond_factor()
        z[prec] = ctx.precond_apply(r)
        assert ctx.check_finite()
        ctx.close()
    assert (z[bfs.BFS_FP32C] - z[bfs.BFS_FP64]).norm() <= bar * z[bfs.BFS_FP64].norm()


@pytest.mark.parametrize("prec", [0, 1])
def test_in_place_and_another_froude_number(prec):
    """r may equal z, and the factors stay those of the Froude number they were formed for."""
    from paper_1709_08803_gb300 import bfs
    mesh = W.mesh_box(142, 9, 0.3, 0.3)
    ctx = bfs.Context(mesh, W.flat_topography(mesh), 0.7, bfs.default_options(precond_precision=prec))
    ctx.precond_factor(2)
    r = torch.tensor(np.random.default_rng(1).standard_normal(mesh.n_unknowns), device="cuda")
    z = ctx.precond_apply(r)
    ctx.set_froude(0.9)
    assert torch.equal(ctx.precond_apply(r), z)
    x = r.clone()
    ctx.precond_apply(x, out=x)
    assert torch.equal(x, z)
    assert ctx.check_finite()
    ctx.close()


def test_refused_inverse():
    """Diagonal blocks that the double-float inverses are not good enough for are inverted
    again in FP64: more launches, and the same bar."""
    import ctypes
    from paper_1709_08803_gb300 import bfs
    mesh, launches = W.mesh_box(64, 5, 0.3, 0.3), {}
    for F in (0.7, 1e-3):
        ctx = bfs.Context(mesh, W.flat_topography(mesh), F)
        n0, n1 = ctypes.c_ulonglong(), ctypes.c_ulonglong()
        bfs.lib().bfs_profile_read(ctx._ctx, None, ctypes.byref(n0))
        ctx.precond_factor(1)
        bfs.lib().bfs_profile_read(ctx._ctx, None, ctypes.byref(n1))
        launches[F] = n1.value - n0.value
        ctx.close()
    assert launches[1e-3] > launches[0.7]
    P, r, z = _apply(mesh, 1, 0, 1e-3)
    assert np.abs(P @ z - r).max() <= 1e-9 * np.abs(r).max() * np.abs(P).max()
