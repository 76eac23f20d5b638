"""Calls that find too little device memory: BFS_ENOMEM, and a context that works as
before once there is enough.  In processes of their own, where nothing else gives
memory back meanwhile."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

COMMON = """
import torch
from paper_1709_08803_gb300 import bfs, workloads as W

MB = 1 << 20


def leave(nbytes):  # takes the device memory but for about nbytes
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    return torch.empty(torch.cuda.mem_get_info()[0] - nbytes, dtype=torch.uint8, device="cuda")


def context(**kw):
    mesh = W.mesh_box(302, 104, 0.3, 0.3)
    return bfs.Context(mesh, W.gaussian_bumps(mesh, [(0.1, 0.7, 0.0, 0.0)]), 0.7, bfs.default_options(**kw))


def no_memory(call, *args):
    try:
        call(*args)
    except bfs.BfsError as e:
        assert e.code == bfs.BFS_ENOMEM, e
        return
    raise AssertionError("it found memory")


"""

# 121 Krylov vectors (88 MB), then their 120 images (87 MB), then eight work vectors (6 MB):
# none fits | the first | the first two
SOLVER = COMMON + """
for size in (None, 40, 130, 178):  # None loads the kernels
    ctx = context(gmres_restart=120, tol=1e3)  # met by the starting iterate
    ctx.precond_factor(0)
    u = ctx.flat_guess()
    if size:
        hog = leave(size * MB)
        for _ in range(2):  # the second call finds nothing half allocated
            no_memory(ctx.solve, u)
            assert ctx.solve(u, raise_on_error=False)["status"] == bfs.BFS_ENOMEM
        del hog
        torch.cuda.empty_cache()
    assert ctx.solve(u)["status"] == bfs.BFS_OK
    ctx.close()
"""

# the factors (877 MB, 607 rows a slice and half band 1), then scratch (34 MB), then the
# slices of the products (169 MB), without which other kernels take the products
FACTOR = COMMON + """
ctx = context()
ctx.precond_factor(1)
r = torch.randn(ctx.n, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
ref = ctx.precond_apply(r)
ctx.close()
for size, fits in ((500, False), (890, False), (960, True)):
    ctx = context()
    hog = leave(size * MB)
    for _ in range(1 if fits else 2):
        ctx.precond_factor(1) if fits else no_memory(ctx.precond_factor, 1)
    del hog
    torch.cuda.empty_cache()
    if not fits:
        ctx.precond_factor(1)
    # two factorisations to FP64 accuracy
    assert (ctx.precond_apply(r) - ref).norm() <= 1e-9 * ref.norm()
    ctx.close()
"""


@pytest.mark.parametrize("script", [SOLVER, FACTOR], ids=["solver", "factor"])
def test_too_little_memory(script):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_08803_gb300 import build
    build.build()
    torch.cuda.empty_cache()
    p = subprocess.run([sys.executable, "-c", script], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert p.returncode == 0, p.stderr[-2000:]
