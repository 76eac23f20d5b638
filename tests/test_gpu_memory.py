"""Calls that find too little device memory: BFS_ENOMEM, and a context that works as
before once there is enough."""
import pytest

from paper_1709_08803_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_08803_gb300 import build
    build.build()


def _leave(nbytes):
    """Takes the device memory but for about nbytes."""
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    return torch.empty(torch.cuda.mem_get_info()[0] - nbytes, dtype=torch.uint8, device="cuda")


def _context(**kw):
    from paper_1709_08803_gb300 import bfs
    mesh = W.mesh_box(302, 104, 0.3, 0.3)
    return bfs.Context(mesh, W.gaussian_bumps(mesh, [(0.1, 0.7, 0.0, 0.0)]), 0.7, bfs.default_options(**kw))


# 121 Krylov vectors (92 MB), then their 120 images (91 MB), then eight work vectors (6 MB):
# none fits | the first | the first two
@pytest.mark.parametrize("leave", [40, 130, 186])
def test_solver_buffers(leave):
    from paper_1709_08803_gb300 import bfs
    for k in range(2):  # the first context loads the kernels
        ctx = _context(gmres_restart=120, tol=1e3)  # met by the starting iterate
        ctx.precond_factor(0)
        u = ctx.flat_guess()
        if k:
            hog = _leave(leave * MB)
            for _ in range(2):  # the second call finds nothing half allocated
                with pytest.raises(bfs.BfsError) as e:
                    ctx.solve(u)
                assert e.value.code == bfs.BFS_ENOMEM
            del hog
            torch.cuda.empty_cache()
        assert ctx.solve(u)["status"] == bfs.BFS_OK
        ctx.close()


# the factors (878 MB, 607 rows a slice and half band 1), then scratch (34 MB), then the
# slices of the products (169 MB), without which other kernels take the products
@pytest.mark.parametrize("leave,fits", [(500, 0), (890, 0), (960, 1)])
def test_factor_buffers(leave, fits):
    from paper_1709_08803_gb300 import bfs
    ctx = _context()
    ctx.precond_factor(1)
    r = torch.randn(ctx.n, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    ref = ctx.precond_apply(r)
    ctx.close()
    ctx = _context()
    hog = _leave(leave * MB)
    if fits:
        ctx.precond_factor(1)
    else:
        for _ in range(2):
            with pytest.raises(bfs.BfsError) as e:
                ctx.precond_factor(1)
            assert e.value.code == bfs.BFS_ENOMEM
    del hog
    torch.cuda.empty_cache()
    if not fits:
        ctx.precond_factor(1)
    # two factorisations to FP64 accuracy
    assert (ctx.precond_apply(r) - ref).norm() <= 1e-9 * ref.norm()
    ctx.close()
