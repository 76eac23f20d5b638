"""What a solve with Eisenstat-Walker terms does near its tolerance: GMRES of the last
step goes on to a tenth of it, and an iterate which meets it by less than a factor of
five gets one more step."""
import numpy as np
import pytest

from paper_1709_08803_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_08803_gb300 import build
    build.build()


def _options(**kw):
    from paper_1709_08803_gb300 import bfs
    return bfs.default_options(krylov_precision=bfs.BFS_FP32C, outer_precision=bfs.BFS_DF64, eta=1e-2, refine_below=1e-5,
                               precond_precision=bfs.BFS_FP32C, forcing=1, **kw)


def _solve(problem, **kw):
    """A solve with its steps launched one by one."""
    from paper_1709_08803_gb300 import bfs
    ctx = bfs.Context(*problem, _options(wait_polls=4000, **kw))
    ctx.precond_factor()
    ctx.profile_enable()
    u = ctx.flat_guess()
    return ctx, u, ctx.solve(u, raise_on_error=False)


def _tolerance_with_extra_step(problem):
    """A tolerance at which the last step is the extra one, and the solve without it
    (the step limit one lower: an iterate at the limit is returned as it is)."""
    for tol in np.geomspace(1e-6, 1e-11, 101):
        _, _, st = _solve(problem, tol=tol)
        if st["status"] == 0 and st["newton_its"] > 1:
            ctx, u, before = _solve(problem, tol=tol, max_newton=st["newton_its"] - 1)
            if before["status"] == 0:
                assert 0.2 * tol < before["fnorm_inf"] <= tol
                return tol, u, before, st
    pytest.fail("no tolerance with an extra step")


def test_timeout_in_the_extra_step():
    """A sweep of the extra step times out: the iterate before it is returned with
    BFS_OK, and the next apply runs."""
    from paper_1709_08803_gb300 import bfs
    problem = W.config_small_half()
    tol, u0, before, st = _tolerance_with_extra_step(problem)
    ctx = bfs.Context(*problem, _options(wait_polls=4000, tol=tol))
    ctx.precond_factor()
    r = torch.tensor(np.random.default_rng(3).standard_normal(ctx.n), device="cuda")
    ref = ctx.precond_apply(r)
    assert ctx.check_finite()
    tbl, ntask = bfs.sweep_schedule(problem[0].M, ctx.precond_info()["half_band"], ctx.precond_info()["twist"] >= 0)
    ctx.profile_enable()
    ctx.debug_stall_sweep(int(np.flatnonzero(tbl[:, 2] > 0)[-1]), skip=before["precond_applies"])
    u = ctx.flat_guess()
    got = ctx.solve(u, raise_on_error=False)
    assert got["status"] == bfs.BFS_OK
    assert got["precond_applies"] > before["precond_applies"]  # the step was taken
    assert got["newton_its"] == before["newton_its"] and got["fnorm_inf"] == before["fnorm_inf"]
    assert torch.equal(u, u0)
    z = torch.full_like(r, float("nan"))
    ctx.precond_apply(r, out=z)
    assert torch.equal(z, ref)
    assert ctx.check_finite()
    ctx.close()


@pytest.mark.parametrize("batch", [0, 1])
def test_stall_is_against_the_forcing_term(batch):
    """A forcing term of 0.9 that three Krylov iterations reach in every step is no
    stall, although the last steps ask for more than three iterations give."""
    from paper_1709_08803_gb300 import bfs
    mesh, topo, F = W.config_small_half()
    o = bfs.default_options(tol=1e-8, krylov_precision=bfs.BFS_FP32C, outer_precision=bfs.BFS_DF64, eta=0.9,
                            refine_below=1e-5, forcing=1, max_krylov=3, stall_newton=1, max_newton=200)
    if batch:
        b = bfs.Batch([mesh], [topo], [F], o)
        rc, st = b.solve(b.flat_guesses())
        assert rc == bfs.BFS_OK and st[0]["fnorm_inf"] <= 1e-8, st
        b.close()
    else:
        ctx = bfs.Context(mesh, topo, F, o)
        st = ctx.solve(ctx.flat_guess(), raise_on_error=False)
        assert st["status"] == bfs.BFS_OK and st["fnorm_inf"] <= 1e-8, st
        ctx.close()


def _final(problem, batch, stop, **kw):
    """Status and statistics of a solve, alone or as a batch of one."""
    from paper_1709_08803_gb300 import bfs
    mesh, topo, F = problem
    if batch:
        b = bfs.Batch([mesh], [topo], [F], _options(**kw))
        b.set_stop_at_tol(stop)
        _, st = b.solve(b.flat_guesses())
        b.close()
        return st[0]
    ctx = bfs.Context(mesh, topo, F, _options(**kw))
    ctx.set_stop_at_tol(stop)
    st = ctx.solve(ctx.flat_guess(), raise_on_error=False)
    ctx.close()
    return st


@pytest.mark.parametrize("batch", [0, 1])
def test_stop_at_tol(batch):
    """With it a solve never passes over an iterate that meets the tolerance, alone and in
    a batch; without it, the solve alone takes the extra step for some of these tolerances."""
    from paper_1709_08803_gb300 import bfs
    problem = W.config_small_half()
    passed = 0
    for tol in np.geomspace(1e-7, 1e-11, 21):
        for stop in (True, False):
            st = _final(problem, batch, stop, tol=tol)
            assert st["status"] == bfs.BFS_OK and st["fnorm_inf"] <= tol
            short = _final(problem, batch, stop, tol=tol, max_newton=st["newton_its"] - 1)
            assert short["status"] in (bfs.BFS_OK, bfs.BFS_ENOCONV)
            if stop:
                assert short["status"] == bfs.BFS_ENOCONV
            else:
                passed += short["status"] == bfs.BFS_OK
    assert passed > 0 if not batch else passed == 0
