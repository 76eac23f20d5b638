"""FP64 and double-float pair kernels at the edges of their tiles and branches,
against the FP64 oracle: targets around one tile of 128, sources around the
units of 8 that the splits are cut in, and both forms of s^2 + t^2 in the
double-float kernel -- one exact float (dx == dy, at most 1024 columns, 512 rows
and 1/dx <= 1024) and the general pair.

Bar: 1e-10 of the row's sum of absolute terms plus 1e-13, the parity bar of the
FP64-accurate residuals (a term of the double-float sums carries about 46 bits,
1e-14, so rounding alone stays far below it)."""
import numpy as np
import pytest

import oracle as O
from paper_1709_08803_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MESHES = {
    "tile_minus_2": W.Mesh(N=4, M=42, x1=-0.4, y1=-4.1, dx=0.2, dy=0.2),            # 126 targets, 168 sources
    "tile": W.Mesh(N=5, M=32, x1=-0.4, y1=-3.1, dx=0.2, dy=0.2),    # 128 targets, 160 sources
    "tile_plus_1": W.Mesh(N=4, M=43, x1=-0.4, y1=-4.2, dx=0.2, dy=0.2),  # 129 targets, 172 sources
    "sources_mod_8": W.Mesh(N=7, M=3, x1=-0.6, y1=-0.2, dx=0.2, dy=0.2),  # 21 sources
    "half": W.Mesh(N=9, M=5, x1=-0.8, y1=0.0, dx=0.2, dy=0.2, half=1),
    "dy_not_dx": W.Mesh(N=13, M=7, x1=-1.2, y1=-0.9, dx=0.2, dy=0.3),
    "wide_general": W.Mesh(N=1030, M=3, x1=-100.0, y1=-0.2, dx=0.2, dy=0.2),
    "fine_general": W.Mesh(N=9, M=5, x1=-4 / 2048, y1=-2 / 2048, dx=1 / 2048, dy=1 / 2048),
    "fine_exact": W.Mesh(N=9, M=5, x1=-4 / 1024, y1=-2 / 1024, dx=1 / 1024, dy=1 / 1024),
}


@pytest.mark.parametrize("precision", ["fp64", "df64"])
@pytest.mark.parametrize("name", sorted(MESHES))
def test_residual_at_tile_edges(name, precision):
    from paper_1709_08803_gb300 import bfs, build
    build.build()
    mesh = MESHES[name]
    topo = W.gaussian_bumps(mesh, [(0.05, 0.5, 0.0, 0.0)])
    u = W.smooth_guess(mesh, 4)
    ref, scale = O.residual(O.problem(mesh, 0.8), topo, u, with_scale=True)
    ctx = bfs.Context(mesh, topo, 0.8)
    got = ctx.residual(torch.tensor(u, device="cuda"),
                       precision={"fp64": bfs.BFS_FP64, "df64": bfs.BFS_DF64}[precision]).cpu().numpy()
    assert (np.abs(got - ref) <= 1e-10 * scale + 1e-13).all()
