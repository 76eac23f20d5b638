"""The reciprocal square root of the FP64 pair sum against exact arithmetic and against
the one of CUDA (torch.rsqrt).

Bound: 1.6 2^-53 relative -- the last operation's half unit, 2^-54 from the rounding of a
times the seed, and what the series drops (a seed good to 2^-19 leaves less than 2^-58)."""
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_reciprocal_root():
    from paper_1709_08803_gb300 import bfs, build
    build.build()
    rng = np.random.default_rng(5)
    x = np.concatenate([np.exp(rng.uniform(np.log(0.25), np.log(1e6), 20000)),  # squares of distances in mesh cells
                        np.ldexp(rng.uniform(1.0, 2.0, 2000), rng.integers(-60, 1000, 2000)),
                        *[np.nextafter(4.0 ** k, [0.0, 4.0 ** k, np.inf]) for k in range(-5, 12)], [1e-300, 1e300]])
    xd = torch.tensor(x, device="cuda")
    y = bfs.rsqrt_probe(xd).cpu().numpy()
    assert np.abs(y / torch.rsqrt(xd).cpu().numpy() - 1.0).max() <= 4 * 2.0 ** -53  # CUDA's: one unit
    for a, v in zip(x[::7], y[::7]):  # 1 - a v^2 is twice the relative error
        a, v = Fraction(float(a)), Fraction(float(v))
        assert abs(1 - a * v * v) <= Fraction(16, 10) * 2 / 2 ** 53
    y = bfs.rsqrt_probe(torch.tensor([np.inf, np.nan], device="cuda", dtype=torch.float64)).cpu().numpy()
    assert y[0] == 0.0 and np.isnan(y[1])
