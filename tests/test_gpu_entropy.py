"""Entropy density and the statistics' reductions where their arithmetic
changes: deviations at the edges of the series' table, tiny grids and
partial tiles."""
import math

import numpy as np
import pytest

import oracle as O
from gpu_helpers import representable

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f64", "f32", "f16"])
@pytest.mark.parametrize("top", [1e-12, 1.0 / 256, 0.1, 0.496, 0.504, 0.9, 3.0])
@pytest.mark.parametrize("shape", [(1, 1), (64, 8), (65, 9), (200, 31)])
def test_entropy_of_deviations_up_to(top, dtype, shape):
    """Relative deviations x_i = d_i / W_i spread over [-min(top, 0.95), top]:
    S and its spread against long double sums of the stored values.  x = +-1/2
    divides the table from the library's logarithm."""
    from paper_1507_02509_gb300 import Lattice

    nx, ny = shape
    rng = np.random.default_rng(7)
    w = O.weights().reshape(9, 1, 1)
    x = rng.uniform(-min(top, 0.95), top, (9, ny, nx))
    x[:, :, 0] = 0.0
    g = representable(w * (1.0 + x), dtype)
    lat = Lattice(nx, ny, variant="B", beta=0.97, dtype=dtype)
    lat.set_populations(g)
    got = lat.diagnostics_ext()
    lat.close()
    f, wl = g.astype(np.longdouble), w.astype(np.longdouble)
    s = -(f * np.log(f / wl)).sum(0)
    # a logarithm's and a sum's rounding per term: some ulp of the terms; the
    # weights' own rounding in f / W (1 ulp) counts as the terms do
    scale = float(np.abs(f).sum(0).max()) * max(1.0, math.log(4.0))
    assert abs(got["S"] - float(s.mean())) <= 30 * 2.0 ** -52 * scale
    assert abs(got["S_std"] - float(s.std())) <= 1e-11 * scale


@pytest.mark.parametrize("shape", [(1, 1), (3, 1), (64, 8), (129, 17), (640, 400)])
def test_statistics_of_few_and_many_nodes(shape):
    """Means and spreads do not depend on how many nodes a thread, a block or
    the last fold has (some none)."""
    from paper_1507_02509_gb300 import Lattice

    nx, ny = shape
    rng = np.random.default_rng(9)
    rho = 1.0 + 0.01 * rng.standard_normal((ny, nx))
    ux, uy = 0.03 + 0.02 * rng.standard_normal((2, ny, nx))
    g = O.init_feq(rho, ux, uy)
    lat = Lattice(nx, ny, variant="lbgk", beta=0.97, dtype="f64")
    lat.set_populations(g)
    d = lat.diagnostics()
    lat.close()
    r, vx, vy = O.macro(g)
    ke = 0.5 * (vx * vx + vy * vy)
    om = 0.5 * (np.roll(vy, -1, 1) - np.roll(vy, 1, 1)) - 0.5 * (np.roll(vx, -1, 0) - np.roll(vx, 1, 0))
    zz = 0.5 * om * om
    for key, want in (("mass", r.sum()), ("E", ke.mean()), ("Z", zz.mean()), ("px", (r * vx).sum())):
        assert d[key] == pytest.approx(want, rel=1e-12, abs=1e-14)
    for key, q in (("E_std", ke), ("Z_std", zz)):
        assert d[key] == pytest.approx(q.std(), rel=1e-10, abs=1e-15)
    assert d["gamma_mean"] == d["gamma_min"] == d["gamma_max"] == 2.0
