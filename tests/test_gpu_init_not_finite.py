"""Equilibrium initialisation from values that are not finite: NaN and infinities
where the equilibrium's polynomial has them."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f64", "f32", "f16"])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("where", ["rho", "ux", "uy"])
def test_not_finite_where_the_polynomial_is_not(where, value, dtype):
    from paper_1507_02509_gb300 import Lattice

    nx, ny = 37, 8
    rng = np.random.default_rng(1)
    fields = {"rho": 1.0 + 0.01 * rng.standard_normal((ny, nx)), "ux": 0.03 * rng.standard_normal((ny, nx)),
              "uy": 0.03 * rng.standard_normal((ny, nx))}
    fields[where][3, 5::4] = value
    fields["ux"][6, ::3] = fields["uy"][6, ::3] = 0.0
    lat = Lattice(nx, ny, variant="B", beta=0.97, dtype=dtype)
    lat.init(fields["rho"], fields["ux"], fields["uy"])
    got = lat.populations().cpu().numpy()
    lat.close()
    rho, ux, uy = fields["rho"], fields["ux"], fields["uy"]
    w = O.weights().reshape(9, 1, 1)
    a = np.array([i % 3 - 1 for i in range(9)]).reshape(9, 1, 1)
    b = np.array([i // 3 - 1 for i in range(9)]).reshape(9, 1, 1)
    with np.errstate(all="ignore"):
        xi = a * ux + b * uy
        dev = w * ((rho - 1.0) + rho * (xi * (3.0 + 4.5 * xi) - 1.5 * (ux * ux + uy * uy)))
        if dtype == "f32":
            dev = dev.astype(np.float32).astype(np.float64)
        elif dtype == "f16":
            dev = (dev / w).astype(np.float16).astype(np.float64) * w
        want = dev + w
    assert np.array_equal(np.isnan(got), np.isnan(want))
    assert np.array_equal(np.isinf(got), np.isinf(want)) and np.array_equal(got[np.isinf(got)], want[np.isinf(want)])
    fine = np.isfinite(want)
    tol = {"f64": 1e-15, "f32": 1e-7, "f16": 1e-3}[dtype]
    assert np.all(np.abs(got[fine] - want[fine]) <= tol * np.maximum(1.0, np.abs(want[fine])))
