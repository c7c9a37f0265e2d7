"""Moments of nodes whose density vanishes, nearly vanishes or is negative: what
the sums of the stored deviations give, in double."""
import numpy as np
import pytest

import oracle as O
from gpu_helpers import representable

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "f16"])
def test_moments_of_thin_nodes(dtype):
    from paper_1507_02509_gb300 import Lattice

    rng = np.random.default_rng(8)
    nx, ny = 96, 21
    w = O.weights().reshape(9, 1, 1)
    rho = np.ones((ny, nx))
    rho[::2] = 10.0 ** rng.uniform(-7, -2, rho[::2].shape)
    rho[1::4] = -0.5
    f = O.init_feq(rho, 0.05 * rng.standard_normal((ny, nx)), 0.05 * rng.standard_normal((ny, nx)))
    f[:, :, 5::7] = 0.0  # nothing there
    f = representable(f, dtype)
    lat = Lattice(nx, ny, variant="B", beta=0.97, dtype=dtype)
    lat.set_populations(f)
    r, ux, uy = (t.cpu().numpy() for t in lat.moments())
    lat.close()
    d = f - w
    order = [0, 8, 2, 6, 1, 7, 3, 5, 4]
    want = 1.0 + d[order].sum(0)
    # nine sums of deviations below 1: 2^-53 each, twice for the stored value's own
    assert np.max(np.abs(r - want)) <= 18 * 2.0 ** -53
    empty = np.broadcast_to(np.arange(nx) % 7 == 5, (ny, nx))
    if dtype == "f16":  # the code of f = 0 is -1 exactly: rho = 0, and u has no value
        assert (r[empty] == 0.0).all() and np.isnan(ux[empty]).all() and np.isnan(uy[empty]).all()
    jx = f[[2, 5, 8]].sum(0) - f[[0, 3, 6]].sum(0)
    live = np.abs(want) > 1e-3
    assert np.max(np.abs(ux - jx / np.where(live, want, 1.0))[live]) < 1e-11
