"""The guard pass of float storage keeps every SM busy: a list of some ten
thousand nodes, lying together, that the attempt in single precision does not
settle costs little more than their double collision alone."""
import numpy as np
import pytest

from gpu_helpers import representable

pytestmark = pytest.mark.gpu

SETTLED = float(np.float32(1e-12))
DOUBLE = float(np.nextafter(np.float32(1e-12), np.float32(1)))  # no attempt


@pytest.mark.parametrize("rows", [28, 80, 300])
def test_unsettled_nodes_are_spread_over_the_blocks(rows):
    import torch

    import oracle as O
    from paper_1507_02509_gb300 import Lattice

    n = 1024
    rng = np.random.default_rng(2)
    ux, uy = 0.03 * rng.standard_normal((2, n, n))
    ux[:rows] = uy[:rows] = 0.0  # at rest: <dh|dh> = 0
    g = torch.as_tensor(representable(O.init_feq(np.ones((n, n)), ux, uy), "f32")).cuda()
    lats = {}
    for guard in (SETTLED, DOUBLE):
        lats[guard] = Lattice(n, n, variant="B", beta=0.985, dtype="f32")
        lats[guard].set_guard(guard)
    t = {guard: [] for guard in lats}
    for _ in range(80):  # in turn
        for guard, lat in lats.items():
            lat.set_populations(g)
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            lat.step(1)
            b.record()
            torch.cuda.synchronize()
            t[guard].append(a.elapsed_time(b))
    took = {guard: float(np.median(x[10:])) for guard, x in t.items()}
    count = {guard: lat.guard_count() for guard, lat in lats.items()}
    out = {guard: lat.populations() for guard, lat in lats.items()}
    for lat in lats.values():
        lat.close()
    assert count[SETTLED] == count[DOUBLE] >= (rows - 2) * n
    assert torch.equal(out[SETTLED], out[DOUBLE])
    # 28 rows: 26 us and 39 when blocks of 512 entries left two thirds of the SMs idle
    assert took[SETTLED] < 1.3 * took[DOUBLE], took
