"""Doubles with a fixed gamma: the entropic weights and products, two fifths of
a step's FP64 instructions, are not formed."""
import numpy as np
import pytest

import oracle as O
from gpu_helpers import random_field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", ["A", "B", "C", "D"])
def test_fixed_gamma_takes_less_than_entropic(variant):
    import torch

    from paper_1507_02509_gb300 import Lattice

    n = 512
    g = random_field(n, n, 3, amp=1e-3)
    lat = Lattice(n, n, variant=variant, beta=0.97, dtype="f64")
    took = []
    for gamma in (None, 1.0 / 0.97):
        lat.set_gamma(gamma)
        lat.set_populations(g)
        lat.step(32)
        t = []
        for _ in range(7):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            lat.step(32)
            b.record()
            torch.cuda.synchronize()
            t.append(a.elapsed_time(b))
        took.append(float(np.median(t)))
    lat.set_populations(g)
    got = lat.step(3).populations().cpu().numpy()
    lat.close()
    ref = O.step(g, {"A": O.A, "B": O.B, "C": O.C, "D": O.D}[variant], 0.97, 3, gamma_mode=1, gamma_fixed=1.0 / 0.97)
    assert np.max(np.abs(got - ref)) < 1e-14
    assert took[1] < 0.8 * took[0], took  # 0.95 with the products
