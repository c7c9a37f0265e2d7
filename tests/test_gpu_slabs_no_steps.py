"""SlabGroup.step with no steps to take."""
import pytest

from gpu_helpers import random_field, representable

pytestmark = pytest.mark.gpu


def test_no_steps_ask_nothing_of_the_slabs():
    import torch

    from paper_1507_02509_gb300 import KBCError
    from paper_1507_02509_gb300.slabs import SlabGroup

    group = SlabGroup(32, 9, 2, variant="C", beta=0.97, dtype="f32")
    assert group.step(0) is group and group.step(-3) is group  # before initialisation, too
    with pytest.raises(KBCError):
        group.step(1)
    f = representable(random_field(32, 9, 3), "f32")
    group.set_populations(f)
    before = group.populations().clone()
    assert torch.equal(group.step(-1).step(0).step(0.5).populations(), before)
    f[4, 2, 5] = float("nan")
    group.set_populations(f)
    group.step(2)
    with pytest.raises(KBCError):
        group.sync()
    group.step(0).step(-1)  # a field that blew up is reported when it is advanced
    with pytest.raises(KBCError):
        group.step(1)
    group.close()
