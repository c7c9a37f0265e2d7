"""kbc_slabs_step: all slabs of a grid advanced by one call."""
import pytest

from gpu_helpers import random_field, representable

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,parts", [(64, 9, 1), (33, 20, 3), (128, 37, 17), (7, 40, 40)])
@pytest.mark.parametrize("dtype", ["f64", "f32", "f16"])
def test_group_step_equals_exchange_and_step(nx, ny, parts, dtype):
    """Rows of any alignment, more faces than one launch moves, slabs of one
    row: the bits of the exchange through buffers, and of the periodic grid."""
    import torch

    from paper_1507_02509_gb300 import Lattice
    from paper_1507_02509_gb300.slabs import SlabGroup

    kw = dict(variant="B", beta=0.97, dtype=dtype)
    f = torch.as_tensor(representable(random_field(nx, ny, 8), dtype)).cuda()
    one, group, single = SlabGroup(nx, ny, parts, **kw), SlabGroup(nx, ny, parts, **kw), Lattice(nx, ny, **kw)
    for g in (one, group, single):
        g.set_populations(f)
    for _ in range(5):
        one.exchange()
        for s in one.slabs:
            s.step(1)
    group.step(2).step(0).step(3)
    group.sync()
    assert torch.equal(group.populations(), one.populations())
    assert torch.equal(group.populations(), single.step(5).populations())


def test_group_step_refuses_handles_that_do_not_fit():
    from paper_1507_02509_gb300 import KBCError, Lattice, capi

    def lat(nx=32, ny=4, slab=True, dtype="f32"):
        return Lattice(nx, ny, slab=slab, dtype=dtype)

    ready, other, plain, wider, wide64 = lat(), lat(), lat(slab=False), lat(nx=40), lat(dtype="f64")
    f = representable(random_field(32, 4, 1), "f32")
    ready.set_populations(f)
    for bad in ([], [ready.h, ready.h], [plain.h], [ready.h, wider.h], [ready.h, wide64.h]):
        with pytest.raises(KBCError) as e:
            capi.kbc_slabs_step(bad, 1)
        assert e.value.status == capi.KBC_ERR_ARG
    with pytest.raises(KBCError) as e:
        capi.kbc_slabs_step([ready.h, other.h], 1)  # not initialised
    assert e.value.status == capi.KBC_ERR_STATE
    other.set_populations(f)
    with pytest.raises(KBCError) as e:
        capi.kbc_slabs_step([ready.h, other.h], -1)
    assert e.value.status == capi.KBC_ERR_ARG
    capi.kbc_slabs_step([ready.h, other.h], 2)
    ready.sync()
