"""kbc_adjoint where the allocator has the parts of its work space but no piece
as large as all of them."""
import numpy as np
import pytest

from paper_1507_02509_gb300 import flows

pytestmark = pytest.mark.gpu

NX, NY = 64, 48


def gradients(lat, steps, every, objective):
    from paper_1507_02509_gb300 import capi

    rho, ux, uy = flows.turbulence(64, k0=3, urms=0.04, seed=5, kcut=16)
    rho, u = np.ascontiguousarray(rho[:NY]), np.ascontiguousarray(np.stack((ux, uy))[:, :NY])
    target = np.ascontiguousarray(0.5 * u[::-1]) if objective else None
    g = np.empty((2, NY, NX))
    J, gb = capi.kbc_adjoint(lat.h, rho, u, steps, every, objective, target, g)
    return J, gb, g


@pytest.mark.parametrize("dtype,steps,every,objective", [("f32", 4, 2, 1), ("f32", 1, 3, 0), ("f64", 6, 2, 0)])
@pytest.mark.parametrize("last", [False, True])
def test_parts_in_place_of_one_piece(dtype, steps, every, objective, last):
    """last: the copy of a checkpoint, which only saves launches, is refused too."""
    import torch

    import paper_1507_02509_gb300 as pkg
    from paper_1507_02509_gb300 import KBCError, Lattice, capi

    kw = dict(variant="B", beta=0.97, dtype=dtype)
    field = NX * NY * (72 if dtype == "f64" else 36)
    plain = Lattice(NX, NY, **kw)
    want = gradients(plain, steps, every, objective)
    plain.close()
    live, refuse = {}, {"above": 1 << 40, "fields": 1 << 40, "refused": 0}

    def alloc(nbytes, stream, user):
        fields = sum(1 for b in live.values() if b == field)
        if nbytes > refuse["above"] or (nbytes == field and fields >= refuse["fields"]):
            refuse["refused"] += 1
            if nbytes == field:
                refuse["fields"] = 1 << 40  # that one
            return None
        p = torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(), int(stream or 0))
        live[p] = nbytes
        return p

    def release(p, stream, user):
        del live[p]
        torch.cuda.caching_allocator_delete(int(p))

    hooks = (capi.ALLOC_FN(alloc), capi.FREE_FN(release))
    capi.kbc_set_allocator(hooks[0], hooks[1], None)
    try:
        lat = Lattice(NX, NY, torch_allocator=False, **kw)
        # a slab of three checkpoints at most; all parts together are larger
        refuse["above"] = 3 * field
        if last and steps // every >= 2:
            refuse["fields"] = 6  # the handle's two, the call's two and two lambdas are there
        got = gradients(lat, steps, every, objective)
        assert refuse["refused"] >= 1
        assert got[0] == want[0] and got[1] == want[1] and np.array_equal(got[2], want[2])
        refuse["above"] = field - 1
        with pytest.raises(KBCError) as e:
            gradients(lat, steps, every, objective)
        assert e.value.status == capi.KBC_ERR_NOMEM
        refuse["above"] = 1 << 40
        assert gradients(lat, steps, every, objective)[0] == want[0]
        lat.close()
        assert not live
    finally:
        pkg.use_torch_allocator()
        capi.kbc_set_allocator(*pkg._torch_hooks, None)
