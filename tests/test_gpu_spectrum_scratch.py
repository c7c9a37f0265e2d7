"""kbc_spectrum where the allocator has room for one component's half spectrum
only, and where it has none."""
import numpy as np
import pytest

from oracle import spectra as ospec

pytestmark = pytest.mark.gpu


class Limited:
    """Allocator hooks over PyTorch's that refuse single requests above `one`
    bytes and totals above `total`."""

    def __init__(self, one, total):
        import torch

        from paper_1507_02509_gb300 import capi

        self.live, self.refused = {}, 0

        def alloc(nbytes, stream, user):
            if nbytes > one or sum(self.live.values()) + nbytes > total:
                self.refused += 1
                return None
            p = torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(), int(stream or 0))
            self.live[p] = nbytes
            return p

        def release(p, stream, user):
            del self.live[p]
            torch.cuda.caching_allocator_delete(int(p))

        self.hooks = (capi.ALLOC_FN(alloc), capi.FREE_FN(release))

    def __enter__(self):
        from paper_1507_02509_gb300 import capi

        capi.kbc_set_allocator(self.hooks[0], self.hooks[1], None)
        return self

    def __exit__(self, *a):
        import paper_1507_02509_gb300 as pkg
        from paper_1507_02509_gb300 import capi

        pkg.use_torch_allocator()
        capi.kbc_set_allocator(*pkg._torch_hooks, None)


@pytest.mark.parametrize("n", [254, 256, 510])
@pytest.mark.parametrize("kind", ["drift", "noise", "along x"])
@pytest.mark.parametrize("limit", ["one", "total"])
def test_half_spectra_where_the_complex_field_does_not_fit(n, kind, limit):
    import torch

    from paper_1507_02509_gb300 import spectra

    rng = np.random.default_rng(n)
    ux, uy = rng.standard_normal((2, n, n))
    if kind == "drift":
        ux, uy = 1e-3 * ux + 0.4, 1e-3 * uy - 0.2
    elif kind == "along x":
        x = 2 * np.pi * np.arange(n)[None, :] / n
        ux, uy = 0.0 * ux, 0.0 * uy + sum(np.cos(k * x) / k for k in range(1, n // 2 + 1))
    tx, ty = torch.as_tensor(ux).cuda(), torch.as_tensor(uy).cuda()
    # 16 n^2 bytes and up to as much work area for the complex transform, half of each for a real one
    with Limited(12 * n * n if limit == "one" else 1 << 40, 24 * n * n if limit == "total" else 1 << 40) as a:
        k, E, Z = spectra.energy_spectrum(tx, ty)
        assert not a.live and (limit == "total" or a.refused >= 1)
    _, ref, _ = ospec.energy_spectrum(ux, uy)
    E, Z, k = E.cpu().numpy(), Z.cpu().numpy(), k.cpu().numpy()
    m = min(len(ref), len(E))
    # double transforms and sums: log2(n^2) roundings of the field's energy
    tol = 2 * np.log2(n * n) * 2.0 ** -52 * (ux ** 2 + uy ** 2).mean()
    assert np.max(np.abs(E[:m] - ref[:m])) <= tol
    assert np.all(np.abs(E[m:]) <= tol) and np.all(np.abs(ref[m:]) <= tol)
    assert np.allclose(Z, (2 * np.pi * k / n) ** 2 * E, rtol=1e-14, atol=0)


def test_no_room_at_all_is_reported():
    import torch

    from paper_1507_02509_gb300 import KBCError, capi, spectra

    u = torch.ones(64, 64, dtype=torch.float64, device="cuda")
    with Limited(1 << 40, 20000) as a:
        with pytest.raises(KBCError) as e:
            spectra.energy_spectrum(u, u)
        assert e.value.status == capi.KBC_ERR_NOMEM and not a.live
    spectra.energy_spectrum(u, u)
