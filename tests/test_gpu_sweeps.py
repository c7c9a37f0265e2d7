"""Fields beyond L2, which successive steps sweep in opposite directions and
whose kernels differ from those of smaller ones."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", ["lbgk", "B", "C"])
@pytest.mark.parametrize("dtype,nx,ny", [("f32", 2048, 901), ("f16", 2048, 1801), ("f64", 2048, 451)])
def test_kernels_and_slabs_agree_beyond_l2(variant, dtype, nx, ny):
    """Vector rows, bulk copies and the per-node kernel give the same bits
    after three steps (one replay parity broken on purpose), and so do uneven
    slabs."""
    import torch

    from paper_1507_02509_gb300 import Lattice
    from paper_1507_02509_gb300.slabs import SlabGroup

    g = torch.Generator(device="cuda")
    g.manual_seed(4)
    rho = 1.0 + 0.01 * torch.randn(ny, nx, dtype=torch.float64, device="cuda", generator=g)
    ux, uy = 0.03 * torch.randn(2, ny, nx, dtype=torch.float64, device="cuda", generator=g)
    kw = dict(variant=variant, beta=0.98, dtype=dtype)
    out = []
    for kernel in ("rows", "bulk", "nodes", "auto"):
        lat = Lattice(nx, ny, **kw)
        lat.set_kernel(kernel)
        lat.init(rho, ux, uy).step(1).step(2)
        out.append(lat.populations())
        lat.close()
    group = SlabGroup(nx, ny, 3, **kw)
    group.init(rho, ux, uy).step(1).step(2)
    out.append(group.populations())
    group.close()
    for q in out[1:]:
        assert torch.equal(out[0], q)
