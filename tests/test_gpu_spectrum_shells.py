"""Shell sums of kbc_spectrum for fields with a mean, one direction only, and
sizes at the edges of the binning's runs of eight columns and warps of 256."""
import numpy as np
import pytest

from oracle import spectra as ospec

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 4, 6, 14, 16, 18, 254, 256, 258, 510, 520])
@pytest.mark.parametrize("kind", ["drift", "noise", "along x", "long waves"])
def test_shell_sums_match_the_plain_loop(n, kind):
    import torch

    from paper_1507_02509_gb300 import spectra

    rng = np.random.default_rng(n)
    ux, uy = rng.standard_normal((2, n, n))
    x = 2 * np.pi * np.arange(n)[None, :] / n
    if kind == "drift":
        ux, uy = 1e-3 * ux + 0.4, 1e-3 * uy - 0.2
    elif kind == "along x":
        ux, uy = 0.0 * ux, 0.0 * uy + sum(np.cos(k * x) / k for k in range(1, n // 2 + 1))
    elif kind == "long waves":
        ux, uy = np.cos(x) * np.sin(x.T), 1.0 + 0.5 * np.sin(x) * np.cos(x.T)
    k, E, Z = spectra.energy_spectrum(torch.as_tensor(ux).cuda(), torch.as_tensor(uy).cuda())
    _, ref, _ = ospec.energy_spectrum(ux, uy)
    E, Z, k = E.cpu().numpy(), Z.cpu().numpy(), k.cpu().numpy()
    m = min(len(ref), len(E))
    # double transforms and sums: log2(n^2) roundings of the field's energy
    tol = 2 * np.log2(n * n) * 2.0 ** -52 * (ux ** 2 + uy ** 2).mean()
    assert np.max(np.abs(E[:m] - ref[:m])) <= tol
    assert np.all(np.abs(E[m:]) <= tol) and np.all(np.abs(ref[m:]) <= tol)
    assert np.allclose(Z, (2 * np.pi * k / n) ** 2 * E, rtol=1e-14, atol=0)
