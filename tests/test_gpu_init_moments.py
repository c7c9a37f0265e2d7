"""Equilibrium initialisation and moments where their double arithmetic is
replaced by pairs of floats and integer sums: the stored values are those of
the double computation, and rho and u are those of the stored values."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

W = np.array([1 / 36, 1 / 9, 1 / 36, 1 / 9, 4 / 9, 1 / 9, 1 / 36, 1 / 9, 1 / 36])
A = np.array([i % 3 - 1 for i in range(9)])
B = np.array([i // 3 - 1 for i in range(9)])


def fields(kind, ny, nx, seed):
    rng = np.random.default_rng(seed)
    rho = 1.0 + 0.02 * rng.standard_normal((ny, nx))
    ux, uy = 0.05 * rng.standard_normal((2, ny, nx))
    if kind == "constant density":
        rho[:] = 1.0
    elif kind == "dense":
        rho += 6.5          # rho - 1 at the edge of the split's range and above it
        rho[0, 0] = 9.5
    elif kind == "wide":    # magnitudes down to where the split cuts off, and zeros
        ux *= np.exp2(-90 * rng.random((ny, nx)))
        uy *= np.exp2(-30 * rng.random((ny, nx)))
        uy[::2] = 0.0
        ux[0, 0] = 0.0
        rho[:, ::3] = 1.0
    return rho, ux, uy


def deviations(rho, ux, uy):
    """f^eq - W in long double."""
    r, x, y = (q.astype(np.longdouble) for q in (rho, ux, uy))
    xi = [a * x + b * y for a, b in zip(A, B)]
    n, d = np.longdouble(1), []
    for i in range(9):
        w = {0: n * 4 / 9, 1: n / 9, 2: n / 36}[abs(A[i]) + abs(B[i])]
        d.append(w * ((r - 1) + r * (3 * xi[i] + 4.5 * xi[i] ** 2 - 1.5 * (x * x + y * y))))
    return np.array(d)


@pytest.mark.parametrize("kind", ["turbulent", "constant density", "dense", "wide"])
@pytest.mark.parametrize("shape", [(1, 1), (3, 1), (257, 3), (512, 300)])
@pytest.mark.parametrize("dtype,scale", [("f32", 1.0), ("f16", 1.0), ("f16", 6.0), ("f16", 0.0625)])
def test_init_stores_the_rounded_equilibrium(kind, shape, dtype, scale):
    from paper_1507_02509_gb300 import Lattice

    nx, ny = shape
    rho, ux, uy = fields(kind, ny, nx, 5)
    lat = Lattice(nx, ny, variant="B", beta=0.97, dtype=dtype)
    if dtype == "f16":
        lat.set_f16_scale(scale)
    lat.init(rho, ux, uy)
    got = lat.populations().cpu().numpy()
    lat.close()
    d, w = deviations(rho, ux, uy), W.reshape(9, 1, 1)
    if dtype == "f32":
        want = d.astype(np.float32).astype(np.float64) + w
    else:
        s = float(np.float32(scale))
        code = (d / np.longdouble(1) / w * s).astype(np.float16).astype(np.float64)
        want = code * (w * float(np.float32(1.0 / s))) + w  # the codec keeps 1 / S as a float
    # a double computation is within 2^-50 of the terms it adds: the rounding
    # to the stored type may differ from the long double one only where the
    # value is that close to halfway, about 2^-50 2^24 of all float values and
    # fewer halves; f itself carries the rounding of + W and of W / S
    far = np.abs(got - want) > 4e-16 * np.abs(want)
    assert far.sum() <= 2, f"{far.sum()} of {far.size} stored values differ"
    assert np.all(np.abs(got - want) <= np.abs(d.astype(np.float64)) * (2.0 ** -22 if dtype == "f32" else 2.0 ** -9) + 1e-15)


def test_init_passes_nonfinite_values_on():
    from paper_1507_02509_gb300 import Lattice

    for dtype in ("f64", "f32", "f16"):
        for bad in (np.nan, np.inf):
            rho, ux, uy = fields("turbulent", 3, 40, 1)
            ux[1, 7] = bad
            lat = Lattice(40, 3, variant="C", beta=0.97, dtype=dtype)
            lat.init(rho, ux, uy)
            f = lat.populations().cpu().numpy()
            m = lat.moments()
            lat.close()
            assert not np.isfinite(f[:, 1, 7]).any()
            assert np.isfinite(np.delete(f.reshape(9, -1), 47, axis=1)).all()
            assert not np.isfinite(m[1].cpu().numpy()[1, 7])


@pytest.mark.parametrize("dtype,scale", [("f32", 1.0), ("f16", 1.0), ("f16", 6.0), ("f64", 1.0)])
@pytest.mark.parametrize("kind", ["ordinary", "spread", "tiny", "rest"])
def test_moments_of_the_stored_populations(dtype, scale, kind):
    from paper_1507_02509_gb300 import Lattice

    nx, ny = 65, 7
    rng = np.random.default_rng(11)
    d = 0.01 * rng.standard_normal((9, ny, nx)) * W.reshape(9, 1, 1) * 9
    if kind == "spread":   # some nodes with values more than 30 binary places apart
        d *= np.exp2(-60 * rng.random((9, ny, nx)) * (rng.random((ny, nx)) < 0.3))
    elif kind == "tiny":
        d *= 2.0 ** -70
    elif kind == "rest":
        d[:, :, ::2] = 0.0
    lat = Lattice(nx, ny, variant="B", beta=0.97, dtype=dtype)
    if dtype == "f16":
        lat.set_f16_scale(scale)
    f0 = d + W.reshape(9, 1, 1)
    lat.set_populations(f0)
    rho, ux, uy = (q.cpu().numpy() for q in lat.moments())
    lat.close()
    # what the storage holds, from the definition of the codecs
    dev = f0 - W.reshape(9, 1, 1)
    if dtype == "f32":
        dev = dev.astype(np.float32).astype(np.longdouble)
    elif dtype == "f16":
        iw = np.array([36.0, 9.0, 36.0, 9.0, 2.25, 9.0, 36.0, 9.0, 36.0]).reshape(9, 1, 1)
        dev = (dev * (iw * scale)).astype(np.float16).astype(np.longdouble) / iw * np.longdouble(np.float32(1.0 / scale))
    dev = dev.astype(np.longdouble)
    r = 1 + dev.sum(0)
    jx, jy = np.tensordot(A, dev, 1), np.tensordot(B, dev, 1)
    size = np.abs(dev).sum(0)
    # one rounding of rho, at most eight of a sum and three of the quotient
    eps = 2.0 ** -52
    assert np.all(np.abs(rho - r) <= eps * np.abs(r) + 8 * eps * size)
    for got, j in ((ux, jx), (uy, jy)):
        assert np.all(np.abs(got - j / r) <= 4 * eps * np.abs(j / r) + 8 * eps * size)
