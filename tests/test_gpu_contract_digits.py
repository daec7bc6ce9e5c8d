"""The digit-split contraction where its integer sums and exponents can go wrong.

Bound: an entry A[j][k] is a sum of n terms |a||b|, each off by at most 2^-54 of the largest |a| times
|b| and vice versa (rounding to 55 bits below the largest real of a tile) plus FP64 roundings of the
drained partial sums: |dA| <= 2^-50 (max_j sum|b| + max_k sum|a|) over the timeslice, far above what is
seen and far below a wrong digit (2^-8 and up of a digit's weight: the lowest weigh 2^-46).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_0905_3331_gb300 import Lattice  # noqa: E402


def gram(x, T):
    """In extended precision: numpy's own FP64 sums are off by as much as the bound."""
    re, im = (v.reshape(12, T, -1).astype(np.longdouble) for v in (x.real, x.imag))
    dot = lambda a, b: np.einsum("jtn,ktn->tjk", a, b)  # noqa: E731
    return (dot(re, re) + dot(im, im)).astype(float) + 1j * (dot(re, im) - dot(im, re)).astype(float)


def propagators(kind, T, L):
    rng = np.random.default_rng(11)
    shape = (12, T, L, L, L, 4, 3)
    x = rng.normal(size=shape) + 1j * rng.normal(size=shape)
    if kind == "digits":  # every digit at -128 or 127, all products of one sign
        a, b = float(int("7f" * 6, 16)), -float(int("80" * 6, 16))
        x = np.where(rng.random(shape[:1] + (1,) * 6) < 0.5, a, b) * (1 + 1j) * np.ones(shape) * 2.0 ** -46
    if kind == "growing":  # the exponents grow tile by tile, for half of the propagators
        g = np.exp2(np.linspace(0, 60, L ** 3)).reshape(1, 1, L, L, L, 1, 1)
        x[::2] = (x * g)[::2]
    if kind == "sparse":  # a propagator that is zero, and one that is zero but for the last site
        x[3] = 0.0
        x[7] = 0.0
        x[7, :, -1, -1, -1] = 1.0
    if kind == "tiny":  # reals outside the fixed-point range next to ordinary ones
        x[2] *= 1e-290
        x[5, :, :1] *= 1e295
    return x


@pytest.mark.parametrize("T,L", [(2, 2), (4, 4), (2, 6), (2, 10)])
@pytest.mark.parametrize("kind", ["gauss", "digits", "growing", "sparse", "tiny"])
def test_digits(T, L, kind):
    x = propagators(kind, T, L)
    with np.errstate(over="ignore", invalid="ignore"):
        ref = gram(x, T)
    with Lattice(T, L, 0.16, 0.01) as lat:
        got = lat.meson_contract(torch.from_numpy(x).cuda(),
                                 out=torch.zeros((T, 12, 12), dtype=torch.complex128, device="cuda")).cpu().numpy()
    f = np.isfinite(ref)
    assert np.array_equal(f, np.isfinite(got))
    a = np.abs(x).reshape(12, T, -1)
    with np.errstate(over="ignore", invalid="ignore"):
        m, s = a.max(-1).T, a.sum(-1).T
        bound = 2.0 ** -50 * (m[:, :, None] * s[:, None, :] + s[:, :, None] * m[:, None, :])
    assert np.all(np.abs(got[f] - ref[f]) <= bound[f] + 1e-300)


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_non_finite(bad):
    """A non-finite entry makes that propagator's entries of its timeslice non-finite, and no others."""
    T, L = 4, 4
    x = propagators("gauss", T, L)
    x[4, 2, 3, 1, 0, 2, 1] = bad
    with Lattice(T, L, 0.16, 0.01) as lat:
        got = lat.meson_contract(torch.from_numpy(x).cuda(),
                                 out=torch.zeros((T, 12, 12), dtype=torch.complex128, device="cuda")).cpu().numpy()
    hit = np.zeros((T, 12, 12), dtype=bool)
    hit[2, 4, :] = hit[2, :, 4] = True
    assert not np.isfinite(got[hit]).any()
    assert np.isfinite(got[~hit]).all()
