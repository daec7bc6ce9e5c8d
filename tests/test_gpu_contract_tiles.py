"""The digit-split contraction with many tiles per block: 16^3 sites in 384 tiles over 19 blocks a
timeslice, 20 or 21 tiles a block -- three exact sums of 1024 components, raw buffers used ten times, and
exponents that change over running sums.

Bound as in test_gpu_contract_digits.py: |dA| <= 2^-50 (max_j sum|b| + max_k sum|a|) over the timeslice.
All timeslices hold the same numbers, so that one of them is compared and the others have to be equal.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_0905_3331_gb300 import Lattice  # noqa: E402

T, L = 16, 16
SITES = L ** 3
TILE = 128 // 12  # whole sites in a tile, about


def slice_of(kind):
    """(12, sites, 12) complex: one timeslice of the twelve propagators."""
    rng = np.random.default_rng(12)
    x = rng.normal(size=(12, SITES, 12)) + 1j * rng.normal(size=(12, SITES, 12))
    along = np.linspace(0.0, 1.0, SITES).reshape(1, SITES, 1)
    if kind == "digits":  # every digit at -128 or 127, all products of one sign: sums up to 2^24
        a, b = float(int("7f" * 6, 16)), -float(int("80" * 6, 16))
        x = np.where(rng.random((12, 1, 1)) < 0.5, a, b) * (1 + 1j) * np.ones(x.shape) * 2.0 ** -46
    if kind == "rising":  # three binades from one tile of a block to its next, for half of the propagators
        x[::2] = (x * np.exp2(60 * along))[::2]
    if kind == "falling":
        x[1::2] = (x * np.exp2(-60 * along))[1::2]
    if kind == "steps":  # up and down by 24 binades every seven tiles of a block
        x[::3] = (x * np.exp2(24.0 * (np.arange(SITES) // (7 * 19 * TILE) % 2)).reshape(1, SITES, 1))[::3]
    if kind == "amid":  # one tile of every block, amid its running sums, below the fixed-point range
        x[:, 10 * 19 * TILE:11 * 19 * TILE] *= 1e-290
    if kind == "sparse":  # a propagator that is zero, and one that is zero but for the last site
        x[3] = 0.0
        x[7] = 0.0
        x[7, -1] = 1.0
    return x


@pytest.mark.parametrize("kind", ["gauss", "digits", "rising", "falling", "steps", "amid", "sparse"])
def test_many_tiles(kind):
    x = slice_of(kind)
    flat = x.reshape(12, -1)
    re, im = (v.astype(np.longdouble) for v in (flat.real, flat.imag))
    dot = lambda a, b: np.einsum("jn,kn->jk", a, b)  # noqa: E731
    ref = (dot(re, re) + dot(im, im)).astype(float) + 1j * (dot(re, im) - dot(im, re)).astype(float)
    props = torch.from_numpy(x).cuda().view(12, 1, SITES, 12).expand(12, T, SITES, 12).contiguous()
    with Lattice(T, L, 0.16, 0.01) as lat:
        got = lat.meson_contract(props, out=torch.zeros((T, 12, 12), dtype=torch.complex128, device="cuda")).cpu().numpy()
    m, s = np.abs(flat).max(1), np.abs(flat).sum(1)
    bound = 2.0 ** -50 * (m[:, None] * s[None, :] + s[:, None] * m[None, :])
    assert np.all(np.abs(got[0] - ref) <= bound + 1e-300)
    assert np.array_equal(got, np.broadcast_to(got[0], got.shape))
