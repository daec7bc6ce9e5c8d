"""The fixed-point form of the FP64 hopping sum (18-real links) at the places where it can go wrong.

Bounds.  A site's sum is off by a few units of 2^-57 of its largest neighbour real (times eight hops)
before it is rounded to FP64, and the oracle's own FP64 sum by its ~48 roundings: below 4e-15 of the
largest neighbour real.  A lost carry between the two 32-bit limbs is 2^-27 ~ 7e-9 of it.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_0905_3331_gb300 import F64, LINK18, Lattice, inputs  # noqa: E402
from tests._util import from_half, to_half  # noqa: E402

TOL = 4e-15


def largest_neighbour(src_full):
    """Per site, the largest |re| or |im| of its eight neighbours."""
    m = np.maximum(np.abs(src_full.real), np.abs(src_full.imag)).max((-2, -1))
    return np.max([np.roll(m, s, axis=a) for a in range(4) for s in (1, -1)], axis=0)


def fields(kind, T, L):
    rng = np.random.default_rng(5)
    shape = (T, L, L, L, 4, 3)
    psi = inputs.gaussian_spinor(T, L, 8)
    if kind == "limbs":  # multiples of 2^-27 below 2: low limbs of exactly -2^31, 0 and neighbours of them
        n = rng.integers(-2 ** 28, 2 ** 28, shape + (2,))
        n = (n >> 3 << 3) + rng.integers(0, 3, n.shape)
        return (n[..., 0] + 1j * n[..., 1]) * 2.0 ** -27
    if kind == "point":  # zero neighbours on one side, one component on the other
        q = np.zeros_like(psi)
        q[0, 0, 0, 0, 1, 2] = 1.0
        q[1, 0, 0, 0, 0, 0] = 1e-3j
        return q
    if kind == "wide":  # neighbours of very different size: the sum is shifted right, also by over 63 bits
        return psi * 10.0 ** rng.uniform(-30, 30, shape[:4] + (1, 1))
    if kind == "growing":  # each time slice far above the one before
        return psi * 10.0 ** (4.0 * np.arange(T)).reshape(T, 1, 1, 1, 1, 1)
    return psi * 10.0 ** rng.choice([-305.0, -280.0, 0.0, 290.0, 297.0], shape[:4] + (1, 1))  # "range"


@pytest.mark.parametrize("T,L", [(4, 4), (10, 6)])
@pytest.mark.parametrize("threads", [1, 2, 4])
@pytest.mark.parametrize("kind", ["limbs", "point", "wide", "growing", "range"])
def test_fixed_point_sum(T, L, threads, kind):
    U = inputs.random_gauge(T, L, 0.5, 3)
    olat = oracle.Lattice.cubic(T, L)
    psi = fields(kind, T, L)
    with Lattice(T, L, 0.16, 0.01) as lat:
        lat.set_gauge(torch.from_numpy(U).cuda())
        lat.set_hop_threads(F64, LINK18, threads)
        nb = lat.half_field_bytes(F64)
        for p in (0, 1):
            src = to_half(psi, 1 - p)
            full = from_half(src, 1 - p, T, L)
            ref = to_half(oracle.hopping(olat, U, full, out_parity=p), p)
            size = to_half(np.broadcast_to(largest_neighbour(full)[..., None, None], psi.shape), p)[:, 0, 0]
            din = torch.empty(nb, dtype=torch.uint8, device="cuda")
            dout = torch.empty(nb, dtype=torch.uint8, device="cuda")
            got = torch.empty(src.shape, dtype=torch.complex128, device="cuda")
            lat.pack_half(F64, din, torch.from_numpy(src).cuda())
            lat.apply_hopping_eo(p, dout, din, F64, LINK18)
            lat.unpack_half(F64, got, dout)
            # (a site may be beyond the FP64 range in squares: largest entry, not norm)
            err = np.abs(got.cpu().numpy() - ref).max((1, 2))
            assert np.all(err <= TOL * size), float((err / np.maximum(size, 1e-300)).max())


@pytest.mark.parametrize("threads", [1, 2, 4])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_non_finite_neighbours(threads, bad):
    """A non-finite entry makes exactly the sites next to it non-finite; the others are untouched."""
    T, L = 6, 4
    U = inputs.random_gauge(T, L, 0.5, 3)
    psi = inputs.gaussian_spinor(T, L, 8)
    psi[2, 1, 3, 0, 2, 1] = bad
    p = (2 + 1 + 3 + 0 + 1) & 1
    clean = psi.copy()
    clean[2, 1, 3, 0] = 0.0
    near = np.zeros(psi.shape[:4], dtype=bool)
    near[2, 1, 3, 0] = True
    near = np.any([np.roll(near, s, axis=a) for a in range(4) for s in (1, -1)], axis=0)
    near = to_half(np.broadcast_to(near[..., None, None], psi.shape), p)[:, 0, 0].astype(bool)
    with Lattice(T, L, 0.16, 0.01) as lat:
        lat.set_gauge(torch.from_numpy(U).cuda())
        lat.set_hop_threads(F64, LINK18, threads)
        out = []
        for f in (psi, clean):
            src = to_half(f, 1 - p)
            din = torch.empty(lat.half_field_bytes(F64), dtype=torch.uint8, device="cuda")
            dout = torch.empty_like(din)
            got = torch.empty(src.shape, dtype=torch.complex128, device="cuda")
            lat.pack_half(F64, din, torch.from_numpy(src).cuda())
            lat.apply_hopping_eo(p, dout, din, F64, LINK18)
            lat.unpack_half(F64, got, dout)
            out.append(got.cpu().numpy())
    assert not np.isfinite(out[0][near]).all((1, 2)).any()
    assert np.array_equal(out[0][~near], out[1][~near])
