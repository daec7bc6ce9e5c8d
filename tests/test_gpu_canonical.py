"""Canonical fields through the shared-memory tiles: addresses, ragged tails, extreme values, many
right-hand sides of the full operator."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_0905_3331_gb300 import DF64, F16, F32, F64, Lattice, inputs  # noqa: E402


def off8(x):
    """A copy of x at an address that is a multiple of 8 and not of 16."""
    buf = torch.empty(2 * x.numel() + 2, dtype=torch.float64, device="cuda")
    skip = 1 if buf.data_ptr() % 16 == 0 else 2
    v = buf[skip:skip + 2 * x.numel()]
    v.copy_(torch.view_as_real(x).reshape(-1))
    assert v.data_ptr() % 16 == 8
    return v


def cgauss(*shape, seed=4):
    return torch.from_numpy(np.random.default_rng(seed).normal(size=shape + (2,)).view(np.complex128)[..., 0]).cuda()


@pytest.mark.parametrize("T,L", [(2, 2), (4, 6), (10, 6)])
@pytest.mark.parametrize("prec", [F64, F32, F16, DF64])
def test_half_fields_at_8_byte_addresses(T, L, prec):
    with Lattice(T, L, 0.16, 0.01) as lat:
        x = cgauss(3, lat.h, 4, 3)
        a, b = (torch.zeros(3 * lat.half_field_bytes(prec), dtype=torch.uint8, device="cuda") for _ in range(2))
        lat.pack_half(prec, a, x, nrhs=3)
        lat.pack_half(prec, b, off8(x), nrhs=3)
        assert torch.equal(a, b)
        u, w = torch.zeros_like(x), off8(torch.zeros_like(x))
        lat.unpack_half(prec, u, a, nrhs=3)
        lat.unpack_half(prec, w, a, nrhs=3)
        assert torch.equal(torch.view_as_real(u).reshape(-1), w)
        if prec == F64:
            assert torch.equal(u, x)


@pytest.mark.parametrize("T,L", [(2, 2), (4, 6), (10, 6)])
@pytest.mark.parametrize("dagger", [False, True])
def test_apply_D_at_8_byte_addresses(T, L, dagger):
    U = inputs.random_gauge(T, L, 0.5, 3)
    with Lattice(T, L, 0.16, 0.01) as lat:
        lat.set_gauge(torch.from_numpy(U).cuda())
        x = cgauss(2, T, L, L, L, 4, 3)
        a, b = torch.zeros_like(x), off8(torch.zeros_like(x))
        lat.apply_D(a, x, dagger=dagger, nrhs=2)
        lat.apply_D(b, off8(x), dagger=dagger, nrhs=2)
        assert torch.equal(torch.view_as_real(a).reshape(-1), b)


@pytest.mark.parametrize("threads", [1, 2, 4])
@pytest.mark.parametrize("dagger", [False, True])
def test_apply_D_of_extreme_values(threads, dagger):
    """Sites outside the fixed-point range next to ordinary ones: every entry within 1e-14 of the
    largest real of the site and its neighbours (FP64 sums of ~50 terms; see test_gpu_fixed_point)."""
    T, L = 4, 6
    U = inputs.random_gauge(T, L, 0.5, 3)
    rng = np.random.default_rng(7)
    psi = inputs.gaussian_spinor(T, L, 8) * 10.0 ** rng.choice([-305.0, -290.0, 0.0, 295.0], (T, L, L, L, 1, 1))
    g5 = np.array([1, 1, -1, -1])[:, None]
    olat = oracle.Lattice.cubic(T, L)
    mu = 0.01
    ref = g5 * oracle.apply_M(olat, U, g5 * psi, 0.16, -mu) if dagger else oracle.apply_M(olat, U, psi, 0.16, mu)
    m = np.maximum(np.abs(psi.real), np.abs(psi.imag)).max((-2, -1))
    size = np.max([m] + [np.roll(m, s, axis=a) for a in range(4) for s in (1, -1)], axis=0)
    with Lattice(T, L, 0.16, mu) as lat:
        lat.set_gauge(torch.from_numpy(U).cuda())
        lat.set_hop_threads(F64, 18, threads)
        x = torch.from_numpy(psi).cuda()
        out = torch.zeros_like(x)
        lat.apply_D(out, x, dagger=dagger)
    d = out.cpu().numpy() - ref
    assert np.all(np.maximum(np.abs(d.real), np.abs(d.imag)).max((-2, -1)) <= 1e-14 * size)


def test_apply_D_of_many_right_hand_sides():
    """More right-hand sides than the scratch holds at a time: each as by itself."""
    T, L, n = 24, 12, 34
    with Lattice(T, L, 0.16, 0.01) as lat:
        lat.set_gauge(torch.from_numpy(inputs.random_gauge(T, L, 0.5, 3)).cuda())
        x = torch.randn((n, T, L, L, L, 4, 3), dtype=torch.complex128, device="cuda")
        out, one = torch.zeros_like(x), torch.zeros_like(x[0])
        lat.apply_D(out, x, nrhs=n)
        for r in (0, 31, 32, 33):
            lat.apply_D(one, x[r])
            assert torch.equal(out[r], one)


@pytest.mark.parametrize("T,L", [(2, 4), (10, 6), (16, 8), (16, 10), (24, 12)])
def test_apply_D_of_a_field_beside_others(T, L):
    """A field's result has the same bits alone and beside enough others to pass 65536 sites, for one,
    two and four thread pairs per site; sites outside the fixed-point range and zero sites among them."""
    n = 65536 // (T * L ** 3) + 1
    with Lattice(T, L, 0.16, 0.01) as lat:
        lat.set_gauge(torch.from_numpy(inputs.random_gauge(T, L, 0.5, 3)).cuda())
        g = torch.Generator(device="cuda").manual_seed(5)
        x = torch.randn((n, T, L, L, L, 4, 3), dtype=torch.complex128, device="cuda", generator=g)
        scale = torch.tensor([0.0, 1e-306, 1e-20, 1.0, 1.0, 1.0, 1.0, 1e300], dtype=torch.float64, device="cuda")
        x *= scale[torch.randint(8, (n, T, L, L, L, 1, 1), device="cuda", generator=g)]
        out, one = torch.zeros_like(x), torch.zeros_like(x[0])
        for dagger in (False, True):
            lat.apply_D(out, x, dagger=dagger, nrhs=n)
            for r in (0, n - 1):
                lat.apply_D(one, x[r], dagger=dagger)
                assert torch.equal(out[r], one)
