"""Solvers on fields whose reals leave the range of the fixed-point form (below 2^-894 ~ 1e-269), by whole
sites and by spin components, and solutions with components of very different size.

The solvers keep intermediate fields in that form; in FP64 arithmetic such reals add nothing to any norm
and disturb nothing.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_0905_3331_gb300 import (CG_FP64, CG_RELIABLE, CG_SQRT_EPS, F32, F64, LINK12, Lattice,  # noqa: E402
                                   inputs, solve_cg_batch)
from tests._util import from_half, rel, to_half  # noqa: E402

T, L, KAPPA, MU = 16, 4, 0.1, 0.05
SOLVES = {
    "cg_fp64": lambda lat, x, b: lat.solve_cg(x, b, mode=CG_FP64),
    "cg_sqrt_eps": lambda lat, x, b: lat.solve_cg(x, b, mode=CG_SQRT_EPS, sloppy_prec=F32, sloppy_link=LINK12),
    "cg_f32": lambda lat, x, b: lat.solve_cg(x, b, mode=CG_RELIABLE, sloppy_prec=F32, sloppy_link=LINK12),
    "bicgstab_fp64": lambda lat, x, b: lat.solve_bicgstab(x, b, mode=CG_FP64),
    "bicgstab_f32": lambda lat, x, b: lat.solve_bicgstab(x, b, mode=CG_RELIABLE, sloppy_prec=F32),
    "mr_fp64": lambda lat, x, b: lat.solve_mr(x, b, mode=CG_FP64),
    "batch": lambda lat, x, b: solve_cg_batch([(lat, MU, x, b)]),
}


def tail(seed):
    """A source that falls by 39 decades a time slice: 1e-273 and 1e-312 on the farthest."""
    t = np.arange(T)
    return inputs.gaussian_spinor(T, L, seed) * (10.0 ** (-39.0 * np.minimum(t, T - t))).reshape(T, 1, 1, 1, 1, 1)


def half(lat, full):
    out = torch.empty(lat.half_field_bytes(F64) // 8, dtype=torch.float64, device="cuda")
    lat.pack_half(F64, out, torch.from_numpy(to_half(full, 1)).cuda())
    return out


def canonical(lat, d):
    out = torch.empty((lat.h, 4, 3), dtype=torch.complex128, device="cuda")
    lat.unpack_half(F64, out, d)
    return from_half(out.cpu().numpy(), 1, lat.T, lat.L)


@pytest.mark.parametrize("solve", sorted(SOLVES))
def test_tail_source(solve):
    U = inputs.random_gauge(T, L, 0.5, 3)
    b = tail(21)
    with Lattice(T, L, KAPPA, MU) as lat:
        lat.set_gauge(torch.from_numpy(U).cuda())
        x = torch.zeros(b.shape, dtype=torch.complex128, device="cuda")
        SOLVES[solve](lat, x, torch.from_numpy(b).cuda())
        r = b - oracle.apply_M(oracle.Lattice.cubic(T, L), U, x.cpu().numpy(), KAPPA, MU)
    assert np.linalg.norm(r) < 2e-10 * np.linalg.norm(b)  # tol is relative to the prepared source


@pytest.mark.parametrize("mode", [CG_FP64, CG_SQRT_EPS, CG_RELIABLE])
def test_tail_normal(mode):
    U = inputs.random_gauge(T, L, 0.5, 3)
    phi = from_half(to_half(tail(22), 1), 1, T, L)
    with Lattice(T, L, KAPPA, MU) as lat:
        lat.set_gauge(torch.from_numpy(U).cuda())
        X = torch.zeros(lat.half_field_bytes(F64) // 8, dtype=torch.float64, device="cuda")
        lat.solve_normal(X, half(lat, phi), mode=mode)
        r = phi - oracle.normal_op(oracle.Lattice.cubic(T, L), U, canonical(lat, X), KAPPA, MU)
    assert np.linalg.norm(r) < 1e-10 * np.linalg.norm(phi)


def test_tail_chrono():
    U = inputs.random_gauge(T, L, 0.5, 3)
    chi = [from_half(to_half(tail(s), 1), 1, T, L) for s in (23, 24, 25)]
    phi = from_half(to_half(inputs.gaussian_spinor(T, L, 26), 1), 1, T, L)
    with Lattice(T, L, KAPPA, MU) as lat:
        lat.set_gauge(torch.from_numpy(U).cuda())
        X0 = torch.zeros(lat.half_field_bytes(F64) // 8, dtype=torch.float64, device="cuda")
        lat.chrono_guess(X0, [half(lat, c) for c in chi], half(lat, phi))
        ref = oracle.chrono_guess(oracle.Lattice.cubic(T, L), U, chi, phi, KAPPA, MU)
        assert rel(canonical(lat, X0), ref[0] if isinstance(ref, tuple) else ref) < 1e-11


def test_tiny_site_away_from_the_source():
    """A tiny even site that the odd solution does not reach: its neighbours' residual reads it."""
    U = inputs.random_gauge(T, L, 0.5, 3)
    b = np.zeros((T, L, L, L, 4, 3), dtype=np.complex128)
    b[0, 0, 0, 1, 0, 0] = 1.0
    b[8, 0, 0, 0] = 1e-290
    with Lattice(T, L, 1e-3, MU) as lat:
        lat.set_gauge(torch.from_numpy(U).cuda())
        x = torch.zeros(b.shape, dtype=torch.complex128, device="cuda")
        info, = solve_cg_batch([(lat, MU, x, torch.from_numpy(b).cuda())], tol=1e-4)
    assert np.isfinite(info.true_rel_residual) and np.isfinite(x.cpu().numpy()).all()


def test_one_lane_out_of_range():
    """Sites whose spins 1 and 3 (one lane's) are all below 2^-894 beside ordinary spins 0 and 2.  Unit links,
    a field constant in space and coefficients that are powers of two: the hopping sum of the small spins
    is exactly zero in fixed point, and Qhat p holds the small reals of p alone."""
    phi = np.zeros((4, 4, 4, 4, 4, 3), dtype=np.complex128)
    phi[..., 0, :] = 1.0 + 0.5j
    phi[..., 2, :] = 0.25
    phi[..., 1::2, :] = 2.0 ** -930
    phi = from_half(to_half(phi, 1), 1, 4, 4)
    U = inputs.unit_gauge(4, 4)
    with Lattice(4, 4, 0.0625, 0.0) as lat:
        lat.set_gauge(torch.from_numpy(U).cuda())
        X = torch.zeros(lat.half_field_bytes(F64) // 8, dtype=torch.float64, device="cuda")
        lat.solve_normal(X, half(lat, phi))
        r = phi - oracle.normal_op(oracle.Lattice.cubic(4, 4), U, canonical(lat, X), 0.0625, 0.0)
    assert np.linalg.norm(r) < 1e-10 * np.linalg.norm(phi)


@pytest.mark.parametrize("solve", sorted(SOLVES))
def test_components_of_a_solution(solve):
    """Without hopping to speak of (kappa 1e-60, mu~ 0.02) x = b (1 - i mu~ gamma5) / (1 + mu~^2), component by
    component; the FP64 numbers returned keep small components beside large ones.  FP64 roundings: 1e-14
    covers a few dozen; on the odd sites the mixed solvers and MR stop at a residual of tol."""
    rng = np.random.default_rng(6)
    b = inputs.gaussian_spinor(4, 4, 7) * 10.0 ** -rng.uniform(0, 25, (4, 4, 4, 4, 4, 3))
    mut = 0.02
    U = inputs.random_gauge(4, 4, 0.5, 3)
    with Lattice(4, 4, 1e-60, mut / 2e-60) as lat:
        lat.set_gauge(torch.from_numpy(U).cuda())
        x = torch.zeros(b.shape, dtype=torch.complex128, device="cuda")
        SOLVES[solve](lat, x, torch.from_numpy(b).cuda()) if solve != "batch" else solve_cg_batch(
            [(lat, mut / 2e-60, x, torch.from_numpy(b).cuda())])
    sign = np.array([1.0, 1.0, -1.0, -1.0]).reshape(4, 1)
    ref = b * (1.0 - 1j * mut * sign) / (1.0 + mut * mut)
    err = np.abs(x.cpu().numpy() - ref) / np.abs(ref)
    t, z, y, w = np.indices(b.shape[:4])
    even = (t + z + y + w) % 2 == 0
    assert err[even].max() < 1e-14
    if solve in ("cg_fp64", "bicgstab_fp64"):
        assert err[~even].max() < 1e-14
