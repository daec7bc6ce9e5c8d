"""Solvers on fields whose reals leave the range of the fixed-point form (below 2^-894 ~ 1e-269).

The solvers keep intermediate fields in that form; in FP64 arithmetic such reals add nothing to any norm
and disturb nothing.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_0905_3331_gb300 import F64, Lattice, inputs  # noqa: E402
from tests._util import from_half, to_half  # noqa: E402


def half(lat, full):
    out = torch.empty(lat.half_field_bytes(F64) // 8, dtype=torch.float64, device="cuda")
    lat.pack_half(F64, out, torch.from_numpy(to_half(full, 1)).cuda())
    return out


def canonical(lat, d):
    out = torch.empty((lat.h, 4, 3), dtype=torch.complex128, device="cuda")
    lat.unpack_half(F64, out, d)
    return from_half(out.cpu().numpy(), 1, lat.T, lat.L)


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
