"""The check of set_gauge: any one entry of any one link, the determinant, overflowing products."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_0905_3331_gb300 import Lattice, TMError, inputs  # noqa: E402


@pytest.mark.parametrize("T,L", [(2, 2), (4, 6)])  # 64 links; 3456: 13.5 blocks
def test_one_bad_link_is_refused(T, L):
    U = inputs.random_gauge(T, L, 0.5, 3)
    flat = U.reshape(-1, 3, 3)
    n = flat.shape[0]

    def status(link, change):
        bad = flat.copy()
        bad[link] = change(bad[link])
        with Lattice(T, L, 0.16, 0.01) as lat:
            try:
                lat.set_gauge(torch.from_numpy(bad.reshape(U.shape)).cuda())
            except TMError as e:
                return e.status_name
        return None

    def add(a, b, d):
        def f(m):
            m = m.copy()
            m[a, b] += d
            return m
        return f

    assert status(0, lambda m: m) is None
    for a in range(3):
        for b in range(3):
            for link in (0, 31, n - 1):
                # |U^dag U - 1| changes by |d| times a row of U, whose largest entry is at least 1 / sqrt(3)
                assert status(link, add(a, b, 1e-9)) == "TM_ERR_NOT_SU3"
            assert status(n - 1, add(a, b, 1e-12j)) is None
            assert status(n - 2, add(a, b, 1e200)) == "TM_ERR_NOT_SU3"
            assert status(n - 2, add(a, b, 1e200 - 1e200j)) == "TM_ERR_NOT_SU3"
            assert status(n - 3, add(a, b, np.inf)) == "TM_ERR_NONFINITE"
    assert status(n - 1, lambda m: m * np.exp(1e-9j)) == "TM_ERR_NOT_SU3"  # unitary, det exp(3e-9 i)
