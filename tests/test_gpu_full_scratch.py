"""The work buffer of the full operator: one size per lattice, whatever the number of right-hand sides."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_0905_3331_gb300 import Lattice, inputs  # noqa: E402

BIG = (20, 16)  # 81920 sites: the form with a work buffer


def fields(n, T, L, seed=4):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.view_as_complex(torch.randn((n, T, L, L, L, 4, 3, 2), generator=g, device="cuda", dtype=torch.float64))


def lattice(T, L):
    lat = Lattice(T, L, 0.16, 0.01)
    lat.set_gauge(torch.from_numpy(inputs.random_gauge(T, L, 0.5, 3)).cuda())
    return lat


def test_more_fields_allocate_nothing():
    with lattice(*BIG) as lat:
        x = fields(12, *BIG)
        y = torch.zeros_like(x)
        lat.apply_D(y[:1], x[:1])
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        lat.apply_D(y, x, nrhs=12)
        torch.cuda.synchronize()
        assert torch.cuda.mem_get_info()[0] == free


def test_captured_call_before_more_fields():
    """A graph of a one-field call, replayed after a call with more fields; and that call captured too."""
    with lattice(*BIG) as lat:
        x = fields(12, *BIG)
        y, z, w = (torch.zeros_like(x) for _ in range(3))
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):
            lat.apply_D(z[:1], x[:1])
            one, many = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
            with torch.cuda.graph(one, stream=s):
                lat.apply_D(y[:1], x[:1])
            lat.apply_D(z, x, nrhs=12)
            with torch.cuda.graph(many, stream=s):
                lat.apply_D(w, x, nrhs=12)
            one.replay()
            many.replay()
        torch.cuda.synchronize()
        assert torch.equal(y[0], z[0]) and torch.equal(w, z)
