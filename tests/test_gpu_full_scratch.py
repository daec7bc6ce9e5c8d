"""The full operator with more right-hand sides than before: its work buffer has one size per lattice, and its
launches stay within a grid's extents."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_0905_3331_gb300 import F64, LINK18, Lattice, inputs  # noqa: E402

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


def test_capture_before_the_buffer_exists():
    """Two fields of 54880 sites need the buffer, one does not: captured first, they do without."""
    T, L = 20, 14
    with lattice(T, L) as lat:
        x = fields(2, T, L)
        y, z = torch.zeros_like(x), torch.zeros_like(x)
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):
            lat.apply_D(z[:1], x[:1])
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                lat.apply_D(y, x, nrhs=2)
            g.replay()
            lat.apply_D(z, x, nrhs=2)
        torch.cuda.synchronize()
        assert torch.equal(y, z)


@pytest.mark.parametrize("threads", [0, 1])
def test_more_fields_than_a_grid_dimension(threads):
    """65600 fields on 2^4 against the same fields in three calls."""
    n = 65600
    with lattice(2, 2) as lat:
        if threads:
            lat.set_hop_threads(F64, LINK18, threads)
        x = fields(n, 2, 2)
        y, z = torch.zeros_like(x), torch.zeros_like(x)
        lat.apply_D(y, x, nrhs=n)
        for a, b in ((0, 30000), (30000, 60000), (60000, n)):
            lat.apply_D(z[a:b], x[a:b], nrhs=b - a)
        assert torch.equal(y, z)
