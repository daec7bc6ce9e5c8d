"""Double-float fields unpacked by whole records (small calls) and through the shared-memory tile (large
ones): the same numbers, at 16-byte and at 8-byte addresses."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_0905_3331_gb300 import DF64, Lattice  # noqa: E402

MANY = 330  # fields of 1080 sites: 68 MB canonical, the tile


@pytest.mark.parametrize("offset", [0, 1])
def test_unpack_of_many_fields(offset):
    with Lattice(10, 6, 0.16, 0.01) as lat:
        g = torch.Generator(device="cuda").manual_seed(3)
        x = torch.randn((MANY, 24 * lat.h), generator=g, device="cuda", dtype=torch.float64)
        half = torch.zeros((MANY, lat.half_field_bytes(DF64)), dtype=torch.uint8, device="cuda")
        lat.pack_half(DF64, half, x, nrhs=MANY)
        out = [torch.zeros(x.numel() + 1, dtype=torch.float64, device="cuda")[offset:][:x.numel()] for _ in range(2)]
        assert out[0].data_ptr() % 16 == 8 * offset
        lat.unpack_half(DF64, out[0], half, nrhs=MANY)
        for k in range(0, MANY, 110):
            lat.unpack_half(DF64, out[1][k * 24 * lat.h:(k + 110) * 24 * lat.h], half[k:k + 110], nrhs=110)
        assert torch.equal(out[0], out[1])
        hi = x.float()
        kept = hi.double() + (x - hi.double()).float().double()  # (hi, lo) in FP32
        assert torch.equal(out[0].view_as(x), kept)
