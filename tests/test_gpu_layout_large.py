"""Layout conversion of planes of more than 2^32 points (which no 32-bit count holds):
every point of the plane is converted and the halo is zero."""
import pytest
import torch

from paper_2009_04619_gb300 import seisgb
from gpu_util import ensure_lib

pytestmark = pytest.mark.gpu


def _values(row0, rows, nx):
    """Distinct fp32 integers that differ between points 2^32 apart."""
    p = torch.arange(row0 * nx, (row0 + rows) * nx, device="cuda")
    return (((p * 2654435761) >> 9) & 0xFFFFFF).float().view(rows, nx)


def test_planes_above_32_bits():
    ensure_lib()
    nx = ny = 65537  # an odd row length: converted point by point
    g = seisgb.make_grid(nx, ny, 1, 0, 10.0, 10.0, 10.0, 1e-4, 2000.0)
    L = seisgb.layout(g)
    assert nx * ny > 2 ** 32 and int(L.stride_z) > 2 ** 32
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 4 * int(L.elems) + 4 * nx * ny + (8 << 30):
        pytest.skip("needs 180 GB of device memory")
    step = 1024
    src = torch.empty(ny, nx, device="cuda")
    padded = torch.full((int(L.elems),), 7.0, device="cuda")
    for r in range(0, ny, step):
        n = min(step, ny - r)
        src[r:r + n] = _values(r, n, nx)
    seisgb.pack(g, src, padded)
    planes = padded.view(int(L.sz), int(L.sy), int(L.sx))
    for k in range(int(L.sz)):
        for r in range(0, int(L.sy), step):
            got = planes[k, r:r + step]
            if k != 4:
                assert not bool(got.any())
                continue
            want = torch.zeros_like(got)
            lo, hi = max(r, 4), min(r + got.shape[0], 4 + ny)
            want[lo - r:hi - r, 8:8 + nx] = _values(lo - 4, hi - lo, nx)
            assert torch.equal(got, want)
    src.fill_(-1.0)
    seisgb.unpack(g, padded, src)
    for r in range(0, ny, step):
        n = min(step, ny - r)
        assert torch.equal(src[r:r + n], _values(r, n, nx))
    del src, padded, planes
    torch.cuda.empty_cache()
