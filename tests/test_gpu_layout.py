"""Layout conversion (sgb_pack / sgb_unpack) against plain PyTorch indexing: rows that
move as quads and rows that cannot (odd extents, arrays that start off a 16-byte
boundary), planes shorter and longer than one block's items, and halo zeros; and the
model range check that rides on the conversion of the velocity."""
import numpy as np
import pytest
import torch

from paper_2009_04619_gb300 import seisgb, synth
from gpu_util import ensure_lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("ext", [(1, 1, 1, 0), (4, 3, 2, 0), (61, 5, 3, 1), (64, 37, 5, 4), (301, 23, 4, 2)])
def test_pack_unpack_values(ext, shift):
    nx, ny, nz, nb = ext
    g = seisgb.make_grid(nx, ny, nz, nb, 10.0, 10.0, 10.0, 1e-4, 2000.0)
    Nz, Ny, Nx = g.shape
    L = seisgb.layout(g)
    torch.manual_seed(nx)
    n = Nx * Ny * Nz
    src = torch.randn(n + shift, device="cuda")[shift:]  # shift 1: not 16-byte aligned
    dst = torch.full((int(L.elems) + shift,), 7.0, device="cuda")[shift:]
    seisgb.pack(g, src, dst)
    want = torch.zeros(L.sz, L.sy, L.sx, device="cuda")
    want[4:4 + Nz, 4:4 + Ny, 8:8 + Nx] = src.view(Nz, Ny, Nx)
    assert torch.equal(dst, want.reshape(-1))
    back = torch.full((n + shift,), -1.0, device="cuda")[shift:]
    seisgb.unpack(g, dst, back)
    assert torch.equal(back, src)


@pytest.mark.parametrize("bad", [0.0, -1500.0, float("nan"), float("inf")])
@pytest.mark.parametrize("nx", [24, 25])
def test_one_bad_velocity_is_found(nx, bad):
    """A single bad point, in the last place of the model, is rejected; a model at its
    own CFL limit is not, and one point above it is."""
    vel = synth.constant_model((21, 22, nx), 2000.0)
    g0 = seisgb.make_grid(nx, 22, 21, 0, 10.0, 10.0, 10.0, 1.0, 2000.0)
    g = seisgb.make_grid(nx, 22, 21, 0, 10.0, 10.0, 10.0, 0.9 * seisgb.cfl_dt(g0, 2000.0), 2000.0)
    tr, w = np.zeros((2, 1), np.float32), np.ones(2, np.float32)
    args = (w, 2, (3, 3, 3), [(4, 4, 4)], tr)
    seisgb.run_shot(g, vel, *args)
    for v, code in ((bad, seisgb.ERR_INVALID_ARG), (2500.0, seisgb.ERR_UNSTABLE_DT)):
        vel[-1, -1, -1] = v
        with pytest.raises(seisgb.SeisgbError) as e:
            seisgb.run_shot(g, vel, *args)
        assert e.value.code == code
