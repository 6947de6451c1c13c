"""Grids whose steps run in 32 x 32 tiles (extents that 64 x 16 tiles cover badly: just
past a multiple of 64 in x, so the plan takes the square ones): every kernel of that
shape -- one step per storage format, a served shot, the adjoint -- under the bounds of
the other parity tests."""
import numpy as np
import pytest
import torch

import oracle
import test_gpu_adjoint_receivers as receivers
import test_gpu_diff as diff
import test_gpu_parity as parity
from paper_2009_04619_gb300 import seisgb, synth
from gpu_util import abs_term_sum, ensure_lib, from_padded, rel_l2, to_padded

pytestmark = pytest.mark.gpu

# inner extents, PML, spacing: computed 137 x 130 x 60, 65 x 97 x 120 (zero walls), 160 x 97 x 60
CASES = [(121, 114, 44, 8, (10.0, 11.0, 12.0)), (65, 97, 120, 0, (7.0, 7.0, 7.0)),
         (128, 65, 28, 16, (10.0, 10.0, 10.0))]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


@pytest.mark.parametrize("case", CASES)
def test_single_step(case):
    parity.test_single_step_random_fields(case)


@pytest.mark.parametrize("bf16", [False, True], ids=["fp32", "bf16"])
@pytest.mark.parametrize("case", CASES)
def test_single_step_difference_form(case, bf16):
    nx, ny, nz, nb, h = case
    diff.test_stencil_step_diff_vs_oracle((*case, (nx // 2, ny - 4, 5)), bf16)


@pytest.mark.parametrize("fmt", ["fp16", "bf16"])
@pytest.mark.parametrize("case", CASES)
def test_single_step_16bit(case, fmt):
    """Each stored value is one of the two 16-bit neighbours of the oracle's, give or
    take the fp32 evaluation's 1e-6 S."""
    nx, ny, nz, nb, h = case
    t, p, storage = ((torch.float16, 10, seisgb.FP16_SCALED) if fmt == "fp16"
                     else (torch.bfloat16, 7, seisgb.BF16))
    g32, go = parity._grid_pair(nx, ny, nz, nb, h)
    g = seisgb.make_grid(nx, ny, nz, nb, *h, go.dt, 3000.0, 1e-3, storage)
    rng = np.random.default_rng(nx + ny)
    uc, up = (torch.from_numpy(rng.standard_normal(g.shape).astype(np.float32)).to(t).float().numpy()
              for _ in range(2))
    ph = np.zeros(g.shape, np.float32)
    m = ((rng.uniform(1500, 3000, g.shape) * go.dt) ** 2).astype(np.float32)
    d_uc, d_up = to_padded(g32, uc).to(t), to_padded(g32, up).to(t)
    scale = torch.tensor([1.0] * 4 + [float(np.abs(uc).max()), 0.0, 0.0, float(np.abs(up).max())],
                         device="cuda")
    seisgb.stencil_step(g, d_uc, d_up, to_padded(g32, m), to_padded(g32, ph), 0,
                        scale_state=scale if fmt == "fp16" else None)
    seisgb.device_status()
    s = float(scale[1]) if fmt == "fp16" else 1.0
    un = from_padded(g32, d_up.float()) * np.float32(s)
    ref, _ = oracle.step(go, m, up, uc, ph)
    S = abs_term_sum(go, m, up, uc, ph)
    bound = 1.01e-6 * S + 2.0 ** -p * (np.abs(ref) + 1e-6 * S) + 2.0 ** -24 * s
    err = np.abs(un - ref)
    assert np.all(err <= bound), float((err / bound).max())


def test_served_shot():
    nx, ny, nz, nb, nt = 121, 114, 44, 8, 40
    shape = (nz + 2 * nb, ny + 2 * nb, nx + 2 * nb)
    vel = synth.layered_model(shape, seed=3, sigma=2.0)
    dt = float(np.float32(0.4 * oracle.cfl_dt(float(vel.max()), 10, 10, 10)))
    g = seisgb.make_grid(nx, ny, nz, nb, 10.0, 10.0, 10.0, dt, float(vel.max()))
    wav, src = synth.ricker(nt, dt, 40.0, t0=0.01), (nb + 60, nb + 50, nb + 20)
    rec = np.array([(nb + 60 + q, nb + 50 - q, nb + 20 + q % 7) for q in range(-30, 31, 3)], np.int32)
    tr = np.zeros((nt, len(rec)), np.float32)
    seisgb.run_shot(g, vel, wav, nt, src, rec, tr)
    go = oracle.Grid(nx, ny, nz, nb, 10.0, 10.0, 10.0, dt, vmax=float(vel.max()), r0=float(np.float32(1e-3)))
    ref = oracle.run_shot(go, vel, wav, nt, src, rec, want_state=False)["traces"]
    assert rel_l2(tr, ref) <= 2e-5
    with seisgb.Server(2 << 30, max_slots=2) as sv:
        tickets = [sv.submit(g, vel, wav, nt, src, rec) for _ in range(2)]
        for t in tickets:
            code, _, got = sv.poll(t, nt, len(rec), timeout_us=30_000_000)
            assert code == seisgb.OK and np.array_equal(got, tr)


@pytest.mark.parametrize("kind", ["seams", "dense"])
def test_adjoint_receivers(kind, monkeypatch):
    for name, v in zip(("NX", "NY", "NZ", "NB"), (121, 114, 44, 8)):
        monkeypatch.setattr(receivers, name, v)
    receivers.test_receivers_of_every_unit_count(kind)
