"""Residuals enter the adjoint step at the receivers its work unit holds: receivers on
both sides of tile and z-chunk seams and of the domain's corners, one receiver alone
(every other unit has none), and more receivers in one unit than it has threads."""
import numpy as np
import pytest

import oracle
from paper_2009_04619_gb300 import seisgb, synth
from gpu_util import ensure_lib, rel_l2

pytestmark = pytest.mark.gpu

NX, NY, NZ, NB = 126, 30, 40, 4  # computed 134 x 38 x 48: 3 x 3 tiles, several z-chunks


def _receivers(kind):
    lo = NB
    hi = (NB + NX - 1, NB + NY - 1, NB + NZ - 1)
    if kind == "one":
        return np.array([[64, 16, 20]], np.int32)
    if kind == "seams":
        return np.array([(i, j, k) for i in (lo, 63, 64, 127, 128, hi[0]) for j in (lo, 15, 16, 31, 32, hi[1])
                         for k in range(lo, hi[2] + 1, 1)], np.int32)
    return np.array([(i, j, 9) for j in range(lo, hi[1] + 1) for i in range(lo, hi[0] + 1)], np.int32)


@pytest.mark.parametrize("kind", ["one", "seams", "dense"])
def test_receivers_of_every_unit_count(kind):
    """A receiver that a unit missed or took twice changes the residual energy by 1/nrec,
    so the gradient by about 1/sqrt(nrec) >= 1.6e-2; the fp32 run is within 1e-3 of
    the fp64 oracle (the bound of the other adjoint tests)."""
    ensure_lib()
    shape, nt, v = (NZ + 2 * NB, NY + 2 * NB, NX + 2 * NB), 12, 2500.0
    vel = synth.layered_model(shape, seed=4, vmin=1800, vmax=2400, perturb=0.03)
    dt = float(np.float32(0.4 * oracle.cfl_dt(v, 10, 10, 10)))
    wav, src, rec = synth.ricker(nt, dt, 60.0, t0=0.004), (66, 18, 14), _receivers(kind)
    obs = np.random.default_rng(5).standard_normal((nt, len(rec))).astype(np.float32)
    go = oracle.Grid(NX, NY, NZ, NB, 10.0, 10.0, 10.0, dt, vmax=v, r0=float(np.float32(1e-3)))
    # observed samples of the traces' own size
    obs *= float(np.abs(oracle.run_shot(go, vel, wav, nt, src, rec, want_state=False)["traces"]).max())
    J_ref, grad_ref = oracle.adjoint_shot(go, vel, wav, nt, src, rec, obs.astype(np.float64))
    g = seisgb.make_grid(NX, NY, NZ, NB, 10.0, 10.0, 10.0, dt, v)
    grad = np.zeros(shape)
    J = seisgb.adjoint_shot(g, vel, wav, nt, src, rec, obs, grad, ckpt_every=5)
    assert abs(J - J_ref) <= 1e-4 * J_ref and rel_l2(grad, grad_ref) <= 1e-3
