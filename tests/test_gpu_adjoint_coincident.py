"""Receivers of the adjoint close enough to the source that each of them moves the
gradient: several at one point (their residuals add up, as in the misfit), and blocks
of them across tile and z-chunk seams and in the domain's corners."""
import functools

import numpy as np
import pytest

import oracle
from paper_2009_04619_gb300 import seisgb, synth
from gpu_util import ensure_lib, rel_l2

pytestmark = pytest.mark.gpu

NX, NY, NZ, NB, NT = 126, 30, 40, 4, 16  # computed 134 x 38 x 48: seams at x 64, 128 (and 32, 96), y 16, 32
BOUND = 1e-3  # relative gradient error, as in the other adjoint tests


@functools.lru_cache(maxsize=None)
def _shot(src):
    shape, v = (NZ + 2 * NB, NY + 2 * NB, NX + 2 * NB), 2500.0
    vel = synth.layered_model(shape, seed=4, vmin=1800, vmax=2400, perturb=0.03)
    dt = float(np.float32(0.4 * oracle.cfl_dt(v, 10, 10, 10)))
    wav = synth.ricker(NT, dt, 60.0, t0=0.004)
    go = oracle.Grid(NX, NY, NZ, NB, 10.0, 10.0, 10.0, dt, vmax=v, r0=float(np.float32(1e-3)))
    return go, vel, dt, wav


def _reference(src, rec, obs):
    go, vel, dt, wav = _shot(src)
    return oracle.adjoint_shot(go, vel, wav, NT, src, rec, obs.astype(np.float64))


def _observed(src, rec):
    """Samples of the traces' own size at each receiver."""
    go, vel, dt, wav = _shot(src)
    tr = oracle.run_shot(go, vel, wav, NT, src, rec, want_state=False)["traces"]
    noise = np.random.default_rng(5).standard_normal(tr.shape)
    return (noise * np.abs(tr).max(axis=0)).astype(np.float32)


def _check(src, rec, obs, ref):
    ensure_lib()
    go, vel, dt, wav = _shot(src)
    J_ref, grad_ref = ref
    g = seisgb.make_grid(NX, NY, NZ, NB, 10.0, 10.0, 10.0, dt, 2500.0)
    grad = np.zeros(vel.shape)
    J = seisgb.adjoint_shot(g, vel, wav, NT, src, rec, obs, grad, ckpt_every=6)
    assert abs(J - J_ref) <= 1e-4 * J_ref and rel_l2(grad, grad_ref) <= BOUND
    return grad


def _block(src):
    """All points up to two away from the source along each axis."""
    d = range(-2, 3)
    return np.array([(src[0] + a, src[1] + b, src[2] + c) for c in d for b in d for a in d], np.int32)


def _counts(src, rec, obs, ref, keep):
    """Whether the oracle's gradient without the receivers not kept is far outside the bound."""
    _, part = _reference(src, rec[keep], np.ascontiguousarray(obs[:, keep]))
    return rel_l2(part, ref[1]) >= 5 * BOUND


LO, HI = NB + 2, (NB + NX - 3, NB + NY - 3, NB + NZ - 3)
SOURCES = {"xy-seams": (64, 16, 20), "high-seams": (127, 31, 24), "low-corner": (LO, LO, LO), "high-corner": HI}


@pytest.mark.parametrize("where", list(SOURCES))
def test_receivers_across_seams(where):
    src = SOURCES[where]
    rec = _block(src)
    obs = _observed(src, rec)
    ref = _reference(src, rec, obs)
    for axis in range(3):  # no plane of the block may be missed
        for at in range(src[axis] - 2, src[axis] + 3):
            assert _counts(src, rec, obs, ref, rec[:, axis] != at)
    _check(src, rec, obs, ref)


@pytest.mark.parametrize("spread", [False, True], ids=["together", "apart"])
def test_coincident_receivers_add_up(spread):
    """One, two and three receivers at a point, listed one after the other, or all points
    once and then again."""
    src = (64, 16, 20)
    rec = _block(src)
    times = 1 + np.arange(len(rec)) % 3
    if spread:
        rec = np.concatenate([rec[times > q] for q in (2, 0, 1)] + [_block((64, 16, 21))])
    else:
        rec = np.repeat(rec, times, axis=0)
    obs = _observed(src, rec)
    ref = _reference(src, rec, obs)
    first = np.sort(np.unique(rec, axis=0, return_index=True)[1])
    last = np.sort(len(rec) - 1 - np.unique(rec[::-1], axis=0, return_index=True)[1])
    for one in (first, last):  # one receiver per point alone is not enough
        assert len(one) < len(rec) and _counts(src, rec, obs, ref, one)
    grad = _check(src, rec, obs, ref)
    assert np.array_equal(grad, _check(src, rec, obs, ref))  # the same bits every time
