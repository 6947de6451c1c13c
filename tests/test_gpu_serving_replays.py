"""Which replays of a server run as a CUDA graph: a shot of a few replays is enqueued
launch by launch, and a composition that outlives its first batch (at most four
replays) is captured, also while slots are free; the traces are the same bits."""
import numpy as np
import pytest

from paper_2009_04619_gb300 import seisgb, synth
from gpu_util import ensure_lib

pytestmark = pytest.mark.gpu

S = 16


@pytest.mark.parametrize("nt,shots", [(60, 1), (60, 3), (600, 1), (600, 3)])
def test_a_lasting_composition_is_captured(nt, shots):
    ensure_lib()
    n, nb = 112, 8  # 128^3: a step takes the GPU longer than its launch the host
    vel = synth.layered_model((128,) * 3, seed=2)
    g0 = seisgb.make_grid(n, n, n, nb, 10.0, 10.0, 10.0, 1.0, float(vel.max()))
    dt = 0.4 * seisgb.cfl_dt(g0, float(vel.max()))
    g = seisgb.make_grid(n, n, n, nb, 10.0, 10.0, 10.0, dt, float(vel.max()))
    wav, src, rec = synth.ricker(nt, dt, 20.0), (64, 64, nb + 2), [(60 + q, 64, nb) for q in range(9)]
    want = np.zeros((nt, len(rec)), np.float32)
    seisgb.run_shot(g, vel, wav, nt, src, rec, want)
    with seisgb.Server(8 << 30, max_slots=8, steps_per_graph=S) as sv:
        tickets = [sv.submit(g, vel, wav, nt, src, rec) for _ in range(shots)]
        for t in tickets:
            code, _, got = sv.poll(t, nt, len(rec), timeout_us=60_000_000)
            assert code == seisgb.OK and np.array_equal(got, want)
        st = sv.stats()
    replays, graphs = st.step_launches // S, st.graph_replays
    if nt == 60:  # four replays or fewer from the first admission to each change
        assert graphs == 0
    else:  # the batches after each admission, and the last replays before a shot ends
        assert replays >= (nt + 1) // S and 0 < graphs <= replays - 1
        assert replays - graphs <= shots * (4 + 8)
