"""serve_submit's model check: one bad value in the first, a middle or the last place
(models of whole blocks of 1024 values, and with a remainder) is refused, denormal and
huge positive values are not bad by themselves, and the CFL limit uses the maximum."""
import numpy as np
import pytest

from paper_2009_04619_gb300 import seisgb
from gpu_util import ensure_lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(16, 16, 16), (15, 17, 19)])
def test_submit_checks_every_value(shape):
    ensure_lib()
    nz, ny, nx = shape
    g0 = seisgb.make_grid(nx, ny, nz, 0, 10.0, 10.0, 10.0, 1.0, 3000.0)
    g = seisgb.make_grid(nx, ny, nz, 0, 10.0, 10.0, 10.0, 0.9 * seisgb.cfl_dt(g0, 3000.0), 3000.0)
    w, rec, n = np.ones(2, np.float32), [(4, 4, 4)], nx * ny * nz
    with seisgb.Server(1 << 30, max_slots=2) as sv:
        def submit(at, value):
            vel = np.full(shape, 3000.0, np.float32)
            vel.reshape(-1)[at] = value
            return sv.submit(g, vel, w, 2, (3, 3, 3), rec)

        for at in (0, 1023, n // 2, n - 1):
            for bad in (0.0, -0.0, -1.0, np.nan, -np.nan, np.inf, -np.inf):
                with pytest.raises(seisgb.SeisgbError) as e:
                    submit(at, bad)
                assert e.value.code == seisgb.ERR_INVALID_ARG
            with pytest.raises(seisgb.SeisgbError) as e:
                submit(at, 3400.0)
            assert e.value.code == seisgb.ERR_UNSTABLE_DT
            t = submit(at, 1e-39)
            assert sv.poll(t, 2, 1, timeout_us=10_000_000)[0] == seisgb.OK
