"""cupso_get_gbest: the current parity's key, position and status out of the arena's head, with and
without the position, positions short and long (read apart), both precisions."""
import ctypes as C

import numpy as np
import pytest

from tests.gpu_common import BOUNDS, C12, W, load_cupso

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("N,D", [(5, 1), (300, 7), (3, 8192), (3, 8193), (3, 16384), (3, 16385), (2, 40001)])
def test_gbest_is_the_best_pbest(dtype, N, D):
    P = load_cupso()
    rng = np.random.default_rng(D)
    dt = np.float32 if dtype == "f32" else np.float64
    with P.Swarm(D, N, BOUNDS[0], W, C12, C12, 0, 5, mode="tree", dtype=dtype) as s:
        for t in range(4):   # both parities, loaded and (t = 3, where a kernel takes these dimensions) stepped to
            if t == 3 and D <= 8192:
                s.step(1)
                st = s.state()
                pb, pf = st["pbest_pos"], st["pbest_fit"]
            else:
                pos0, v0, pb = (rng.uniform(-100, 100, (N, D)).astype(dt) for _ in range(3))
                pf = rng.standard_normal(N).astype(dt)
                s.set_state(pos0, v0, pb, pf, t)
            rc, fit, idx, pos = s.gbest()
            best = int(np.argmin(pf))
            assert (rc, idx, fit) == (P.CUPSO_OK, best, pf[best])
            np.testing.assert_array_equal(pos, pb[best])
            alone = C.c_int64()
            get = P.lib().cupso_get_gbest_fp64 if dtype == "f64" else P.lib().cupso_get_gbest
            assert get(s.h, None, None, C.byref(alone)) == P.CUPSO_OK and alone.value == best


@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_gbest_reports_the_sticky_status(dtype):
    P = load_cupso()
    dt = np.float32 if dtype == "f32" else np.float64
    with P.Swarm(4, 100, BOUNDS[0], W, C12, C12, 0, 5, mode="tree", dtype=dtype) as s:
        a = np.ones((100, 4), dt)
        fit = np.ones(100, dt)
        fit[7] = np.nan
        s.set_state(a, a, a, fit, t=4)
        s.step(1)
        assert s.gbest()[0] == P.CUPSO_ERR_NAN
        s.set_option(P.CUPSO_OPT_CLEAR_STATUS, 1)
        assert s.gbest()[0] == P.CUPSO_OK
