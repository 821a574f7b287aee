"""State in and out through host memory, from and to every layout, bit for bit: where there is no device memory
for a staging buffer, and of swarms small enough for one copy."""
import numpy as np
import pytest

from tests.gpu_common import BOUNDS, C12, W, load_cupso

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,D,kernel,dtype", [(1, 1, "auto", "f32"), (129, 7, "auto", "f32"), (5000, 33, "pipelined3", "f32"),
                                              (3001, 64, "panel8", "f32"), (3001, 64, "panel16", "f32"),
                                              (1000, 33, "auto", "f64")])
def test_state_round_trip_without_staging(N, D, kernel, dtype):
    P = load_cupso()
    rng = np.random.default_rng(N + D)
    dt = np.float32 if dtype == "f32" else np.float64
    arrays = [rng.uniform(-100, 100, (N, D)).astype(dt) for _ in range(3)] + [rng.standard_normal(N).astype(dt)]
    names = ("pos", "v", "pbest_pos", "pbest_fit")

    def run(staging):
        with P.Swarm(D, N, BOUNDS[0], W, C12, C12, 0, 1, mode="sync", dtype=dtype) as s:
            s.set_option(P.CUPSO_OPT_SYNC_KERNEL, P.SYNC_KERNELS[kernel])
            s.set_option(P.CUPSO_OPT_FAULT_NO_STAGING, 0 if staging else 1)
            s.set_state(*arrays, t=5)
            loaded = s.state()
            s.step(2)
            return loaded, s.state(), s.gbest()

    loaded, after, best = run(False)
    for name, a in zip(names, arrays):
        assert loaded[name].tobytes() == a.tobytes(), name
    _, after1, best1 = run(True)
    for name in names:
        assert after[name].tobytes() == after1[name].tobytes(), name
    assert best[:3] == best1[:3] and best[3].tobytes() == best1[3].tobytes()


# either side of 10000 values and of 512 KB with the padding
@pytest.mark.parametrize("N,D,kernel", [(1, 2, "auto"), (1, 340, "auto"), (1, 342, "auto"), (77, 129, "auto"), (78, 129, "auto"),
                                        (150, 64, "panel8"), (150, 64, "panel16"), (156, 64, "panel16"), (300, 33, "pipelined3")])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_small_states(N, D, kernel, dtype):
    P = load_cupso()
    rng = np.random.default_rng(N + D)
    dt = np.float32 if dtype == "f32" else np.float64
    arrays = [rng.uniform(-100, 100, (N, D)).astype(dt) for _ in range(3)] + [rng.standard_normal(N).astype(dt)]
    with P.Swarm(D, N, BOUNDS[0], W, C12, C12, 0, 1, mode="sync", dtype=dtype) as s:
        s.set_option(P.CUPSO_OPT_SYNC_KERNEL, P.SYNC_KERNELS[kernel])
        s.set_state(*arrays, t=5)
        st = s.state()
        for name, a in zip(("pos", "v", "pbest_pos", "pbest_fit"), arrays):
            assert st[name].tobytes() == a.tobytes(), name
        if dtype == "f32":   # only one of the arrays
            pf = np.empty(N, np.float32)
            assert P.lib().cupso_get_state(s.h, None, None, None, P._f32p(pf), None) == P.CUPSO_OK
            assert pf.tobytes() == arrays[3].tobytes()
