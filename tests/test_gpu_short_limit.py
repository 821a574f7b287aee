"""A wait limit shorter than an iteration, set for another mode's waits: swarms of SYNC and AUTO calls, which have
steps without waits between CTAs, report no timeout and get the same bits."""
import pytest

from tests.gpu_common import C12, W, load_cupso

pytestmark = pytest.mark.gpu

BOX = (-30.0, 30.0, 6.0)


@pytest.mark.parametrize("mode,dtype,N,D,limit", [("auto", "f32", 1024, 32, 1000), ("sync", "f32", 20011, 30, 1000),
                                                  ("auto", "f64", 2000, 4, 1000), ("sync", "f64", 16384, 120, 20_000)])
def test_no_timeout_where_no_wait_was(mode, dtype, N, D, limit):
    P = load_cupso()
    runs = []
    for ns in (limit, 2_000_000_000):
        with P.Swarm(D, N, BOX, W, C12, C12, 3, 7, mode=mode, dtype=dtype) as s:
            s.set_option(P.CUPSO_OPT_WAIT_LIMIT_NS, ns)
            s.step(60)
            runs.append((s.gbest(), s.state()))
            assert runs[-1][0][0] == P.CUPSO_OK
            assert (s.info()["one_launch_iters"] > 0) == (ns > limit)
    (g0, s0), (g1, s1) = runs
    assert g0[:3] == g1[:3] and g0[0] == P.CUPSO_OK
    for name in ("pos", "v", "pbest_pos", "pbest_fit"):
        assert s0[name].tobytes() == s1[name].tobytes(), name
