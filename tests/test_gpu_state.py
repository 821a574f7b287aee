"""State in and out (cupso_set_state / cupso_get_state) bit for bit through every device
layout: ragged particle counts and dimensions, both panel widths, both precisions,
a state larger than one staging chunk; the gbest found from it."""
import numpy as np
import pytest

from tests.gpu_common import BOUNDS, C12, W, load_cupso

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    return load_cupso()


def _arrays(N, D, dtype, seed=0):
    rng = np.random.default_rng(seed + N + D)
    pos, v, pb = (rng.uniform(-100, 100, (N, D)).astype(dtype) for _ in range(3))
    pf = rng.standard_normal(N).astype(dtype)
    pf[rng.integers(0, N)] = pf.min()      # maybe a tie: the lowest index wins
    return pos, v, pb, pf


@pytest.mark.parametrize("N,D,kernel", [(1, 1, "auto"), (129, 1, "auto"), (5000, 7, "pipelined3"), (33, 33, "tiled"),
                                        (3001, 64, "panel8"), (3001, 64, "panel16"), (1025, 24, "panel8"),
                                        (70001, 128, "auto"), (70001, 129, "auto")])
def test_state_round_trip_fp32(P, N, D, kernel):
    arrays = _arrays(N, D, np.float32)
    with P.Swarm(D, N, BOUNDS[0], W, C12, C12, 0, 1, mode="sync") as s:
        s.set_option(P.CUPSO_OPT_SYNC_KERNEL, P.SYNC_KERNELS[kernel])
        for k in range(2):                  # the second time over a stepped swarm, from its own layout
            s.set_state(*arrays, t=5 + k)
            _, fit, idx, pos = s.gbest()
            st = s.state()
            assert st["t"] == 5 + k
            for name, a in zip(("pos", "v", "pbest_pos", "pbest_fit"), arrays):
                np.testing.assert_array_equal(st[name].view(np.uint32), a.view(np.uint32), err_msg=name)
            assert (idx, fit) == (int(np.argmin(arrays[3])), arrays[3].min())
            np.testing.assert_array_equal(pos, arrays[2][idx])
            s.step(2)


@pytest.mark.parametrize("N,D", [(1, 1), (130, 1), (129, 3), (1000, 33), (33001, 130)])
def test_state_round_trip_fp64(P, N, D):
    arrays = _arrays(N, D, np.float64)
    with P.Swarm(D, N, BOUNDS[0], W, C12, C12, 0, 1, mode="sync", dtype="f64") as s:
        s.set_state(*arrays, t=5)
        _, fit, idx, pos = s.gbest()
        st = s.state()
        for name, a in zip(("pos", "v", "pbest_pos", "pbest_fit"), arrays):
            np.testing.assert_array_equal(st[name].view(np.uint64), a.view(np.uint64), err_msg=name)
        assert (idx, fit) == (int(np.argmin(arrays[3])), arrays[3].min())
        np.testing.assert_array_equal(pos, arrays[2][idx])


def test_state_loaded_for_one_mode_steps_in_another(P):
    """Loaded in panels, then stepped by a dimension-major mode, and back: as the oracle."""
    from tests.gpu_common import assert_state_equal, oracle_swarm
    N, D, fid = 2500, 64, 1
    ref = oracle_swarm(fid, N, D, 9).init().step_sync(3)
    with P.Swarm(D, N, BOUNDS[fid], W, C12, C12, fid, 9, mode="sync") as s:
        s.set_option(P.CUPSO_OPT_SYNC_KERNEL, P.SYNC_KERNELS["panel8"])
        s.set_state(ref.pos, ref.v, ref.pbest_pos, ref.pbest_fit, t=3)
        s.set_mode("tree")
        s.step(2)
        s.set_mode("sync")
        s.step(3)
        assert_state_equal(s.state(), ref.step_sync(5))
