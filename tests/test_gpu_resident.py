"""The resident SYNC kernel (several iterations of a cupso_step call with the swarm in
registers) bit for bit against the oracle: every fitness, 1 to 8 items per thread, odd
dimensions, one particle per CTA, a ragged last CTA, the sizes at its limits, and
the state handed over from and to the other kernels and layouts."""
import numpy as np
import pytest

from tests.gpu_common import BOUNDS, C12, W, assert_state_equal, load_cupso, oracle_swarm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    return load_cupso()


def _swarm(P, fid, N, D, seed):
    return P.Swarm(D, N, BOUNDS[fid], W, C12, C12, fid, seed, mode="sync")


def _check(s, ref):
    _, fit, idx, pos = s.gbest()
    assert_state_equal(s.state(), ref)
    assert idx == ref.gbest_idx and fit == ref.gbest_fit
    np.testing.assert_array_equal(pos, ref.gbest_pos)


@pytest.mark.parametrize("fid", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("N,D", [(1, 1), (150, 2), (153, 7), (4001, 30), (20011, 30), (77824, 1)])
def test_resident_trajectory(P, fid, N, D):
    ref = oracle_swarm(fid, N, D, 3).init()
    with _swarm(P, fid, N, D, 3) as s:
        s.step(2)
        s.step(9)
        _check(s, ref.step_sync(11))


@pytest.mark.parametrize("fid,N,D", [(1, 77824, 16), (3, 77825, 16), (3, 304, 4095), (0, 1216, 1024), (2, 40000, 17)])
def test_resident_at_its_limits(P, fid, N, D):
    ref = oracle_swarm(fid, N, D, 5).init()
    with _swarm(P, fid, N, D, 5) as s:
        s.step(4)
        _check(s, ref.step_sync(4))


@pytest.mark.parametrize("kernel", ["auto", "panel8", "panel16", "pipelined3", "tiled"])
def test_resident_takes_over_and_hands_back(P, kernel):
    """Single steps of another kernel (pending pbest rows, its layout), a resident launch, single steps again."""
    fid, N, D = 1, 5000, 64
    ref = oracle_swarm(fid, N, D, 11).init()
    with _swarm(P, fid, N, D, 11) as s:
        for n in (1, 5, 1, 1, 3):
            s.set_option(P.CUPSO_OPT_SYNC_KERNEL, P.SYNC_KERNELS["auto" if n > 1 else kernel])
            s.step(n)
        _check(s, ref.step_sync(11))
        s.set_option(P.CUPSO_OPT_ITERS_PER_LAUNCH, 3)
        s.step(7)
        s.set_mode("tree")
        s.step(2)
        s.set_mode("sync")
        s.set_option(P.CUPSO_OPT_ITERS_PER_LAUNCH, 1)
        s.step(2)
        _check(s, ref.step_sync(11))


def test_resident_barrier_wait_expires_and_reports(P):
    """A barrier that waits for one CTA more than there are: the wait ends at its limit, the
    status is reported, and the swarm steps again once it is cleared."""
    with _swarm(P, 3, 5000, 30, 7) as s:
        s.set_option(P.CUPSO_OPT_WAIT_LIMIT_NS, 50_000_000)
        s.set_option(P.CUPSO_OPT_FAULT_STALL_BARRIER, 1)
        s.step(3)
        assert s.gbest()[0] == P.CUPSO_ERR_DEVICE_TIMEOUT
        s.set_option(P.CUPSO_OPT_FAULT_STALL_BARRIER, 0)
        s.set_option(P.CUPSO_OPT_CLEAR_STATUS, 1)
        s.step(4)
        assert s.gbest()[0] == P.CUPSO_OK
