"""The bounded waits of the double-precision one-launch steps, and the status they leave."""
import pytest

from tests.gpu_common import load_cupso

pytestmark = pytest.mark.gpu

BOX = (-100.0, 100.0, 20.0)


@pytest.fixture(scope="module")
def P():
    return load_cupso()


@pytest.mark.parametrize("mode", ["sync", "persistent", "auto", "queue_lock"])
def test_status_of_a_double_precision_swarm_can_be_cleared(P, mode):
    with P.Swarm(7, 500, BOX, 1.0, 2.0, 2.0, 0, 5, mode=mode, dtype="f64") as s:
        s.step(6)
        s.set_option(P.CUPSO_OPT_CLEAR_STATUS, 1)
        s.step(6)
        assert s.gbest()[0] == P.CUPSO_OK


# in registers; in memory, Rosenbrock with its second term array
@pytest.mark.parametrize("mode,fid,N,D", [("sync", 0, 500, 7), ("persistent", 4, 2000, 1), ("sync", 3, 20000, 120)])
def test_barrier_wait_expires_and_reports(P, mode, fid, N, D):
    """A barrier that waits for one CTA more than there are: the wait ends at its limit, the status is
    reported, and the swarm steps again once it is cleared."""
    with P.Swarm(D, N, BOX, 1.0, 2.0, 2.0, fid, 7, mode=mode, dtype="f64") as s:
        s.set_option(P.CUPSO_OPT_WAIT_LIMIT_NS, 50_000_000)
        s.set_option(P.CUPSO_OPT_FAULT_STALL_BARRIER, 1)
        s.step(6)
        assert s.gbest()[0] == P.CUPSO_ERR_DEVICE_TIMEOUT
        s.set_option(P.CUPSO_OPT_FAULT_STALL_BARRIER, 0)
        s.set_option(P.CUPSO_OPT_CLEAR_STATUS, 1)
        s.step(6)
        assert s.gbest()[0] == P.CUPSO_OK
