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
