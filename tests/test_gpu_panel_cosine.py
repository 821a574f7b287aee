"""The panel kernel's two forms of cos 2 pi x: bounds up to 2^21 take the one that rounds by
an addition, bounds beyond take the general one; both bit for bit against the oracle."""
import pytest

from tests.gpu_common import C12, W, assert_state_equal, load_cupso, oracle_swarm, same_bits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", ["panel8", "panel16"])
@pytest.mark.parametrize("limit", [2.0 ** 21, 2.0 ** 21 + 0.25, 3e6])
@pytest.mark.parametrize("fid", [1, 2])
def test_cosine_limit_matches_oracle(fid, limit, kernel):
    P = load_cupso()
    bounds, N, D, T = (-limit, limit, 0.1 * limit), 1500, 64, 6
    with P.Swarm(D, N, bounds, W, C12, C12, fid, 3) as s:
        s.set_mode("sync")
        s.set_option(P.CUPSO_OPT_SYNC_KERNEL, P.SYNC_KERNELS[kernel])
        assert s.info()["sync_panel"] == int(kernel[5:])
        s.step(T)
        st = s.state()
        _, fit, idx, pos = s.gbest()
    ref = oracle_swarm(fid, N, D, 3, bounds=bounds).init().step_sync(T)
    assert_state_equal(st, ref)
    assert idx == ref.gbest_idx and same_bits(pos, ref.gbest_pos)
