"""Units handed out CTA by CTA: particle counts whose units fall one short of, onto and one
past the number of SMs, of one warp on each of a CTA's eight, and of all resident ones
(152 SMs), for every number of particles per unit; bit for bit against the oracle."""
import pytest

from tests.gpu_common import BOUNDS, C12, W, assert_state_equal, load_cupso, oracle_swarm, same_bits

pytestmark = pytest.mark.gpu

UNITS = (1, 151, 152, 153, 1215, 1216, 1217)


@pytest.mark.parametrize("units", UNITS)
@pytest.mark.parametrize("kernel,per_unit,D", [("pipelined4", 32, 9), ("pipelined4", 64, 9), ("pipelined3", 128, 7),
                                               ("panel8", 16, 24), ("panel16", 8, 48)])
def test_unit_counts_match_oracle(kernel, per_unit, D, units):
    P = load_cupso()
    N, T, fid = units * per_unit - 3, 5, units % 5
    with P.Swarm(D, N, BOUNDS[fid], W, C12, C12, fid, 3) as s:
        s.set_mode("sync")
        s.set_option(P.CUPSO_OPT_SYNC_KERNEL, P.SYNC_KERNELS[kernel])
        if kernel.startswith("pipelined"):
            s.set_option(P.CUPSO_OPT_PARTICLES_PER_THREAD, per_unit // 32)
        s.step(1)
        s.step(T - 1)
        st = s.state()
        _, fit, idx, pos = s.gbest()
    ref = oracle_swarm(fid, N, D, 3).init().step_sync(T)
    assert_state_equal(st, ref)
    assert idx == ref.gbest_idx and same_bits(pos, ref.gbest_pos)
