"""One-launch steps of small swarms, whose particles go several to a CTA where the SMs would have room for
fewer (single precision 128 pairs of dimensions, double precision 64 dimensions, over at least 8 CTAs):
bit for bit against the oracle on either side of those lines."""
import numpy as np
import pytest

from oracle import oracle as O
from tests.gpu_common import BOUNDS, C12, W, assert_state_equal, load_cupso, oracle_swarm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,D", [(7, 1), (8, 1), (9, 2), (65, 3), (1024, 2), (1025, 1), (19456, 1), (19457, 2), (300, 8),
                                 (500, 16), (305, 86), (305, 85), (200, 127), (200, 129), (153, 256), (153, 257)])
def test_small_swarms_fp32(N, D):
    P = load_cupso()
    for fid in (1, 3):
        ref = oracle_swarm(fid, N, D, 3).init()
        with P.Swarm(D, N, BOUNDS[fid], W, C12, C12, fid, 3, mode="sync") as s:
            s.step(6)
            s.step(7)
            ref.step_sync(13)
            assert_state_equal(s.state(), ref)
            _, fit, idx, pos = s.gbest()
            assert idx == ref.gbest_idx and fit == ref.gbest_fit
            np.testing.assert_array_equal(pos, ref.gbest_pos)


@pytest.mark.parametrize("N,D", [(7, 1), (8, 1), (9, 2), (512, 1), (513, 1), (9728, 1), (9729, 1), (4864, 2), (300, 8), (300, 21),
                                 (300, 22), (200, 64), (200, 65)])
def test_small_swarms_fp64(N, D):
    P = load_cupso()
    for fid in (0, 3):
        box = (-30.0, 30.0, 6.0)
        with P.Swarm(D, N, box, W, C12, C12, fid, 3, mode="sync", dtype="f64") as s:
            s.step(6)
            s.step(7)
            st = s.state()
            _, fit, idx, pos = s.gbest()
        ref = O.Swarm64(N, D, *box, W, C12, C12, fid, 3)
        ref.init()
        ref.step_sync(13)
        for name in ("pos", "v", "pbest_pos", "pbest_fit"):
            assert st[name].tobytes() == np.ascontiguousarray(getattr(ref, name)).tobytes(), (fid, name)
        assert idx == ref.gbest_idx and fit == ref.gbest_fit
        np.testing.assert_array_equal(pos, ref.gbest_pos)


@pytest.mark.parametrize("mode", ["sync", "persistent"])
@pytest.mark.parametrize("N", [1, 31, 32, 33, 64, 1023, 1024, 1025, 1056, 2047, 2048, 2049])
def test_one_dimension_fp64_in_whole_warps(N, mode):
    """32 particles to a CTA up to 1024, then up to 64."""
    P = load_cupso()
    box = (-100.0, 100.0, 100.0)
    with P.Swarm(1, N, box, 1.0, 2.0, 2.0, 4, 5, mode=mode, dtype="f64") as s:
        s.step(9)
        s.step(4)
        st = s.state()
        _, fit, idx, pos = s.gbest()
    ref = O.Swarm64(N, 1, *box, 1.0, 2.0, 2.0, 4, 5)
    ref.init()
    ref.step_sync(13)
    for name in ("pos", "v", "pbest_pos", "pbest_fit"):
        assert st[name].tobytes() == np.ascontiguousarray(getattr(ref, name)).tobytes(), name
    assert idx == ref.gbest_idx and fit == ref.gbest_fit
    np.testing.assert_array_equal(pos, ref.gbest_pos)
