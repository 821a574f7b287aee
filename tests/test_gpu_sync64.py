"""The one-launch FP64 steps bit for bit against the FP64 oracle: the swarm in registers
(1 to 16 dimensions per thread) and in memory (one and several tiles per CTA), ragged
particle counts, the sizes between the two, w = 1 and not, single steps between them."""
import numpy as np
import pytest

from oracle import oracle as O
from tests.gpu_common import load_cupso

pytestmark = pytest.mark.gpu

BOUNDS = {0: (-100.0, 100.0, 20.0), 3: (-30.0, 30.0, 6.0), 4: (-100.0, 100.0, 20.0)}


@pytest.fixture(scope="module")
def P():
    return load_cupso()


@pytest.mark.parametrize("fid", [0, 3, 4])
@pytest.mark.parametrize("N,D", [(1, 1), (2, 300), (153, 2), (4001, 7), (8192, 1), (9000, 30), (31, 120), (2000, 120),
                                 (20000, 30), (100000, 30), (155649, 1), (155000, 2), (200, 4096)])
def test_one_launch_fp64(P, fid, N, D):
    w, c = (1.0, 2.0) if fid == 4 else (0.729, 1.49445)
    steps = (5, 1, 3) if N * D < 1_000_000 else (5,)
    with P.Swarm(D, N, BOUNDS[fid], w, c, c, fid, 17, mode="sync", dtype="f64") as s:
        for n in steps:
            s.step(n)
        st = s.state()
        rc, fit, idx, pos = s.gbest()
    ref = O.Swarm64(N, D, *BOUNDS[fid], w, c, c, fid, 17)
    ref.init()
    ref.step_sync(sum(steps))
    for name in ("pos", "v", "pbest_pos", "pbest_fit"):
        a, b = st[name].view(np.uint64), np.ascontiguousarray(getattr(ref, name)).view(np.uint64)
        assert np.array_equal(a, b), (name, np.argwhere(a != b)[:3])
    assert rc == P.CUPSO_OK and idx == ref.gbest_idx and fit == ref.gbest_fit
    np.testing.assert_array_equal(pos, ref.gbest_pos)
