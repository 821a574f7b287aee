"""Double-precision one-launch steps of many particles of few dimensions, whose tiles hold more particles
than the CTA has threads: one and several tiles per CTA, full and ragged, bit for bit against
the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from tests.gpu_common import load_cupso

pytestmark = pytest.mark.gpu

BOX = {0: (-100.0, 100.0, 20.0), 3: (-30.0, 30.0, 6.0), 4: (-100.0, 100.0, 20.0)}


# 152 CTAs; tiles of at most 4096 / D particles and at least 512
@pytest.mark.parametrize("fid,N,D", [(0, 152 * 4096, 1), (4, 152 * 4096 + 1, 1), (0, 1300001, 1), (3, 152 * 2048, 2),
                                     (4, 400001, 2), (3, 152 * 1365 + 3, 3), (0, 250000, 5), (3, 152 * 585 + 1, 7),
                                     (4, 152 * 512 + 1, 8), (0, 90000, 9)])
@pytest.mark.parametrize("mode", ["sync", "persistent"])
def test_large_tiles_fp64(fid, N, D, mode):
    P = load_cupso()
    with P.Swarm(D, N, BOX[fid], 1.0, 2.0, 2.0, fid, 23, mode=mode, dtype="f64") as s:
        assert 0 < s.info()["one_launch_iters"] <= 5
        s.step(5)
        st = s.state()
        rc, fit, idx, pos = s.gbest()
    ref = O.Swarm64(N, D, *BOX[fid], 1.0, 2.0, 2.0, fid, 23)
    ref.init()
    ref.step_sync(5)
    for name in ("pos", "v", "pbest_pos", "pbest_fit"):
        a, b = st[name].view(np.uint64), np.ascontiguousarray(getattr(ref, name)).view(np.uint64)
        assert np.array_equal(a, b), (name, np.argwhere(a != b)[:3])
    assert rc == P.CUPSO_OK and idx == ref.gbest_idx and fit == ref.gbest_fit
    np.testing.assert_array_equal(pos, ref.gbest_pos)
