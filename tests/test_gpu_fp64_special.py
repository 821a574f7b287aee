"""Double-precision moves of special values (NaN of either sign, infinities, signed zeros,
the bounds themselves and their neighbours) bit for bit against the FP64 oracle, in
every kernel that moves a particle, with w = 1 and not."""
import numpy as np
import pytest

from oracle import oracle as O
from tests.gpu_common import load_cupso

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    return load_cupso()


@pytest.mark.parametrize("mode", ["sync", "persistent", "tree", "queue", "onchip"])
@pytest.mark.parametrize("D", [1, 17])
@pytest.mark.parametrize("w,c,lo", [(1.0, 2.0, -100.0), (0.729, 1.49445, 0.0)])
def test_special_values_fp64(P, mode, D, w, c, lo):
    hi, vmax = 100.0, 20.0
    nan, inf = np.nan, np.inf
    special = np.array([nan, -nan, inf, -inf, 0.0, -0.0, lo, hi, np.nextafter(hi, inf), np.nextafter(lo, -inf), vmax, -vmax,
                        np.nextafter(vmax, inf), 5e-324, -5e-324, 1e308, -1e308, 3.0])
    N = 300
    rng = np.random.default_rng(D)
    pos, v, pb = (rng.uniform(max(lo, -50), 50, (N, D)) for _ in range(3))
    m = len(special)
    for k in range(m):                      # every pair of special pos and v, somewhere
        pos[k * 16:k * 16 + 16, k % D] = special[k]
        v[k * 16:k * 16 + 16, k % D] = special[(np.arange(16) + k) % m]
    pf = rng.uniform(1e6, 2e6, N)
    ref = O.Swarm64(N, D, lo, hi, vmax, w, c, c, 0, 5)
    ref.init()
    ref.set_state(pos, v, pb, pf, 3)
    with P.Swarm(D, N, (lo, hi, vmax), w, c, c, 0, 5, mode=mode, dtype="f64") as s:
        s.set_state(pos, v, pb, pf, 3)
        s.step(1)
        s.step(3)
        st = s.state()
    ref.step_sync(4)
    for name in ("pos", "v", "pbest_pos", "pbest_fit"):
        a, b = st[name].view(np.uint64), np.ascontiguousarray(getattr(ref, name)).view(np.uint64)
        np.testing.assert_array_equal(a, b, err_msg=name)
