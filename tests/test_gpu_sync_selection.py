"""Which kernel AUTO takes for single steps where no panels are, and that the two sides of each line agree."""
import numpy as np
import pytest

from tests.gpu_common import BOUNDS, C12, W, load_cupso

pytestmark = pytest.mark.gpu

# particles per SM up to which the tiled kernel runs
LINES = [(0, 12, 780), (2, 15, 780), (1, 30, 680), (0, 63, 680), (1, 100, 560), (0, 201, 330), (3, 30, 560), (3, 63, 390),
         (3, 100, 224), (0, 8, 780)]


@pytest.mark.parametrize("fid,D,per_sm", LINES)
def test_tiled_up_to_its_line(fid, D, per_sm):
    P = load_cupso()
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for N, tiled in [(per_sm * sms, True), (per_sm * sms + 1, False)]:
        runs = []
        for kernel in ("auto", "pipelined3" if tiled else "tiled"):
            with P.Swarm(D, N, BOUNDS[fid], W, C12, C12, fid, 7, mode="sync") as s:
                s.set_option(P.CUPSO_OPT_ITERS_PER_LAUNCH, 1)
                s.set_option(P.CUPSO_OPT_SYNC_KERNEL, P.SYNC_KERNELS[kernel])
                assert (s.info()["sync_tile"] > 0) == (tiled if kernel == "auto" else kernel == "tiled")
                s.step(3)
                runs.append((s.gbest(), s.state()))
        (g0, s0), (g1, s1) = runs
        assert g0[:3] == g1[:3]
        np.testing.assert_array_equal(g0[3], g1[3])
        for name in ("pos", "v", "pbest_pos", "pbest_fit"):
            assert s0[name].tobytes() == s1[name].tobytes(), name


@pytest.mark.parametrize("N,ctas", [(100, 1), (846, 4), (1536, 6), (1537, 52), (3000, 96)])
def test_few_units_in_few_ctas(N, ctas):
    """Pipelined single steps of a few dozen units of 32 particles: whole CTAs, and the register kernel's bits."""
    P = load_cupso()
    runs = []
    for kernel in ("auto", "register"):
        with P.Swarm(5, N, BOUNDS[1], W, C12, C12, 1, 7, mode="sync") as s:
            s.set_option(P.CUPSO_OPT_ITERS_PER_LAUNCH, 1)
            s.set_option(P.CUPSO_OPT_SYNC_KERNEL, P.SYNC_KERNELS[kernel])
            assert kernel != "auto" or s.info()["sync_grid"] == ctas
            s.step(5)
            runs.append((s.gbest(), s.state()))
    (g0, s0), (g1, s1) = runs
    assert g0[:3] == g1[:3]
    for name in ("pos", "v", "pbest_pos", "pbest_fit"):
        assert s0[name].tobytes() == s1[name].tobytes(), name
