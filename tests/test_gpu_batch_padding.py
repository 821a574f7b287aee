"""Batches on either side of the line from which swarms that whole panels would pad stay out of the panels
(20 units of 128 particles an SM), short and long rows, with and without swarms that padding does
not touch: the results of each swarm alone."""
import numpy as np
import pytest

from tests.gpu_common import BOUNDS, C12, W, load_cupso

pytestmark = pytest.mark.gpu

DIMS = [25, 32, 33, 40, 57, 63, 64, 65, 3, 24]


# 152 SMs: 3040 units; all in panels, the padded ones out, only padded ones (none left in panels)
@pytest.mark.parametrize("swarms,N,dims", [(40, 500, DIMS), (100, 4001, DIMS), (13, 32000, DIMS), (97, 4096, [25, 33, 41])])
def test_batch_equals_each_swarm_alone(swarms, N, dims):
    P = load_cupso()
    probs = [dict(D=dims[k % len(dims)], N=N - k, bounds=BOUNDS[k % 4], w=W, c1=C12, c2=C12, fitness_id=k % 4, seed=k,
                  swarm_id=k) for k in range(swarms)]
    rc, res = P.cupso_solve_batch(probs, 9)
    assert rc == P.CUPSO_OK
    for k in range(0, swarms, max(1, swarms // 13)):
        _, one = P.cupso_solve_batch([probs[k]], 9)
        assert (one[0]["fit"], one[0]["idx"]) == (res[k]["fit"], res[k]["idx"]), (k, probs[k])
        np.testing.assert_array_equal(one[0]["pos"], res[k]["pos"])


def test_batch_that_only_fits_without_padding():
    """Five swarms of 65536 x 25: 98 MB as they are, 126 MB in whole panels, with 113 MB to be had."""
    P = load_cupso()
    import torch

    probs = [dict(D=25, N=65536, bounds=BOUNDS[0], w=W, c1=C12, c2=C12, fitness_id=0, seed=k, swarm_id=k) for k in range(5)]
    rc, free_run = P.cupso_solve_batch(probs, 3)
    assert rc == P.CUPSO_OK
    for env in ("streaming", "tiled"):   # every kernel loaded
        with pytest.MonkeyPatch.context() as m:
            m.setenv("CUPSO_BATCH_KERNEL", env)
            P.cupso_solve_batch(probs, 3)
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (113 << 20), dtype=torch.uint8, device="cuda")
    try:
        rc, res = P.cupso_solve_batch(probs, 3)
    finally:
        del hold
        torch.cuda.empty_cache()
    assert rc == P.CUPSO_OK
    for a, b in zip(free_run, res):
        assert (a["fit"], a["idx"]) == (b["fit"], b["idx"])
        np.testing.assert_array_equal(a["pos"], b["pos"])
