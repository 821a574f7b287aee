"""Several handles: two swarms that run the same kernel at different sizes, each stepped by a host
thread of its own or one after the other, take no launch limit from one another and get the
bits that they get alone."""
import threading

import numpy as np
import pytest

from tests.gpu_common import BOUNDS, C12, W, load_cupso

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    return load_cupso()


def _run(P, fid, N, D, mode, dtype, rounds, iters, start=None):
    with P.Swarm(D, N, BOUNDS[fid], W, C12, C12, fid, N, mode=mode, dtype=dtype) as s:
        if start:
            start.wait()
        for _ in range(rounds):
            s.step(iters)
        return s.gbest(), s.state()


# the larger swarm's kernel takes more shared memory than the smaller one's: 82 and 55 KB in
# registers (8 pairs a thread), 105 and 25 KB in double precision, and on a cluster
@pytest.mark.parametrize("mode,dtype,fid,large,small", [
    ("sync", "f32", 1, (77824, 16), (20000, 48)),
    ("sync", "f64", 0, (16384, 120), (200000, 7)),
    ("onchip", "f32", 1, (3072, 48), (512, 8)),
    ("onchip", "f64", 0, (4096, 16), (512, 16))])
def test_two_threads_step_two_sizes(P, mode, dtype, fid, large, small):
    rounds, iters = 300, 5
    got, errors, start = {}, [], threading.Barrier(2)

    def work(size):
        try:
            got[size] = _run(P, fid, *size, mode, dtype, rounds, iters, start)
        except Exception as e:
            errors.append((size, e))
            start.abort()   # the other thread may be waiting for this one

    threads = [threading.Thread(target=work, args=(size,)) for size in (large, small)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for size in (large, small):
        (rc, fit, idx, pos), st = got[size]
        (rc1, fit1, idx1, pos1), st1 = _run(P, fid, *size, mode, dtype, rounds, iters)
        assert (rc, fit, idx) == (rc1, fit1, idx1) == (P.CUPSO_OK, fit, idx)
        np.testing.assert_array_equal(pos, pos1)
        for name in ("pos", "v", "pbest_pos", "pbest_fit"):
            assert st[name].tobytes() == st1[name].tobytes(), name


def test_lsq_rescoring_keeps_its_limit_beside_a_smaller_swarm(P):
    """The FP64 Gram rescoring of 1600 dimensions (51 KB of shared memory) after a swarm of 64 was set up."""
    import torch

    torch.manual_seed(1)

    def swarm(D, N=256):
        A, b = torch.randn(D, D, device="cuda"), torch.randn(D, device="cuda")
        s = P.Swarm(D, N, (-5.0, 5.0, 1.0), W, C12, C12, "lsq", 3)
        s.set_option(P.CUPSO_OPT_LSQ_RESCORE, 1)
        s.set_lsq(A.data_ptr(), b.data_ptr(), D, "bf16")
        return s, A, b

    large, A, b = swarm(1600)
    small, A2, b2 = swarm(64)
    for s in (large, small):
        before = s.gbest_f64()
        s.step(5)
        assert s.gbest()[0] == P.CUPSO_OK and s.gbest_f64() <= before
        s.close()
