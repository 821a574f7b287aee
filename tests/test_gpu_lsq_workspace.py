"""The exact least-squares fitness with and without its residual workspace: the same bits as the oracle through
a swarm, whose tiles, chunks of rows and chunks of particles go through it, and through an evaluation, which
mostly does without; and the same bits where less device memory is to be had than it would take."""
import numpy as np
import pytest

from oracle import oracle as O
from tests.gpu_common import C12, W, load_cupso

pytestmark = pytest.mark.gpu


# M, D, N, floats by which A is shifted off its allocation
@pytest.mark.parametrize("M,D,N,shift", [
    (520, 36, 1300, 0), (520, 36, 1300, 1), (521, 33, 1281, 0), (129, 16, 5000, 0), (4000, 4, 4500, 0), (65, 17, 257, 0),
    (128, 129, 300, 0), (2501, 21, 2490, 0),
    (66, 33, 140000, 0),                  # chunks of particles
    (145, 2, 20000, 0), (70, 16, 9728, 0), (70, 16, 9696, 0),   # few dimensions: without from 304 blocks on in FP32,
    (70, 32, 58368, 0), (70, 32, 58336, 0),                     # up to 32 from 1824 on
])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_swarm_fitness_bits(precision, M, D, N, shift):
    P = load_cupso()
    import torch

    rng = np.random.default_rng(M + N)
    A, b = rng.standard_normal((M, D)).astype(np.float32), rng.standard_normal(M).astype(np.float32)
    buf = torch.zeros(M * D + 4, device="cuda")
    dA = buf[shift:shift + M * D]
    dA.copy_(torch.from_numpy(A.ravel()))
    db = torch.from_numpy(b).cuda()
    with P.Swarm(D, N, (-2.0, 2.0, 1.0), W, C12, C12, "lsq", 3) as s:
        s.set_lsq(dA.data_ptr(), db.data_ptr(), M, precision)
        st = s.state()
    one = (lambda x: O.lsq_f32(A, b, x)) if precision == "fp32" else (lambda x: np.float32(O.lsq_f64(A, b, x)))
    some = np.unique(np.r_[0:min(N, 300), N - 40:N, rng.integers(0, N, 300), [i for i in range(131000, 131100) if i < N]])
    ref = np.array([one(st["pbest_pos"][i]) for i in some.astype(int)], np.float32)
    np.testing.assert_array_equal(st["pbest_fit"][some.astype(int)].view(np.uint32), ref.view(np.uint32))


# either side of the lines from which an evaluation takes a workspace
@pytest.mark.parametrize("M,D,N", [(300, 8, 3000), (2000, 2, 64), (1000, 300, 300), (2100, 300, 300), (700, 100, 10000),
                                   (130, 400, 12000), (65, 2, 40000)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_evaluation_bits(precision, M, D, N):
    P = load_cupso()
    import torch

    rng = np.random.default_rng(M + N)
    A, b = rng.standard_normal((M, D)).astype(np.float32), rng.standard_normal(M).astype(np.float32)
    X = rng.uniform(-2, 2, (N, D)).astype(np.float32)
    dA, db, dX = (torch.from_numpy(a).cuda() for a in (A, b, X))
    f = torch.full((N,), float("nan"), device="cuda")
    P.cupso_lsq_eval(dA.data_ptr(), db.data_ptr(), M, D, dX.data_ptr(), N, P.LSQ_PRECISIONS[precision], f.data_ptr(),
                     torch.cuda.current_stream().cuda_stream)
    one = (lambda x: O.lsq_f32(A, b, x)) if precision == "fp32" else (lambda x: np.float32(O.lsq_f64(A, b, x)))
    some = np.unique(np.r_[0:60, N - 60:N])
    ref = np.array([one(X[i]) for i in some], np.float32)
    np.testing.assert_array_equal(f.cpu().numpy()[some].view(np.uint32), ref.view(np.uint32))


# 64 MB of workspace in FP32 (N = 16384), and in FP64 of its first chunk; a swarm and an evaluation, an evaluation
@pytest.mark.parametrize("M,D,N,left,swarm", [(1000, 40, 16384, 50, True), (1000, 300, 8192, 36, False)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_smaller_workspace_same_bits(precision, M, D, N, left, swarm):
    P = load_cupso()
    import torch

    torch.manual_seed(0)
    A, b, X = torch.randn(M, D, device="cuda"), torch.randn(M, device="cuda"), torch.randn(N, D, device="cuda")

    def run():
        f = torch.full((N,), float("nan"), device="cuda")
        P.cupso_lsq_eval(A.data_ptr(), b.data_ptr(), M, D, X.data_ptr(), N, P.LSQ_PRECISIONS[precision], f.data_ptr(),
                         torch.cuda.current_stream().cuda_stream)
        out = [f.cpu().numpy()]
        if swarm:
            with P.Swarm(D, N, (-5.0, 5.0, 1.0), W, C12, C12, "lsq", 3) as s:
                s.set_lsq(A.data_ptr(), b.data_ptr(), M, precision)
                s.step(3)
                st = s.state()
                out += [st[name] for name in ("pos", "v", "pbest_pos", "pbest_fit")] + [s.gbest()[3]]
        return out

    ample = run()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (left << 20), dtype=torch.uint8, device="cuda")
    try:
        short = run()
    finally:
        del hold
        torch.cuda.empty_cache()
    for a, c in zip(ample, short):
        assert a.tobytes() == c.tobytes()
