"""The candidates of the tensor-core least-squares fitness at the edges of the blocks that
select them (64 particles), of the lists a block merges at once (128) and of those that
the rescoring merges itself (256); and their FP64 residuals with more dimensions than
rows, entries of A that are zero or subnormal included."""
import numpy as np
import pytest
import torch

from tests.gpu_common import C12, W, load_cupso

pytestmark = pytest.mark.gpu

BOX = (-2.0, 2.0, 0.4)


def problem(M, D, seed):
    rng = np.random.default_rng(seed)
    A = (rng.standard_normal((M, D)) / np.sqrt(M)).astype(np.float32)
    b = (A.astype(np.float64) @ rng.uniform(-1, 1, D)).astype(np.float32)
    return A, b


def lsq_swarm(P, A, b, N, seed, precision):
    dA, db = torch.from_numpy(A).cuda(), torch.from_numpy(b).cuda()
    torch.cuda.synchronize()
    s = P.Swarm(A.shape[1], N, BOX, W, C12, C12, "lsq", seed)
    s.set_lsq(dA.data_ptr(), db.data_ptr(), A.shape[0], precision)
    return s, dA, db


def residuals(A, b, X):
    R = X.astype(np.float64) @ A.astype(np.float64).T - b.astype(np.float64)
    return (R * R).sum(1)


@pytest.mark.parametrize("precision", ["bf16", "fp8"])
@pytest.mark.parametrize("N", [1, 2, 16, 63, 64, 65, 8192, 8193, 16384, 16385, 24700])
def test_best_of_all_particles(N, precision):
    """The first gbest and that of a few iterations: the lowest FP64 residual of the pbest
    positions that were candidates. The approximate fitness is within a few percent of the
    residual, far less than the lowest and the 17th lowest of a random swarm differ by, so at
    the first evaluation that is the lowest of all."""
    P = load_cupso()
    A, b = problem(96, 24, N)
    s, *held = lsq_swarm(P, A, b, N, 7, precision)
    with s:
        f = residuals(A, b, s.state()["pos"])
        _, fit, idx, pos = s.gbest()
        assert idx == int(np.argmin(f))
        last = fit
        for _ in range(4):
            s.step(2)
            _, fit, idx, pos = s.gbest()
            assert fit <= last
            # the Gram form is within a few units of 2^-44 of the sum of its terms'
            # magnitudes, and the result is rounded once to FP32
            terms = (np.abs(A).astype(np.float64) @ np.abs(pos).astype(np.float64) + np.abs(b)) ** 2
            ref = residuals(A, b, pos[None])[0]
            assert abs(fit - ref) <= 2.0 ** -24 * ref + 2.0 ** -42 * terms.sum()
            last = fit


@pytest.mark.parametrize("M,D", [(1, 33), (8, 31), (9, 127), (17, 129), (40, 100), (100, 260)])
def test_residuals_of_wide_problems(M, D):
    """D > M: the rescored fitness is the FP64 residual."""
    P = load_cupso()
    A, b = problem(M, D, M)
    A[0, :: 3] = 0.0
    A[M // 2, 1 :: 5] = np.float32(1e-41)
    A[M - 1, 2 :: 7] = np.float32(-1e-39)
    s, *held = lsq_swarm(P, A, b, 300, 3, "bf16")
    with s:
        for _ in range(3):
            s.step(1)
            _, fit, _, pos = s.gbest()
            ref = residuals(A, b, pos[None])[0]
            # FP64 sums of D terms, squared, and of M rows on both sides, then one rounding to FP32
            terms = (np.abs(A).astype(np.float64) @ np.abs(pos).astype(np.float64) + np.abs(b)) ** 2
            assert abs(fit - ref) <= 2.0 ** -24 * ref + 2.0 ** -53 * 4 * (D + M) * terms.sum()
