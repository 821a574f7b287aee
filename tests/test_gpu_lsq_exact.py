"""The exact least-squares fitness (residual tiles, then the ordered sum) bit for bit
against the oracle where its tiling can go wrong: large and small tiles with
ragged edges, rows read as vectors and one by one, several chunks of rows and of
particles in the residual workspace."""
import numpy as np
import pytest

from oracle import oracle as O
from tests.gpu_common import load_cupso

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    return load_cupso()


# M, D, N, floats by which A is shifted off its allocation
@pytest.mark.parametrize("M,D,N,shift", [
    (1, 1, 1, 0), (520, 36, 1300, 0), (520, 36, 1300, 1), (521, 33, 1281, 0), (129, 16, 5000, 0), (127, 17, 63, 0),
    (4000, 4, 4500, 0), (3, 2, 140000, 0), (66, 2, 140000, 0), (64, 17, 257, 0), (65, 17, 257, 0), (128, 128, 300, 0), (128, 129, 300, 0),
    (101, 33, 40, 1),
    (2501, 21, 2490, 0),   # 128 x 128 tiles, ragged on every side
])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_exact_fitness_bits(P, precision, M, D, N, shift):
    import torch
    rng = np.random.default_rng(M + N)
    A = rng.standard_normal((M, D)).astype(np.float32)
    b = rng.standard_normal(M).astype(np.float32)
    X = rng.uniform(-2, 2, (N, D)).astype(np.float32)
    buf = torch.zeros(M * D + 4, device="cuda")
    dA = buf[shift:shift + M * D]
    dA.copy_(torch.from_numpy(A.ravel()))
    db, dX = torch.from_numpy(b).cuda(), torch.from_numpy(X).cuda()
    f = torch.full((N,), float("nan"), device="cuda")
    P.cupso_lsq_eval(dA.data_ptr(), db.data_ptr(), M, D, dX.data_ptr(), N, P.LSQ_PRECISIONS[precision], f.data_ptr(),
                     torch.cuda.current_stream().cuda_stream)
    one = (lambda x: O.lsq_f32(A, b, x)) if precision == "fp32" else (lambda x: np.float32(O.lsq_f64(A, b, x)))
    some = range(N) if N * M * D <= 1 << 27 and N < 10000 else np.unique(np.r_[0:40, N - 40:N, rng.integers(0, N, 2000),
                                                                               131000:131100])
    ref = np.array([one(X[i]) for i in some], np.float32)
    np.testing.assert_array_equal(f.cpu().numpy()[list(some)].view(np.uint32), ref.view(np.uint32))
