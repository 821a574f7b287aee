"""The exact least-squares fitness where its residual tiles are partly used -- few dimensions, rows that end
inside a tile and inside a warp's rows -- bit for bit against the oracle: the multiplications past
both ends are left out."""
import numpy as np
import pytest

from oracle import oracle as O
from tests.gpu_common import load_cupso

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [1, 2, 3, 15, 16, 17, 31, 33, 64, 65, 72])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_partly_used_tiles(precision, D):
    P = load_cupso()
    import torch

    rng = np.random.default_rng(D)
    for M, N in [(1, 33), (15, 100), (16, 31), (17, 64), (33, 129), (48, 40), (63, 40), (65, 40), (79, 40), (112, 300), (129, 40),
                 (145, 2600), (257, 5000)]:   # 64 x 32, 128 x 32, 128 x 64 and 128 x 128 tiles in FP32
        A, b = rng.standard_normal((M, D)).astype(np.float32), rng.standard_normal(M).astype(np.float32)
        X = rng.uniform(-2, 2, (N, D)).astype(np.float32)
        dA, db, dX = (torch.from_numpy(a).cuda() for a in (A, b, X))
        f = torch.full((N,), float("nan"), device="cuda")
        P.cupso_lsq_eval(dA.data_ptr(), db.data_ptr(), M, D, dX.data_ptr(), N, P.LSQ_PRECISIONS[precision], f.data_ptr(),
                         torch.cuda.current_stream().cuda_stream)
        some = range(N) if N < 500 else np.unique(np.r_[0:200, N - 200:N])
        one = (lambda x: O.lsq_f32(A, b, x)) if precision == "fp32" else (lambda x: np.float32(O.lsq_f64(A, b, x)))
        ref = np.array([one(X[i]) for i in some], np.float32)
        np.testing.assert_array_equal(f.cpu().numpy()[list(some)].view(np.uint32), ref.view(np.uint32), err_msg=str((M, N)))
