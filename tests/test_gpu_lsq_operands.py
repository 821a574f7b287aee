"""cupso_lsq_eval on the tensor cores where its operand preparation can go wrong:
rows read as vectors and one by one (D, and where A and X start), padding in
every direction, a zero row of A and all-zero positions."""
import numpy as np
import pytest

from oracle import oracle as O
from tests.gpu_common import load_cupso

pytestmark = pytest.mark.gpu

RTOL_ACC = {"bf16": 2e-5, "fp8": 1e-4}      # the FP32 accumulation, as in test_gpu_lsq.py


@pytest.fixture(scope="module")
def P():
    return load_cupso()


@pytest.mark.parametrize("fmt", ["bf16", "fp8"])
@pytest.mark.parametrize("M,D,N,shift,zero", [(1, 1, 1, 0, False), (257, 65, 130, 0, False), (300, 64, 129, 1, False),
                                              (512, 130, 300, 2, False), (40, 12, 20, 0, True)])
def test_operands_of_given_positions(P, fmt, M, D, N, shift, zero):
    import torch
    rng = np.random.default_rng(M + D)
    A = (rng.standard_normal((M, D)) / 16).astype(np.float32)
    A[M // 2] = 0
    b = rng.standard_normal(M).astype(np.float32)
    X = np.zeros((N, D), np.float32) if zero else rng.uniform(-2, 2, (N, D)).astype(np.float32)

    def shifted(a):
        buf = torch.zeros(a.size + 4, device="cuda")
        buf[shift:shift + a.size] = torch.from_numpy(a.ravel()).cuda()
        return buf, buf.data_ptr() + 4 * shift

    kA, pA = shifted(A)
    kX, pX = shifted(X)
    db = torch.from_numpy(b).cuda()
    f = torch.full((N,), float("nan"), device="cuda")
    P.cupso_lsq_eval(pA, db.data_ptr(), M, D, pX, N, P.LSQ_PRECISIONS[fmt], f.data_ptr(),
                     torch.cuda.current_stream().cuda_stream)
    top = np.abs(X).max()
    sx = np.float32(448.0) / top if top > 0 else np.float32(1)
    ref = np.array([O.lsq_disp(A, b, X[i], np.zeros(D, np.float32), fmt, sx) for i in range(N)])
    np.testing.assert_allclose(f.cpu().numpy().astype(np.float64), ref, rtol=RTOL_ACC[fmt], atol=1e-7)
