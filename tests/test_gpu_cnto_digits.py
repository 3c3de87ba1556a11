"""The CNTO matrices on the tensor cores:
column tiles of 16 to 64, 128-row tiles, 32-wide K steps and their remainders, against
the closed form of Eqs. M and N, at the repository's absolute bound of 1e-13 for a
unit vector."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
from paper_2202_08612_gb300 import cnto  # noqa: E402


@pytest.mark.parametrize("NO,NV", [(7, 73), (8, 64), (16, 33), (3, 200), (17, 129), (65, 16), (130, 9), (23, 150)])
def test_matrices_match_closed_form(NO, NV):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(NO + 31 * NV)
    R1 = rng.normal(size=(NV, NO))
    P = rng.normal(size=(NV * NO, NV * NO))
    P = P + P.T
    s = np.sqrt(np.sum(R1 * R1) + 0.5 * np.sum(P * P))
    R1, R2 = R1 / s, (P / s).reshape(NV, NO, NV, NO)
    X, Y = R2.transpose(1, 0, 2, 3).reshape(NO, -1), R2.reshape(NV, -1)
    dd = np.einsum("aiai->ai", R2)
    Mo = R1.T @ R1 + 0.5 * X @ X.T + 0.5 * np.diag((dd * dd).sum(0))
    No = R1 @ R1.T + 0.5 * Y @ Y.T + 0.5 * np.diag((dd * dd).sum(1))
    for _ in range(2):  # the second call takes its workspace from the pool
        M, N = cnto.cnto_matrices(torch.from_numpy(R1).cuda(), torch.from_numpy(R2).cuda())
        assert np.allclose(M.cpu().numpy(), Mo, rtol=0, atol=1e-13)
        assert np.allclose(N.cpu().numpy(), No, rtol=0, atol=1e-13)
        assert torch.equal(M, M.T) and torch.equal(N, N.T)
