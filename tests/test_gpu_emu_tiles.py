"""The digit-slice tensor-core kernel (mlcc3_fp64emu_gemm) at the edges of its tiles.

Integers of few enough bits fill only leading digits t with 2 t < slices, so no
digit pair is dropped, and their sums of products stay below 2^53: the result
has to equal the integer product exactly, whatever the tiling.
"""
import numpy as np
import pytest

from paper_2202_08612_gb300 import binding

pytestmark = pytest.mark.gpu

# bits per element that fill digits 0 .. (slices - 1) // 2 (8 bits each, one for the sign)
BITS = {2: 7, 3: 14, 4: 14, 5: 20, 6: 20}


@pytest.mark.parametrize("M,N,K,slices", [
    (1, 1, 1, 5), (127, 79, 31, 5), (128, 80, 32, 5), (129, 81, 33, 5),   # one tile, one over, one under
    (130, 160, 255, 3), (256, 161, 257, 4), (64, 96, 513, 6),             # accumulation chains of 256
    (200, 17, 8190, 6), (140, 90, 8300, 5), (1300, 1100, 70, 2)])         # pieces of K, many tiles
def test_integer_products_are_exact(M, N, K, slices):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(M + 3 * N + 7 * K + slices)
    top = 1 << BITS[slices]
    A = rng.integers(-top + 1, top, size=(M, K)).astype(np.float64)
    B = rng.integers(-top + 1, top, size=(N, K)).astype(np.float64)
    # equal exponents in every row, so that no element's digits start lower
    A[:, 0], B[:, 0] = top - 1, 1 - top
    c = torch.empty((M, N), dtype=torch.float64, device="cuda")
    binding.fp64emu_gemm(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), c, slices=slices)
    want = A.astype(np.int64) @ B.astype(np.int64).T
    assert np.array_equal(c.cpu().numpy().astype(np.int64), want)


def test_rows_that_are_not_finite_give_nan_and_no_other_row_does():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(11)
    A, B = rng.standard_normal((140, 70)), rng.standard_normal((90, 70))
    A[5, 3], A[130, 69], B[7, 0] = np.inf, np.nan, -np.inf
    c = torch.empty((140, 90), dtype=torch.float64, device="cuda")
    binding.fp64emu_gemm(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), c, slices=5)
    bad = np.zeros((140, 90), dtype=bool)
    bad[[5, 130]] = True
    bad[:, 7] = True
    assert np.array_equal(np.isnan(c.cpu().numpy()), bad)
