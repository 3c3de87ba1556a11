"""The FP64-accurate product into one of its own operands: both are read whole before C is
written, also where a tile's reduction is cut into pieces that add into a cleared C
(N = 1100 from K = 1024 on).  Compared bit for bit with the product into another array when
the reduction is whole, and to the pieces' rounding when it is cut."""
import numpy as np
import pytest

from paper_2202_08612_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N", [(64, 300), (64, 1100), (300, 1100)])
@pytest.mark.parametrize("into", ["A", "B"])
def test_product_into_an_operand(M, N, into):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(M + N)
    # C = A B^T fits A's place for K = N, and B's for K = N = M
    M = M if into == "A" else N
    A, B = rng.standard_normal((M, N)), rng.standard_normal((N, N))
    dev = lambda x: torch.from_numpy(x).cuda()
    a, b, c = dev(A), dev(B), torch.empty((M, N), dtype=torch.float64, device="cuda")
    binding.fp64emu_gemm(a, b, c, slices=5)
    want = c.cpu().numpy()
    target = a if into == "A" else b
    binding.fp64emu_gemm(a, b, target, slices=5)
    got = target.cpu().numpy()
    # three pieces at most, one rounding each
    assert np.abs(got - want).max() <= 3 * 2.0 ** -52 * np.abs(want).max()
