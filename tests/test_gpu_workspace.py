"""The workspace that the calls without a context keep between calls is given back on request,
and the calls go on as before."""
import pytest

from paper_2202_08612_gb300 import binding, cnto

pytestmark = pytest.mark.gpu


def test_workspace_is_given_back():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    a, b, c = (torch.ones((2048, 2048), dtype=torch.float64, device="cuda") for _ in range(3))
    R1, R2 = torch.ones((60, 20), dtype=torch.float64, device="cuda"), torch.ones((60, 20, 60, 20), dtype=torch.float64, device="cuda")
    free = lambda: torch.cuda.mem_get_info()[0]
    for _ in range(2):
        binding.release_workspace()
        torch.cuda.synchronize()
        before = free()
        binding.fp64emu_gemm(a, b, c, slices=5)
        cnto.cnto_matrices(R1, R2)
        torch.cuda.synchronize()
        assert before - free() > (64 << 20)  # 2 x 5 slices of 8 MiB are kept
        binding.release_workspace()
        assert before - free() < (16 << 20)  # (torch's own blocks for M and N)
        assert float(c[0, 0]) == 2048.0
