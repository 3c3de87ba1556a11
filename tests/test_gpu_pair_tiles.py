"""Densities at the occupied extents where the pair dots change between 3 x 3 and 4 x 4
tiles of outputs, for virtual extents that are and are not a multiple of four, in both
precisions, against the oracle.  D^{0-0} is compared without the reference density that
would hide the triples' part; the bounds are those of the two modes."""
import numpy as np
import pytest

from gpu_common import Case, oracle_all, run_all
from paper_2202_08612_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [(binding.MLCC3_FP64, 1e-10), (binding.MLCC3_SPLIT_BF16X3, 1e-4)])
@pytest.mark.parametrize("dims", [(4, 16, 1, 9, 20), (5, 14, 2, 8, 20), (5, 20, 3, 10, 20), (6, 15, 4, 7, 20),
                                  (7, 18, 5, 8, 20), (8, 17, 6, 9, 20), (9, 14, 7, 4, 20), (11, 12, 9, 5, 20),
                                  (11, 13, 10, 4, 20), (14, 10, 13, 3, 20)])
def test_pair_dots_tiles(dims, precision, tol):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = Case(*dims, nstates=1, t2_norm=0.3)
    got, ref = run_all(c, c.context(precision=precision)), oracle_all(c)
    NO = dims[0]
    for k in ("D00", "D0m", "Dm0"):
        a, b = got[k], ref[k]
        if k == "D00":
            a, b = a - c.D00_in, b - c.D00_in
        for x, y in ((a, b), (a[:NO, :NO], b[:NO, :NO])):
            assert np.linalg.norm(x - y) < tol * np.linalg.norm(y) + 1e-14, k
