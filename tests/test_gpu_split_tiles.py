"""The split mode at extents around the tiles of its strided contractions (16 to 128
outputs, K steps of 32, FP32 sums of 64) and with either operand longer than a tile,
against the oracle at the split mode's bound of 1e-4."""
import numpy as np
import pytest

from gpu_common import Case, oracle_all, run_all
from paper_2202_08612_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(3, 5, 2, 3, 7), (17, 33, 3, 9, 33), (33, 31, 2, 17, 63), (16, 65, 3, 16, 65),
                                  (64, 40, 2, 7, 130), (70, 129, 2, 10, 32), (5, 150, 3, 12, 64)])
def test_split_mode_matches_oracle(dims):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = Case(*dims, nstates=1, t2_norm=0.3)
    got = run_all(c, c.context(precision=binding.MLCC3_SPLIT_BF16X3))
    for k, ref in oracle_all(c).items():
        err = np.linalg.norm(got[k] - ref) / np.linalg.norm(ref)
        assert err < 1e-4, (k, err)
