"""Split-precision sums below binary32's normal range are kept: vectors scaled by 2^-100 bring
the sums of the singles' terms (products of a vector, a triples and an integral element) to
10^-38 to 10^-42, which binary32 holds in steps of 10^-45.  Bound: the split mode's 1e-4."""
import numpy as np
import pytest

from gpu_common import Case
from paper_2202_08612_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(6, 24, 4, 8, 72), (12, 60, 5, 20, 120)])
def test_scaled_vectors_give_scaled_results(dims):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = Case(*dims, nstates=1, t2_norm=0.3)
    g = c.context(precision=binding.MLCC3_SPLIT_BF16X3)
    for call, X1, X2 in (("jacobian_right", c.st.R1, c.st.R2), ("jacobian_left", c.st.L1, c.st.L2)):
        out = []
        for s in (1.0, 2.0 ** -100):
            y1, y2 = c.empty_dev(X1.shape), c.empty_dev(X2.shape)
            getattr(g, call)(c.st.omega, c.to_dev(s * X1), c.to_dev(s * X2), y1, y2)
            out.append((c.host(y1) / s, c.host(y2) / s))
        for x, y in zip(*out):
            assert np.linalg.norm(x - y) < 1e-4 * np.linalg.norm(x), call
