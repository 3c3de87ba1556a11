"""The FP64 mode's contractions on the tensor cores (digit slices) against the oracle
and against the same context on the FP64 pipe, at extents around the tiles: 16-column
groups, 64 columns, 128 rows and pairs, 32-wide K chunks.

Both forms are FP64 results: the repository's 1e-10 against the oracle, and 1e-12
between the two (the bound of chunked against unchunked sums).
"""
import numpy as np
import pytest

from gpu_common import Case, oracle_all, rel_err, run_all
from paper_2202_08612_gb300 import binding

pytestmark = pytest.mark.gpu


def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


SIZES = [(2, 3, 2, 1, 3), (6, 24, 4, 8, 72), (7, 31, 3, 15, 33), (5, 18, 2, 17, 65), (9, 33, 3, 32, 40),
         (4, 70, 2, 33, 31), (34, 66, 2, 20, 64)]


@pytest.mark.parametrize("dims", SIZES)
def test_digit_contractions_match_oracle_and_fp64_pipe(dims):
    _cuda()
    c = Case(*dims, nstates=1)
    got = run_all(c, c.context(params={"fp64_tc_from": 1}))
    simt = run_all(c, c.context(params={"fp64_tc_from": 2000}))
    for k, ref in oracle_all(c).items():
        if dims[3] == 1:  # contravariant blocks of one virtual orbital vanish: rounding only
            assert max(np.abs(got[k]).max(), np.abs(simt[k]).max(), np.abs(ref).max()) < 1e-20, k
            continue
        assert rel_err(got[k], ref) < 1e-10, (k, rel_err(got[k], ref))
        assert rel_err(got[k], simt[k]) < 1e-12, (k, rel_err(got[k], simt[k]))


@pytest.mark.parametrize("params", [{"chunk_blocks": 4}, {"release_scratch": 1}])
def test_chunks_and_released_scratch(params):
    _cuda()
    c = Case(7, 30, 5, 13, 40, nstates=2)
    ref = run_all(c, c.context(params={"fp64_tc_from": 2000}))
    g = c.context(params={"fp64_tc_from": 1, **params})
    for _ in range(2):  # the second call's scales and layouts follow the first's
        got = run_all(c, g)
        for k in ref:
            assert rel_err(got[k], ref[k]) < 1e-12, (k, rel_err(got[k], ref[k]))


def test_core_valence_separation():
    _cuda()
    c = Case(6, 22, 4, 9, 30, core=True, nstates=1)
    ref = oracle_all(c)
    got = run_all(c, c.context(params={"fp64_tc_from": 1}))
    for k in ref:
        assert rel_err(got[k], ref[k]) < 1e-10, (k, rel_err(got[k], ref[k]))


def test_changed_path_needs_new_integrals():
    _cuda()
    c = Case(6, 24, 4, 8, 72, nstates=1)
    g = c.context(params={"fp64_tc_from": 1})
    g.set_param("fp64_tc_from", 2000)
    with pytest.raises(binding.MLCC3Error):
        g.triples_omega(c.empty_dev((24, 6)), c.empty_dev(c.sys.t2c.shape))
    with pytest.raises(binding.MLCC3Error):
        g.set_param("fp64_tc_from", 0)


def test_a_vector_that_is_not_finite_gives_nan():
    _cuda()
    c = Case(6, 24, 4, 8, 72, nstates=1)
    g = c.context(params={"fp64_tc_from": 1})
    R2 = np.array(c.st.R2)
    R2[0, 1, 2, 3, 4] = np.nan
    r1, r2 = c.empty_dev(c.st.R1.shape), c.empty_dev(c.st.R2.shape)
    g.jacobian_right(c.st.omega, c.to_dev(c.st.R1), c.to_dev(R2), r1, r2)
    assert np.isnan(c.host(r2)).any()


@pytest.mark.parametrize("dims", [(9, 24, 8, 9, 30), (25, 20, 24, 3, 24), (5, 40, 2, 24, 40), (7, 24, 5, 14, 30)])
def test_default_rule_around_its_line(dims):
    """n_o n_v = 72 or n_v = 24 take the digits, 5/14 the FP64 pipe: the same results."""
    _cuda()
    c = Case(*dims, nstates=1)
    got, simt = run_all(c, c.context()), run_all(c, c.context(params={"fp64_tc_from": 2000}))
    for k in got:
        assert rel_err(got[k], simt[k]) < 1e-12, (k, rel_err(got[k], simt[k]))
