"""The split-K parameter of the strided contractions: 0 leaves every reduction whole, in both
precisions, and larger values cut small launches into more pieces."""
import pytest

from host_common import run_host


@pytest.mark.parametrize("precision,kernel", [(0, "bstc64"), (1, "bstc32")])
def test_fill_zero_never_splits(tmp_path_factory, precision, kernel):
    run_host(tmp_path_factory, f"""
        NO, NV, no, nv, NJ = 12, 60, 4, 12, 200
        pieces = {{}}
        for fill in (0, 1, 4):
            F.fake_watch(b"{kernel}")
            c, _ = context(NO, NV, no, nv, NJ, precision={precision}, bstc_fill=fill, fp64_tc_from=100000)
            w = np.array([0.3])
            X1, X2, y1, y2 = Dev(NV, NO), Dev(no, nv, NO, NV), Dev(NV, NO), Dev(no, nv, NO, NV)
            assert L.mlcc3_jacobian_right(c, 1, w.ctypes.data, X1.p, X2.p, y1.p, y2.p) == 0
            assert L.mlcc3_jacobian_left(c, 1, w.ctypes.data, X1.p, X2.p, y1.p, y2.p) == 0
            pieces[fill] = F.fake_watched()
        assert pieces[0] == 1 and 1 < pieces[1] <= pieces[4], pieces
    """)
