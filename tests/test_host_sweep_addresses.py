"""A sweep's graph holds the addresses of its contexts' scratch.  When another call on a
context has moved some of it (larger blocks for the densities' chunks, released scratch), the
next run captures a new graph; calls that move nothing leave the old one."""
import pytest

from host_common import run_host


@pytest.mark.parametrize("precision,tc_from", [(0, 100000), (0, 1), (1, 24)])
def test_scratch_that_moved(tmp_path_factory, precision, tc_from):
    run_host(tmp_path_factory, f"""
        dims = NO, NV, no, nv, NJ = 10, 40, 4, 20, 60
        c, _ = context(*dims, precision={precision}, fp64_tc_from={tc_from}, chunk_blocks=3)
        w = np.array([0.3])
        X1, X2, y1, y2 = Dev(NV, NO), Dev(no, nv, NO, NV), Dev(NV, NO), Dev(no, nv, NO, NV)
        D = [Dev(NO + NV, NO + NV) for _ in range(4)]
        sw = ctypes.c_void_p()
        assert L.mlcc3_sweep_create(ctypes.byref(sw), (ctypes.c_void_p * 1)(c), 1, 0, None) == 0
        assert L.mlcc3_sweep_set_system(sw, 0, 1, X1.p, X2.p, y1.p, y2.p) == 0
        run = lambda: L.mlcc3_sweep_run(sw, w.ctypes.data)
        assert run() == 0
        launches()
        density = lambda: L.mlcc3_transition_density(c, ctypes.c_double(0.3), X1.p, X2.p, X1.p, X2.p, X1.p, X2.p,
                                                     *[d.p for d in D])
        assert run() == 0 and launches() == ["graph", "launch"]
        assert density() == 0                # holds more blocks at a time than the sweep's chunks
        launches()
        assert run() == 0
        assert len(launches()) > 10          # captured again
        assert density() == 0                # nothing grows any more
        launches()
        assert run() == 0 and launches() == ["graph", "launch"]
        # scratch released and allocated again between two runs
        for v in (1, 0):
            assert L.mlcc3_set_param(c, b"release_scratch", v) == 0
        assert density() == 0
        launches()
        assert run() == 0
        assert len(launches()) > 10
        assert run() == 0 and launches() == ["graph", "launch"]
    """)
