"""A call that runs out of device memory, wherever that happens, reports it and leaves the
context usable: the next call, with memory there again, succeeds and does all of its work."""
import pytest

from host_common import run_host

CALLS = {
    "omega": "lambda c: L.mlcc3_triples_omega(c, y1.p, y2.p)",
    "left": "lambda c: L.mlcc3_jacobian_left(c, 1, w.ctypes.data, x1.p, x2.p, y1.p, y2.p)",
    "density": "lambda c: L.mlcc3_transition_density(c, ctypes.c_double(0.3), x1.p, x2.p, x1.p, x2.p, x1.p, x2.p,"
               " D[0].p, D[1].p, D[2].p, D[3].p)",
}


@pytest.mark.parametrize("call", list(CALLS))
@pytest.mark.parametrize("precision,tc_from", [(0, 100000), (0, 1), (1, 24)])
def test_call_after_a_failed_one(tmp_path_factory, call, precision, tc_from):
    run_host(tmp_path_factory, f"""
        from collections import Counter
        dims = NO, NV, no, nv, NJ = 10, 40, 4, 20, 60
        w = np.array([0.3])
        x1, x2, y1, y2 = Dev(NV, NO), Dev(no, nv, NO, NV), Dev(NV, NO), Dev(no, nv, NO, NV)
        D = [Dev(NO + NV, NO + NV) for _ in range(4)]
        call = {CALLS[call]}
        make = lambda: context(*dims, precision={precision}, fp64_tc_from={tc_from})
        c, inputs = make()
        assert call(c) == 0
        whole = Counter(launches())
        again = None
        assert call(c) == 0
        cached = Counter(launches())  # (tau and its layouts are there)
        failed = 0
        for n in range(400):
            c, inputs = make()
            F.fake_fail_malloc(n)
            rc = call(c)
            F.fake_fail_malloc(-1)
            first = Counter(launches())
            if rc == 0:
                break
            failed += 1
            assert rc == -3, (n, rc, L.mlcc3_last_error())
            if {tc_from} == 1:  # (the digits come back with new integrals)
                assert L.mlcc3_build_integrals(c, *[x.p for x in inputs]) == 0
                launches()
                first = Counter()
            assert call(c) == 0, (n, L.mlcc3_last_error())
            second = Counter(launches())
            missing = (whole - cached) - first - second  # what tau takes, in one call or the other
            assert not missing and not cached - second, (n, missing, cached - second)
            L.mlcc3_destroy(c)
        assert 5 < failed < 400, failed
    """)
