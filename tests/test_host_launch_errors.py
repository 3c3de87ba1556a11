"""A launch that the runtime refuses is an error of the call, not a result: the residual
without allocations launches through functions that return the runtime's error."""
import pytest

from host_common import run_host


@pytest.mark.parametrize("kernel,nth", [("triples_build", 0), ("bstc64", 0), ("bstc64", 1), ("bstc_gemv", 0),
                                        ("contra3", 0), ("finalize_doubles", 0)])
def test_refused_launch_fails_the_static_residual(tmp_path_factory, kernel, nth):
    run_host(tmp_path_factory, f"""
        c, _ = context(6, 24, 4, 8, 72)
        o1, o2 = Dev(24, 6), Dev(4, 8, 6, 24)
        assert L.mlcc3_triples_omega_static(c, o1.p, o2.p) == 0
        F.fake_fail(b"{kernel}", {nth})
        rc = L.mlcc3_triples_omega_static(c, o1.p, o2.p)
        assert rc == -2, rc
        assert "too many resources" in L.mlcc3_last_error().decode()
        assert L.mlcc3_triples_omega_static(c, o1.p, o2.p) == 0
    """)
