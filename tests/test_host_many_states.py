"""The densities of many states in one call, on digit slices: every state has scales of its
own, of which there is no largest number."""
from host_common import run_host


def test_densities_of_two_thousand_states(tmp_path_factory):
    run_host(tmp_path_factory, """
        NO, NV, no, nv, NJ = dims = 3, 5, 2, 3, 6
        n = 2000
        c, _ = context(*dims, fp64_tc_from=1)
        w = np.full(n, 0.3)
        X1, X2, D = Dev(n, NV, NO), Dev(n, no, nv, NO, NV), [Dev(n, NO + NV, NO + NV) for _ in range(4)]
        for _ in range(2):
            assert L.mlcc3_transition_densities(c, n, w.ctypes.data, X1.p, X2.p, X1.p, X2.p, X1.p, X2.p,
                                                *[d.p for d in D]) == 0, L.mlcc3_last_error()
            assert any("emu_gemm" in x for x in launches())
    """)
