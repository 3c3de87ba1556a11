"""What FP64 contexts take of the device memory: whether a system's contractions run on digit
slices follows from its sizes and the card alone, the default chunks leave room for all digits
that live at once, and both precisions' chunks follow the layouts that are really kept."""
import pytest

from host_common import run_host

CALLS = """
    def calls(dims, **params):
        NO, NV, no, nv, NJ = dims
        c, inputs = context(*dims, **params)
        w = np.array([0.3])
        X1, X2, y1, y2 = Dev(NV, NO), Dev(no, nv, NO, NV), Dev(NV, NO), Dev(no, nv, NO, NV)
        D = [Dev(NO + NV, NO + NV) for _ in range(4)]
        names = []
        for f in (lambda: L.mlcc3_triples_omega(c, y1.p, y2.p),
                  lambda: L.mlcc3_jacobian_right(c, 1, w.ctypes.data, X1.p, X2.p, y1.p, y2.p),
                  lambda: L.mlcc3_jacobian_left(c, 1, w.ctypes.data, X1.p, X2.p, y1.p, y2.p),
                  lambda: L.mlcc3_transition_density(c, ctypes.c_double(0.3), X1.p, X2.p, X1.p, X2.p, X1.p, X2.p,
                                                     *[d.p for d in D])):
            assert f() == 0, L.mlcc3_last_error()
            names.append(launches())
        return c, names
"""


def test_the_path_does_not_depend_on_what_else_holds_memory(tmp_path_factory):
    run_host(tmp_path_factory, CALLS + """
    dims = NO, NV, no, nv, NJ = 30, 200, 10, 60, 400
    digits = 18 * 15 * no * nv * nv * NV  # the largest part of them
    for used in (0.0, 0.4, 0.7):
        F.fake_total(10 * digits)
        other = Dev(int(used * 10 * digits / 8)) if used else None
        c, names = calls(dims, chunk_blocks=4)
        assert all(any("emu_gemm" in x for x in s) for s in names), used
        # a parameter set again to what it is changes nothing
        assert L.mlcc3_set_param(c, b"fp64_tc_from", 24) == 0
        o1, o2 = Dev(NV, NO), Dev(no, nv, NO, NV)
        assert L.mlcc3_triples_omega(c, o1.p, o2.p) == 0
        if other: F.cudaFree(other.p)
        L.mlcc3_destroy(c)
    """)


@pytest.mark.parametrize("share", [0.05, 0.15, 0.25, 0.35, 0.39])
@pytest.mark.parametrize("dims", [(30, 200, 10, 60, 400), (12, 300, 5, 100, 900), (40, 120, 20, 40, 200)])
def test_default_chunks_leave_room_for_the_digits(tmp_path_factory, dims, share):
    """A card of which the digits would take about `share` (before padding): every call stays
    on them, or, near the line, every call is on the pipe from the start."""
    run_host(tmp_path_factory, CALLS + f"""
    dims = {dims}
    NO, NV, no, nv, NJ = dims
    gv, vV, blk, tl = no * nv * nv * NV, NJ * nv * NV, no * no * nv * NV, no * nv * nv * NO
    digits = 18 * (15 * gv + 5 * vV + 5 * blk + 14 * tl)
    F.fake_total(int(digits / {share}))
    c, names = calls(dims)
    on = [any("emu_gemm" in x for x in s) for s in names]
    assert all(on) or ({share} > 0.3 and not any(on)), on
    """)


@pytest.mark.parametrize("precision", [0, 1])
def test_default_chunks_fill_half_of_the_memory(tmp_path_factory, precision):
    """Eight arrays of a block element and the layouts of those kept converted: three FP64
    ones in digits (18 bytes), four of the split mode (4 bytes), three layouts each.  The
    largest default chunk is what fits half of the memory at that count."""
    run_host(tmp_path_factory, CALLS + f"""
    dims = NO, NV, no, nv, NJ = 24, 60, 20, 40, 100
    element = {84 if precision else 226}
    blocks = 300
    # half of what is left beside the persistent arrays and the digits holds 300 of the 1520 blocks
    F.fake_total(10 << 30)
    c, _ = context(*dims, precision={precision}, build=False)
    before = F.fake_used()
    L.mlcc3_destroy(c)
    gvp = no * nv * nv * 64
    digits = 0 if {precision} else 18 * 15 * gvp
    F.fake_total(before + int(1.2 * digits) + int(2.0 * element * blocks * nv ** 3))
    c, names = calls(dims, precision={precision})
    built = sum("triples_finish" in x for x in names[0])   # one finish per chunk of the residual
    assert 1520 / 300 * 0.75 < built < 1520 / 300 * 1.35, built
    """)
