"""When an FP64 context's digit products may not be used (operands of too wide a range, no
room for the digits), the call runs again on the FP64 pipe, and calls of its kind (all calls,
if the build or the room was the reason) stay there until the next integral build; other
errors stay errors."""
from host_common import run_host

SETUP = """
    dims = (20, 60, 6, 40, 120)
    NO, NV, no, nv, NJ = dims
    c, inputs = context(*dims)
    w = np.array([0.3])
    R1, R2, p1, p2 = Dev(NV, NO), Dev(no, nv, NO, NV), Dev(NV, NO), Dev(no, nv, NO, NV)
    right = lambda: L.mlcc3_jacobian_right(c, 1, w.ctypes.data, R1.p, R2.p, p1.p, p2.p)
    left = lambda: L.mlcc3_jacobian_left(c, 1, w.ctypes.data, R1.p, R2.p, p1.p, p2.p)
    digits = lambda s: [x for x in s if "emu_gemm" in x]
    pipe = lambda s: [x for x in s if "triples_build" in x]
"""


def test_wide_range_runs_again_on_the_pipe(tmp_path_factory):
    run_host(tmp_path_factory, SETUP + """
    assert right() == 0
    s = launches(); assert digits(s) and not pipe(s)
    F.fake_mark(b"emu_gemm", 1, 6, 4)
    assert right() == 0
    s = launches(); assert digits(s) and pipe(s)
    assert right() == 0                    # this kind of call stays on the pipe
    s = launches(); assert not digits(s) and pipe(s)
    assert left() == 0                     # another one does not
    s = launches(); assert digits(s) and not pipe(s)
    assert right() == 0
    s = launches(); assert not digits(s) and pipe(s)
    assert L.mlcc3_build_integrals(c, *[x.p for x in inputs]) == 0
    assert digits(launches())
    assert right() == 0
    s = launches(); assert digits(s) and not pipe(s)
    # in the build itself: nothing of it stays on digits
    F.fake_mark(b"emu_gemm", 1, 6, 4)
    assert L.mlcc3_build_integrals(c, *[x.p for x in inputs]) == 0
    launches()
    for call in (left, right):
        assert call() == 0
        s = launches(); assert not digits(s) and pipe(s)
    """)


def test_other_status_bits_are_errors(tmp_path_factory):
    run_host(tmp_path_factory, SETUP + """
    for bits, rc in ((2, -5), (1, -4), (6, -5)):
        F.fake_mark(b"emu_gemm", 1, 6, bits)
        assert right() == rc, bits
        assert not pipe(launches())
        assert right() == 0
        s = launches(); assert digits(s) and not pipe(s)
    """)


def test_no_room_for_digits(tmp_path_factory):
    run_host(tmp_path_factory, SETUP + """
    assert right() == 0 and left() == 0   # (what both keep is allocated)
    launches()
    c2, _ = context(*dims, fp64_tc_from=100000)
    before = F.fake_used()
    assert L.mlcc3_jacobian_right(c2, 1, w.ctypes.data, R1.p, R2.p, p1.p, p2.p) == 0
    need = F.fake_used() - before          # of the call on the pipe
    launches()
    c3, _ = context(*dims)
    F.fake_total(F.fake_used() + need + (8 << 20))
    right3 = lambda: L.mlcc3_jacobian_right(c3, 1, w.ctypes.data, R1.p, R2.p, p1.p, p2.p)
    assert right3() == 0, L.mlcc3_last_error()
    assert pipe(launches())
    assert right3() == 0
    s = launches(); assert not digits(s) and pipe(s)
    # no room for the pipe either
    c4, _ = context(3, 4, 2, 3, 5)
    F.fake_total(F.fake_used())
    o1, o2 = p1, p2
    assert L.mlcc3_triples_omega(c4, o1.p, o2.p) == -3
    """)


def test_sweep_leaves_the_digits(tmp_path_factory):
    run_host(tmp_path_factory, SETUP + """
    d, _ = context(*dims)
    sw = ctypes.c_void_p()
    both = (ctypes.c_void_p * 2)(c, d)
    assert L.mlcc3_sweep_create(ctypes.byref(sw), both, 2, 0, None) == 0
    q1, q2 = Dev(NV, NO), Dev(no, nv, NO, NV)
    assert L.mlcc3_sweep_set_system(sw, 0, 1, R1.p, R2.p, p1.p, p2.p) == 0
    assert L.mlcc3_sweep_set_system(sw, 1, 1, R1.p, R2.p, q1.p, q2.p) == 0
    ww = np.array([0.3, 0.4])
    run = lambda: L.mlcc3_sweep_run(sw, ww.ctypes.data)
    assert run() == 0
    s = launches(); assert digits(s) and not pipe(s)
    assert run() == 0
    assert launches() == ["graph", "launch"]  # a replay
    F.fake_mark(b"emu_gemm", 1, 6, 4)         # (of the first system, in the eager pass)
    assert L.mlcc3_build_integrals(d, *[x.p for x in _]) == 0
    F.fake_mark(b"emu_gemm", 1, 6, 4)
    launches()
    assert run() == 0
    s = launches(); assert digits(s) and pipe(s)
    assert run() == 0
    assert launches() == ["graph", "launch"]
    assert right() == 0                    # the same kind of call on the first context
    s = launches(); assert not digits(s) and pipe(s)
    assert left() == 0
    s = launches(); assert digits(s) and not pipe(s)
    assert run() == 0
    """)
