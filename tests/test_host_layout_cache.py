"""The layouts of a triples array are converted once per write of it.  A call that runs out of
memory between two of them leaves none marked as there: the next call, which finds tau still
valid, converts what is missing."""
from host_common import run_host


def test_layouts_after_a_failed_allocation(tmp_path_factory):
    run_host(tmp_path_factory, """
        NO, NV, no, nv, NJ = 12, 40, 4, 20, 80
        o1, o2 = Dev(NV, NO), Dev(no, nv, NO, NV)
        layouts = lambda s: [x for x in s if "split_transpose" in x or "split_bf16_k2" in x]
        c, _ = context(NO, NV, no, nv, NJ, precision=1)
        assert L.mlcc3_triples_omega(c, o1.p, o2.p) == 0
        want = len(layouts(launches()))
        assert want >= 3, want
        failed = 0
        for n in range(100):  # allocations fail from the n-th on
            c, _ = context(NO, NV, no, nv, NJ, precision=1)
            F.fake_fail_malloc(n)
            rc = L.mlcc3_triples_omega(c, o1.p, o2.p)
            first = layouts(launches())
            F.fake_fail_malloc(-1)
            if rc != 0:
                failed += 1
                if all(L.mlcc3_triples_omega(c, o1.p, o2.p) for _ in range(2)):
                    continue
                assert len(first) + len(layouts(launches())) >= want, n
            L.mlcc3_destroy(c)
        assert 10 < failed < 100, failed
    """)
