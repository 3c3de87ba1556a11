"""The FP64 sweep with its contractions on the tensor cores (digit slices): the captured
graph holds the operands' scales and conversions, so that a replay with other vectors, of
other magnitudes, gives what the contexts' own calls on the FP64 pipe give; and a replay
whose vectors the digits cannot hold to FP64 accuracy runs again on the pipe.

Bounds: 1e-12 of the largest element between two FP64 forms (as for chunked against
unchunked sums), element by element where the vectors span orders of magnitude
(test_gpu_wide_range.py).
"""
import numpy as np
import pytest

from gpu_common import Case, rel_err
from paper_2202_08612_gb300 import binding

pytestmark = pytest.mark.gpu

SYSTEMS = [((6, 24, 4, 8, 72), 3), ((7, 30, 5, 13, 40), 4), ((9, 40, 6, 16, 60), 1)]


def _sweep(params=None):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cases = [Case(*d, nstates=n, seed=300 + q, t2_norm=0.3) for q, (d, n) in enumerate(SYSTEMS)]
    ctxs = [c.context(params={"fp64_tc_from": 1, **(params or {})}) for c in cases]
    pipes = [c.context(params={"fp64_tc_from": 2000}) for c in cases]
    sw = binding.Sweep(ctxs, tune=False)
    vecs = []
    for q, c in enumerate(cases):
        v = [c.to_dev(c.st.R1), c.to_dev(c.st.R2), c.empty_dev(c.st.R1.shape), c.empty_dev(c.st.R2.shape)]
        sw.set_system(q, *v)
        vecs.append(v)
    return cases, ctxs, pipes, sw, vecs


def _check(cases, pipes, vecs, omegas, factors=None):
    for q, (c, g, v, w) in enumerate(zip(cases, pipes, vecs, omegas)):
        e1, e2 = c.empty_dev(c.st.R1.shape), c.empty_dev(c.st.R2.shape)
        g.jacobian_right(w, v[0], v[1], e1, e2)
        for n in range(e1.shape[0]):  # vector by vector
            for a, b, f in ((v[2], e1, 1.0 if factors is None else factors[q][0]),
                            (v[3], e2, 1.0 if factors is None else factors[q][1])):
                assert rel_err(c.host(a[n]) / f, c.host(b[n]) / f) < (1e-12 if factors is None else 1e-11), (q, n)


def _calls_between(c, g):
    """Other calls on a sweep's context: they use its scratch, scales and layouts."""
    NO, NV = c.sys.dims.n_occ, c.sys.dims.n_vir
    s1, s2 = c.empty_dev(c.st.R1.shape), c.empty_dev(c.st.R2.shape)
    g.jacobian_left(c.st.omega, c.to_dev(1e5 * c.st.L1), c.to_dev(1e5 * c.st.L2), s1, s2)
    D = [c.empty_dev((NO + NV, NO + NV)) for _ in range(3)]
    g.transition_density(float(c.st.omega[0]), c.to_dev(c.lam1), c.to_dev(c.lam2), c.to_dev(c.st.R1[0]),
                         c.to_dev(c.st.R2[0]), c.to_dev(c.st.L1[0]), c.to_dev(c.st.L2[0]), c.to_dev(c.D00_in), *D)
    g.triples_omega(c.empty_dev((NV, NO)), c.empty_dev(c.sys.t2c.shape))


def test_replays_with_other_magnitudes_and_calls_between():
    cases, ctxs, pipes, sw, vecs = _sweep()
    omegas = [c.st.omega for c in cases]
    sw.run(np.concatenate(omegas))
    _check(cases, pipes, vecs, omegas)
    nodes = sw.info()["graph_nodes"]
    for scale in (1e-7, 3e6):
        for c, g in zip(cases, ctxs):
            _calls_between(c, g)
        for v in vecs:
            for k in range(v[0].shape[0]):  # and one vector unlike the next
                v[0][k] *= scale * 10.0 ** k
                v[1][k] *= scale * 10.0 ** k
        omegas = [w + 0.01 for w in omegas]
        sw.run(np.concatenate(omegas))
        _check(cases, pipes, vecs, omegas)
    assert sw.info()["graph_nodes"] == nodes


def test_vectors_of_a_wide_range_run_on_the_fp64_pipe():
    cases, ctxs, pipes, sw, vecs = _sweep()
    omegas = [c.st.omega for c in cases]
    sw.run(np.concatenate(omegas))
    factors = []
    for q, (c, v) in enumerate(zip(cases, vecs)):
        NO, NV, no, nv, _ = c.dims
        d = 7.0 if q == 1 else 0.0  # one system of the three
        so = 10.0 ** (-d * np.arange(NO) / (NO - 1))
        f1 = np.ones((NV, 1)) * so[None, :]
        f2 = (so[:no, None, None, None] * so[None, None, :, None]) * np.ones((no, nv, NO, NV))
        v[0] *= c.to_dev(f1)
        v[1] *= c.to_dev(f2)
        factors.append((np.ones((1, 1)), np.ones((1, 1, 1, 1))))
    sw.run(np.concatenate(omegas))
    _check(cases, pipes, vecs, omegas, factors)
    sw.run(np.concatenate(omegas))  # and a replay of the new graph
    _check(cases, pipes, vecs, omegas, factors)



def test_chunked_replays_after_calls_that_move_the_scratch():
    """The densities hold more blocks at a time than the sweep's chunks: their first call moves
    the triples arrays that the captured graph was made for."""
    cases, ctxs, pipes, sw, vecs = _sweep({"chunk_blocks": 4})
    omegas = [c.st.omega for c in cases]
    for n in range(3):
        sw.run(np.concatenate(omegas))
        _check(cases, pipes, vecs, omegas)
        for c, g in zip(cases, ctxs):
            _calls_between(c, g)
        omegas = [w + 0.01 for w in omegas]
